// Exponents of the scaled-monomial cell basis: X^ea(i) Y^eb(i), ordered by
// total degree, then decreasing exponent of X.
#pragma once

#if defined(__CUDACC__)
#define HHO_CONSTEXPR __host__ __device__ constexpr
#else
#define HHO_CONSTEXPR constexpr
#endif

HHO_CONSTEXPR int deg_of(int i) {
    int d = 0;
    while ((d + 1) * (d + 2) / 2 <= i) ++d;
    return d;
}
HHO_CONSTEXPR int ea(int i) { return deg_of(i) - (i - deg_of(i) * (deg_of(i) + 1) / 2); }
HHO_CONSTEXPR int eb(int i) { return i - deg_of(i) * (deg_of(i) + 1) / 2; }
HHO_CONSTEXPR int eidx(int a, int b) { return (a + b) * (a + b + 1) / 2 + b; }
