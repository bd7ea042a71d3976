// The team form of the stage kernel: a block of W warps works on 32 consecutive
// cells of one class (one warp's cells in stage_kernels.cuh), lane = cell, and
// each warp takes a share of the cells' work.  Included by stage_kernels.cuh.
//
// Why.  GB300 issues one FP64 instruction per 64 cycles on an SM
// sub-partition, whatever the number of independent chains or of active lanes
// (measured), and one per 16 on the SM.  A thread that walks a whole cell
// alone (324 FP64 instructions for a solid square at k = 2, about 2000 for a
// pentagon at k = 3) therefore needs 10 to 60 us however few cells there are,
// behind some twenty dependent rounds of loads.  Here
//   1. all loads of the state and the jumps are issued at once, by all warps;
//   2. warp w forms the rates and targets of rows w, w + W, ... of every field;
//   3. warp w publishes the traces of (face, coefficient) pairs w, w + W, ...
// with the cells' state, jumps and new state in shared memory (column = lane,
// no bank conflicts) and the class matrices beside them.  Roles are uniform
// over a warp, so nothing diverges, and the loops run over the nonzero pattern
// of the class matrices: by parity on rectangles, and on axis-aligned faces of
// triangles and polygons over the half of the trace entries that do not vanish.
// The pattern is in the loop bounds, not in conditions: a predicated-off FP64
// instruction takes its slot on the FP64 pipe all the same.

// Exponents of basis function i at run time, four bits each.
__device__ __forceinline__ int ea_rt(int i) { return (int)((0x0102103210ull >> (4 * (9 - i))) & 0xf); }
__device__ __forceinline__ int eb_rt(int i) { return (int)((0x0010120123ull >> (4 * (9 - i))) & 0xf); }

// Shared memory of a team block in elements of T: class blocks, state, new
// state, jumps, target coefficients.
template <class T, int K>
__host__ __device__ constexpr size_t team_smem_elems(int max_nf) {
    return (size_t)max_nf * Dims<K>::FS + 32 * ((size_t)2 * 5 * Dims<K>::n + (size_t)max_nf * 2 * Dims<K>::f + 3 * MAX_TARGETS + 1);
}

// the integers 1, 2, 3 (a conversion would issue on the FP64 pipe)
template <class T>
__device__ __forceinline__ T small_int(int v) {
    return T(float(v));
}
template <>
__device__ __forceinline__ f2x small_int<f2x>(int v) {
    return f2x(float(v), 0.0f);
}
template <>
__device__ __forceinline__ double small_int<double>(int v) {
    return __hiloint2double(v == 1 ? 0x3ff00000 : v == 2 ? 0x40000000 : 0x40080000, 0);
}

// Jump of component comp (0 in a fluid cell; 0, 1 in a solid cell) on local face j.
template <class T, int K, bool SOLID>
__device__ __forceinline__ void team_jump(const StageArgsT<T>& A, const T* trf, const T* trs, int slot, int comp,
                                          T* jmp) {
    constexpr int f = Dims<K>::f;
    const DevOps& op = A.op;
    const size_t S = SOLID ? op.SS : op.SF;
    const T* w0 = (SOLID ? trs : trf) + (size_t)(SOLID ? comp * f : 0) * S;
    const T* om = w0 + (size_t)(SOLID ? 2 * f : f) * S;
    const int nb = __ldg((SOLID ? op.nb_s : op.nb_f) + slot);
    const T be = __ldg((SOLID ? OpData<T>::beta_s(op) : OpData<T>::beta_f(op)) + slot);   // 0 on boundary and interface
#pragma unroll
    for (int l = 0; l < f; ++l) jmp[l] = om[(size_t)l * S + slot];
    if (nb >= 0) {
#pragma unroll
        for (int l = 0; l < f; ++l) {
            const T w = w0[(size_t)l * S + nb];
            jmp[l] = (l & 1) ? fma(-be, w, jmp[l]) : fma(be, w, jmp[l]);
        }
    } else if (nb < NB_BOUNDARY) {
        const int r = -2 - nb;
        const int no = __ldg(op.if_nb + r);
        const T* co = OpData<T>::if_coef(op) + 6 * r;
#pragma unroll
        for (int l = 0; l < f; ++l) {
            if constexpr (SOLID) {
                const T b = __ldg(co + 4 + comp), wf = trf[(size_t)l * op.SF + no];
                jmp[l] = (l & 1) ? fma(-b, wf, jmp[l]) : fma(b, wf, jmp[l]);
            } else {
                const T ws = fma(__ldg(co + 1), trs[(size_t)l * op.SS + no],
                                 __ldg(co + 2) * trs[(size_t)(f + l) * op.SS + no]);
                jmp[l] = (l & 1) ? jmp[l] - ws : jmp[l] + ws;
            }
        }
    }
}

// What publishing the traces of 32 cells needs (uniform but for lq and tau).
template <class T>
struct TeamFaces {
    int nF, npad, sbase, kind, lq;
    uint32_t hor, other;   // horizontal faces; faces that are neither horizontal nor vertical
    const T* cd;           // the class's face blocks in shared memory
    T tau;
    bool real;
};

// Publishes w and omega of the cells' state V (rows of 32, this lane's column)
// into the trace buffer `tr`: warp w takes (face, coefficient) pairs w, w + W, ...
template <class T, int K, int W, bool SOLID>
__device__ __forceinline__ void team_traces(const DevOps& op, const TeamFaces<T>& F, const T* V, T* tr, int w) {
    constexpr int n = Dims<K>::n, f = Dims<K>::f, FS = Dims<K>::FS, TR = Dims<K>::TR, nP = Dims<K>::nP;
    constexpr int NC = SOLID ? 2 : 1;
    T* out = tr + (SOLID ? (size_t)2 * f * op.SF : 0);
    const size_t S = SOLID ? op.SS : op.SF;
    for (int it = w; it < F.nF * f; it += W) {
        const int j = it / f, l = it - j * f;
        const T* fm = F.cd + j * FS;
        const T* row = fm + TR + l * nP;
        const int slot = F.sbase + j * F.npad + F.lq;
        const int nb = __ldg((SOLID ? op.nb_s : op.nb_f) + slot);
        const T be = __ldg((SOLID ? OpData<T>::beta_s(op) : OpData<T>::beta_f(op)) + slot);
        T u[NC], g[NC];   // traces of the primal field and of the normal flux
#pragma unroll
        for (int c = 0; c < NC; ++c) u[c] = g[c] = T(0);
        if ((F.other >> j) & 1) {
            const T nx = fm[0], ny = fm[1];
            T m0(0), m1(0), m2(0);   // m_x, m_y or s_xx, s_yy, s_xy
#pragma unroll 1
            for (int i = 0; i < n; ++i) {
                const T v = row[i];
                const T* P = V + 32 * i;
#pragma unroll
                for (int c = 0; c < NC; ++c) u[c] = fma(v, P[32 * (SOLID ? 3 + c : 2) * n], u[c]);
                if constexpr (Fp64Form<T>::value) {
                    m0 = fma(v, P[0], m0);
                    m1 = fma(v, P[32 * n], m1);
                    if constexpr (SOLID) m2 = fma(v, P[32 * 2 * n], m2);
                } else if constexpr (SOLID) {   // the flux's coefficients first, as the thread form
                    const T xy = P[32 * 2 * n];
                    g[0] = fma(v, fma(nx, P[0], mul_rn(ny, xy)), g[0]);
                    g[1] = fma(v, fma(nx, xy, mul_rn(ny, P[32 * n])), g[1]);
                } else {
                    g[0] = fma(v, fma(nx, P[0], mul_rn(ny, P[32 * n])), g[0]);
                }
            }
            if constexpr (Fp64Form<T>::value && SOLID) {
                g[0] = fma(nx, m0, mul_rn(ny, m2));
                g[1] = fma(nx, m2, mul_rn(ny, m1));
            } else if constexpr (Fp64Form<T>::value) {
                g[0] = fma(nx, m0, mul_rn(ny, m1));
            }
        } else {
            // on a horizontal face (fixed Y) the monomial (a, b) has coefficients l <= a; l = a only on a rectangle,
            // whose centroid the face is centred on; likewise b on a vertical face
            const bool hor = (F.hor >> j) & 1;
            const bool neg = is_negative(fm[hor ? 1 : 0]);
            const T* F0 = V + 32 * (SOLID ? (hor ? 2 : 0) * n : (hor ? n : 0));   // s_xy / s_xx, m_y / m_x
            const T* F1 = V + 32 * (hor ? n : 2 * n);                             // s_yy / s_xy
            // values of the monomial with exponents l along and e across the face
            auto idx = [&](int e) { return (l + e) * (l + e + 1) / 2 + (hor ? e : l); };
            if (F.kind == KIND_SQUARE) {                    // Horner in +-rho0, see trace_square
                const T rho = signed_face_rho<T>(j == 1 || j == 2 ? 1 : -1);
                int i = idx(K - l);
#pragma unroll
                for (int c = 0; c < NC; ++c) u[c] = V[32 * ((SOLID ? 3 + c : 2) * n + i)];
                g[0] = F0[32 * i];
                if constexpr (SOLID) g[1] = F1[32 * i];
#pragma unroll 1
                for (int e = K - l - 1; e >= 0; --e) {
                    i = idx(e);
#pragma unroll
                    for (int c = 0; c < NC; ++c) u[c] = fma(rho, u[c], V[32 * ((SOLID ? 3 + c : 2) * n + i)]);
                    g[0] = fma(rho, g[0], F0[32 * i]);
                    if constexpr (SOLID) g[1] = fma(rho, g[1], F1[32 * i]);
                }
                if ((l & 1) && j >= 2) {                  // s_t = -1 on faces 2 and 3
#pragma unroll
                    for (int c = 0; c < NC; ++c) {
                        u[c] = -u[c];
                        g[c] = -g[c];
                    }
                }
            } else {
                auto add = [&](int i) {
                    const T v = row[i];
                    const T* P = V + 32 * i;
#pragma unroll
                    for (int c = 0; c < NC; ++c) u[c] = fma(v, P[32 * (SOLID ? 3 + c : 2) * n], u[c]);
                    g[0] = fma(v, F0[32 * i], g[0]);
                    if constexpr (SOLID) g[1] = fma(v, F1[32 * i], g[1]);
                };
                if (F.kind != KIND_GENERIC) {
#pragma unroll 1
                    for (int e = 0; e <= K - l; ++e) add(idx(e));
                } else {
#pragma unroll 1
                    for (int dgr = l; dgr <= K; ++dgr)    // by degree, the order of the basis
#pragma unroll 1
                        for (int b = hor ? 0 : l; b <= (hor ? dgr - l : dgr); ++b) add(dgr * (dgr + 1) / 2 + b);
                }
            }
#pragma unroll
            for (int c = 0; c < NC; ++c) g[c] = neg ? -g[c] : g[c];
        }
        T wv[NC], om[NC];
#pragma unroll
        for (int c = 0; c < NC; ++c) wv[c] = fma(F.tau, u[c], -g[c]);
        if (nb >= NB_BOUNDARY) {
#pragma unroll
            for (int c = 0; c < NC; ++c) om[c] = fma(be, wv[c], -u[c]);
        } else {
            const T* co = OpData<T>::if_coef(op) + 6 * (-2 - nb);
            if constexpr (SOLID) {
                om[0] = fma(__ldg(co), wv[0], fma(__ldg(co + 1), wv[1], -u[0]));
                om[1] = fma(__ldg(co + 2), wv[0], fma(__ldg(co + 3), wv[1], -u[1]));
            } else {
                om[0] = fma(__ldg(co), wv[0], -u[0]);
            }
        }
        if (F.real) {
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                out[(size_t)(c * f + l) * S + slot] = norm(wv[c]);
                out[(size_t)((NC + c) * f + l) * S + slot] = norm(om[c]);
            }
        }
    }
}

template <class T, int K, int MODE, int W, bool SOLID>
__device__ __forceinline__ void team_cells(const StageArgsT<T>& A, int gw, int shot, T* smem) {
    constexpr int n = Dims<K>::n, f = Dims<K>::f, FS = Dims<K>::FS, LI = Dims<K>::LI;
    constexpr int fP = Dims<K>::fP;
    constexpr int NV = SOLID ? 5 * n : 3 * n, NC = SOLID ? 2 : 1;
    const DevOps& op = A.op;
    const int lane = threadIdx.x & 31;
    // a block's tasks rarely divide by its warps: start at another warp from block to block, so that the four sub-
    // partitions of an SM (a warp stays on one) get the same number
    const int w = ((threadIdx.x >> 5) + blockIdx.x * 3) % W;
    const int cls = __ldg(op.warp_class + gw);
    const int* ci = op.cls_int + cls * CI_STRIDE;
    const int q = (gw - (SOLID ? op.n_warps_f : 0)) * 32 + lane;
    const int lq = q - __ldg(ci + CI_START);
    const bool real = lq < __ldg(ci + CI_COUNT);   // class padding computes on its own zeros and stores nothing
    const int nF = __ldg(ci + CI_NF), npad = __ldg(ci + CI_NPAD), sbase = __ldg(ci + CI_SLOT);
    const int kind = __ldg(ci + CI_KIND);
    const bool rect = kind != KIND_GENERIC;
    const int N = SOLID ? op.Ns : op.Nf;
    const size_t soff = (size_t)shot * A.state_stride + (SOLID ? (size_t)3 * n * op.Nf : 0);
    const size_t toff = (size_t)shot * A.trace_stride;
    const T* scal = SOLID ? OpData<T>::scal_s(op) : OpData<T>::scal_f(op);
    const T tau = __ldg(scal + (size_t)(SOLID ? SS_TAU : SF_TAU) * N + q);
    T* cd = smem;                                  // face blocks of the class
    T* U = cd + op.max_nf * FS + lane;             // state [NV][32]
    T* V = U + 32 * 5 * n;                         // new state
    T* J = V + 32 * 5 * n;                         // jumps [nF][NC][f], of a rectangle [2][NC][sigma, delta][f]
    T* CO = J + 32 * op.max_nf * 2 * f;            // target coefficients [n_tgt][3]
    {
        const float4* src = reinterpret_cast<const float4*>(OpData<T>::cls(op) + __ldg(ci + CI_DOFF) + Dims<K>::M0P);
        float4* dst = reinterpret_cast<float4*>(cd);
        for (int e = threadIdx.x; e < nF * FS * (int)sizeof(T) / 16; e += 32 * W) dst[e] = __ldg(src + e);
    }
    // faces by orientation: horizontal, vertical, other (a cell has at most 32)
    const uint32_t faces_h = (uint32_t)__ldg(ci + CI_HOR), faces_v = (uint32_t)__ldg(ci + CI_VER);
    const uint32_t faces_g = (nF >= 32 ? 0xffffffffu : (1u << nF) - 1u) & ~(faces_h | faces_v);
    const T* inp = A.inp + soff + q;
    wait_for_predecessor();   // so far: operator data only
    if constexpr (MODE == MODE_TRACES) {
        for (int i = w; i < NV; i += W) V[32 * i] = inp[(size_t)i * N];
        __syncthreads();
    } else {
        // ---- 1. state, jumps, target coefficients ------------------------------------
        const T* trf = A.tr_in + toff;
        const T* trs = trf + (size_t)2 * f * op.SF;
        {
            T u[(NV + W - 1) / W];
#pragma unroll
            for (int m = 0; m < (NV + W - 1) / W; ++m)
                if (m * W + w < NV) u[m] = inp[(size_t)(m * W + w) * N];
            if (rect) {
                for (int it = w; it < 2 * NC; it += W) {
                    const int ax = it / NC, comp = it % NC;
                    T jb[f], jp[f];
                    team_jump<T, K, SOLID>(A, trf, trs, sbase + ax * npad + lq, comp, jb);
                    team_jump<T, K, SOLID>(A, trf, trs, sbase + (ax + 2) * npad + lq, comp, jp);
#pragma unroll
                    for (int l = 0; l < f; ++l) {   // sigma and delta of the mirror pair, see lift_pair
                        const T jh = (l & 1) ? -jp[l] : jp[l];
                        J[32 * (it * 2 * f + l)] = jb[l] + jh;
                        J[32 * (it * 2 * f + f + l)] = jb[l] - jh;
                    }
                }
            } else {
                for (int it = w; it < nF * NC; it += W) {
                    T jmp[f];
                    team_jump<T, K, SOLID>(A, trf, trs, sbase + (it / NC) * npad + lq, it % NC, jmp);
#pragma unroll
                    for (int l = 0; l < f; ++l) J[32 * (it * f + l)] = jmp[l];
                }
            }
            for (int it = W - 1 - w; it < 3 * A.n_tgt; it += W) {   // the last warps have the fewest jumps
                const int g = it % 3;
                constexpr int row_s[3] = {SS_C1, SS_C3, SS_AV};
                if (SOLID || g < 2) CO[32 * it] = A.tgt[it / 3].coef * __ldg(scal + (size_t)(SOLID ? row_s[g] : g) * N + q);
            }
#pragma unroll
            for (int m = 0; m < (NV + W - 1) / W; ++m)
                if (m * W + w < NV) U[32 * (m * W + w)] = u[m];
        }
        __syncthreads();
        // ---- 2. rates and targets of row i of every field -------------------------------
        for (int i = w; i < n; i += W) {
            constexpr int NFLD = SOLID ? 5 : 3;
            T src[2][NFLD];   // of the first two targets, in flight while the rates are formed
#pragma unroll
            for (int t = 0; t < 2; ++t)
#pragma unroll
                for (int d = 0; d < NFLD; ++d)
                    src[t][d] = t < A.n_tgt && A.tgt[t].src ? A.tgt[t].src[soff + (size_t)(d * n + i) * N + q] : T(0);
            const int ia = ea_rt(i), ib = eb_rt(i), dg = ia + ib;
            // the derivatives: d/dX takes entry (a + 1, b), d/dY entry (a, b + 1)
            T k[NFLD];
#pragma unroll
            for (int d = 0; d < NFLD; ++d) k[d] = T(0);
            if (dg < K) {
                const int ix = (dg + 1) * (dg + 2) / 2 + ib, iy = ix + 1;
                const T cx = small_int<T>(ia + 1), cy = small_int<T>(ib + 1);
                auto at = [&](int row) { return U[32 * row]; };
                if constexpr (SOLID) {
                    k[0] = mul_rn(cx, at(3 * n + ix));
                    k[1] = mul_rn(cy, at(4 * n + iy));
                    k[2] = fma(cx, at(4 * n + ix), mul_rn(cy, at(3 * n + iy)));
                    k[3] = fma(cy, at(2 * n + iy), mul_rn(cx, at(ix)));
                    k[4] = fma(cx, at(2 * n + ix), mul_rn(cy, at(n + iy)));
                } else {
                    k[0] = mul_rn(cx, at(2 * n + ix));
                    k[1] = mul_rn(cy, at(2 * n + iy));
                    k[2] = fma(cy, at(n + iy), mul_rn(cx, at(ix)));
                }
            }
            if (rect) {
                T ks[NC];   // sum_F L j of each component
#pragma unroll
                for (int c = 0; c < NC; ++c) ks[c] = T(0);
#pragma unroll
                for (int ax = 0; ax < 2; ++ax) {
                    const T* L = cd + ax * FS + LI + i * fP;
                    const bool even = ((ax == 0 ? ib : ia) & 1) == 0;
                    const T* P = J + 32 * (ax * NC * 2 * f);
                    const T* Pn = P + (even ? 32 * f : 0);   // normal sum: delta (even) or sigma; tau sum: the other
                    const T* Ps = P + (even ? 0 : 32 * f);
#pragma unroll 1
                    for (int l = (ax == 0 ? ia : ib) & 1; l < f; l += 2) {   // L vanishes at the other parity
                        const T v = L[l];
#pragma unroll
                        for (int c = 0; c < NC; ++c) {
                            // face 0 has normal -e_y: x feeds e_xy (k[2]), y e_yy (k[1]); face 1 +e_x: x e_xx, y e_xy
                            T& e = SOLID ? (ax == 0 ? k[2 - c] : k[2 * c]) : k[1 - ax];
                            e = fma(ax == 0 ? -v : v, Pn[32 * (2 * f * c + l)], e);
                            const T js = Ps[32 * (2 * f * c + l)];
                            if constexpr (Fp64Form<T>::value) ks[c] = fma(v, js, ks[c]);
                            else k[NFLD - NC + c] = fma(v, mul_rn(tau, js), k[NFLD - NC + c]);
                        }
                    }
                }
                if constexpr (Fp64Form<T>::value) {
#pragma unroll
                    for (int c = 0; c < NC; ++c) k[NFLD - NC + c] = fma(tau, ks[c], k[NFLD - NC + c]);
                }
            } else {
                auto lift = [&](int j, T* t) {
                    const T* L = cd + j * FS + LI + i * fP;
                    const T* P = J + 32 * (j * NC * f);
#pragma unroll
                    for (int c = 0; c < NC; ++c) {
                        t[c] = mul_rn(L[0], P[32 * (c * f)]);
#pragma unroll
                        for (int l = 1; l < f; ++l) t[c] = fma(L[l], P[32 * (c * f + l)], t[c]);
                        k[NFLD - NC + c] = fma(tau, t[c], k[NFLD - NC + c]);
                    }
                };
                if constexpr (!Fp64Form<T>::value) {   // local order, see for_faces
#pragma unroll 1
                    for (int j = 0; j < nF; ++j) {
                        T t[NC];
                        lift(j, t);
                        const T nx = cd[j * FS], ny = cd[j * FS + 1];
                        k[0] = fma(nx, t[0], k[0]);
                        k[1] = fma(ny, t[NC - 1], k[1]);
                        if constexpr (SOLID) k[2] = fma(nx, t[1], fma(ny, t[0], k[2]));
                    }
                } else {
#pragma unroll 1
                    for (unsigned m = faces_h; m; m &= m - 1) {
                        const int j = __ffs(m) - 1;
                        T t[NC];
                        lift(j, t);
                        const bool neg = is_negative(cd[j * FS + 1]);
                        if constexpr (SOLID) k[2] += neg ? -t[0] : t[0];
                        k[1] += neg ? -t[NC - 1] : t[NC - 1];
                    }
#pragma unroll 1
                    for (unsigned m = faces_v; m; m &= m - 1) {
                        const int j = __ffs(m) - 1;
                        T t[NC];
                        lift(j, t);
                        const bool neg = is_negative(cd[j * FS]);
                        k[0] += neg ? -t[0] : t[0];
                        if constexpr (SOLID) k[2] += neg ? -t[1] : t[1];
                    }
#pragma unroll 1
                    for (unsigned m = faces_g; m; m &= m - 1) {
                        const int j = __ffs(m) - 1;
                        T t[NC];
                        lift(j, t);
                        const T nx = cd[j * FS], ny = cd[j * FS + 1];
                        k[0] = fma(nx, t[0], k[0]);
                        k[1] = fma(ny, t[NC - 1], k[1]);
                        if constexpr (SOLID) k[2] = fma(nx, t[1], fma(ny, t[0], k[2]));
                    }
                }
            }
            if constexpr (SOLID) {
                const T r = __ldg(scal + (size_t)SS_R * N + q);
                const T a = k[0], b = k[1];
                k[0] = fma(r, b, a);
                k[1] = fma(r, a, b);
            }
            // point sources (stored vectors include the material factor, see stage_kernels.cuh)
            for (int s = 0; s < A.n_src; ++s)
                if (A.src_dom[s] == (SOLID ? 1 : 0) && A.src_q[s] == q) {
                    const T ws = src_value(A, s) / __ldg(scal + (size_t)(SOLID ? SS_AV : SF_AP) * N + q);
                    const T* g = A.src_g + (size_t)s * 2 * n;
                    k[NFLD - NC] = fma(ws, g[i], k[NFLD - NC]);
                    if constexpr (SOLID) k[4] = fma(ws, g[n + i], k[4]);
                }
            if (A.shot_src_q && A.shot_src_dom[shot] == (SOLID ? 1 : 0) && A.shot_src_q[shot] == q) {
                const T ws = shot_src_value(A) / __ldg(scal + (size_t)(SOLID ? SS_AV : SF_AP) * N + q);
                const T* g = A.shot_src_g + (size_t)shot * 2 * n;
                k[NFLD - NC] = fma(ws, g[i], k[NFLD - NC]);
                if constexpr (SOLID) k[4] = fma(ws, g[n + i], k[4]);
            }
            for (int t = A.n_tgt - 1; t >= 0; --t) {
                const TargetT<T>& G = A.tgt[t];
#pragma unroll
                for (int d = 0; d < NFLD; ++d) {
                    const int g = SOLID ? (d < 2 ? 0 : d == 2 ? 1 : 2) : (d < 2 ? 0 : 1);
                    const size_t e = soff + (size_t)(d * n + i) * N + q;
                    const T c = CO[32 * (3 * t + g)];
                    const T u = t == 0 ? src[0][d] : t == 1 ? src[1][d] : G.src ? G.src[e] : T(0);
                    const T v = norm(fma(c, k[d], u));
                    if (real) G.dst[e] = v;
                    if (MODE == MODE_STAGE && t == 0) V[32 * (d * n + i)] = v;
                }
            }
        }
        if constexpr (MODE == MODE_APPLY) return;
        __syncthreads();
    }
    // ---- 3. traces: coefficient l on face j ---------------------------------------------
    // The next stage's blocks may come in where they find idle SMs.  On a fuller
    // GPU they would be placed while this stage still holds its share, unevenly
    // (20 % of a stage at 400 groups), so there they come as blocks leave.
    if (gridDim.x * gridDim.y <= 76) release_successor();
    TeamFaces<T> F;
    F.nF = nF;
    F.npad = npad;
    F.sbase = sbase;
    F.kind = kind;
    F.lq = lq;
    F.hor = faces_h;
    F.other = faces_g;
    F.cd = cd;
    F.tau = tau;
    F.real = real;
    team_traces<T, K, W, SOLID>(op, F, V, A.tr_out + toff, w);
}

// Grid: x over the warps of cells of both domains (fluid, then solid), y over shots.
template <class T, int K, int MODE, int W>
__global__ void __launch_bounds__(32 * W, 32 / W) team_kernel(const StageArgsT<T> A) {
    extern __shared__ __align__(16) unsigned char stage_smem[];
    T* smem = reinterpret_cast<T*>(stage_smem);
    const int gw = A.warp0 + gridDim.x - 1 - blockIdx.x;   // solid cells, the longer ones, first
    if (gw < A.op.n_warps_f) team_cells<T, K, MODE, W, false>(A, gw, blockIdx.y, smem);
    else team_cells<T, K, MODE, W, true>(A, gw, blockIdx.y, smem);
}
