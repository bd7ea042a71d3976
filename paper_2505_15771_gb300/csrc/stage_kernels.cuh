// ERK stage kernels for GB300 (sm_103a) and their launchers, instantiated per
// arithmetic in stage_f64.cu, stage_f32.cu, stage_f2x.cu and stage_tc.cu (so that
// they compile in parallel); the entry points that drive them are in stage.cu.
//
// One stage of Eq. ex_solve (Sec. 4.2) is ONE kernel.  Thread q owns cell q of
// its domain (cells sorted by class, so a warp shares one class and its class
// matrices are read with warp-uniform loads).  The face unknowns are never
// stored: every cell publishes, per local face, two small vectors in the face
// basis psi_l = (rho0 xi)^l (xi along the face in the cell's own
// counter-clockwise orientation; operators.cpp):
//     w     = tau u_T|_F - (dual flux of T on F)      (what the neighbour needs)
//     omega = alpha w - u_T|_F                         (what the cell itself needs)
// where u is p (fluid) or v (solid) and the dual flux is m.n_T or s n_T.  The
// face solve of Eq. ex_solve is block-diagonal; its closed form per
// coefficient is
//     interior:  u_F = (w_T + w_N) / (tau_T + tau_N)
//     boundary:  u_F = 0
//     interface: [p_F; v_F] = A^-1 [w_f; w_s],  A = [tau_f, n^T; -n, tau_s I]
// (rows of the face block of the compact system, Eq. compact_AR, divided by
// the face mass matrix).  So the jump u_F - u_T|_F a cell needs is
// omega + beta * flip(w_N), flip = (-1)^l because the neighbour traverses
// the face in the opposite direction.
//
// A stage thread then: reads its state; forms the exact derivatives of its
// polynomials (sparse, compile-time); lifts each face jump with the class
// matrix Lift_F; scales by the per-cell material factors (inverse mass,
// Eq. mass, folded in); adds point sources; writes the ERK partial sums
// (Eq. ERK_compact with a_{s+1,j} = b_j); and publishes w, omega of the new
// stage value for the next stage (double-buffered traces).
//
// The kernels are templated on the arithmetic: FP64; double-float pairs on
// the FP32 pipes (f2x.cuh, FP64-class accuracy, the single-shot default of
// the benchmark); FP32 for batched shots (shots on blockIdx.y).  Their
// launch parameters (resident blocks, accumulator placement, prefetch hints)
// come from the table in stage_tuning.h.
#pragma once

#include <cuda_runtime.h>

#include <type_traits>

#include "basis.h"
#include "dependent_launch.cuh"
#include "f2x.cuh"
#include "hho_internal.h"
#include "smem_opt_in.h"
#include "stage_launch.h"
#include "stage_tuning.h"

namespace {

template <int K>
struct Dims {
    static constexpr int n = (K + 1) * (K + 2) / 2;
    static constexpr int f = K + 1;
    static constexpr int nP = (n + 3) / 4 * 4;            // padded row lengths (16-byte rows)
    static constexpr int fP = (f + 3) / 4 * 4;
    static constexpr int M0P = (n * n + 3) / 4 * 4;       // class mass block, padded
    static constexpr int FS = 4 + f * nP + n * fP;        // per-face stride: [nx ny 0 0 | Tr | Lift]
    static constexpr int TR = 4;                          // offset of Tr in a face block
    static constexpr int LI = 4 + f * nP;                 // offset of Lift
};

// 16-byte vector loads of class-matrix rows (two doubles or four floats).
template <class T>
struct Vec16;
template <>
struct Vec16<double> {
    static constexpr int w = 2;
    __device__ static void load(const double* p, double* o) {
        const double2 v = __ldg(reinterpret_cast<const double2*>(p));
        o[0] = v.x;
        o[1] = v.y;
    }
};
template <>
struct Vec16<float> {
    static constexpr int w = 4;
    __device__ static void load(const float* p, float* o) {
        const float4 v = __ldg(reinterpret_cast<const float4*>(p));
        o[0] = v.x;
        o[1] = v.y;
        o[2] = v.z;
        o[3] = v.w;
    }
};

template <>
struct Vec16<f2x> {
    static constexpr int w = 2;
    __device__ static void load(const f2x* p, f2x* o) {
        const float4 v = __ldg(reinterpret_cast<const float4*>(p));
        o[0] = f2x(v.x, v.y);
        o[1] = f2x(v.z, v.w);
    }
};

// Operator data in the arithmetic type T (FP64, its FP32 copy, or its
// double-float copy).
template <class T>
struct OpData;
template <>
struct OpData<double> {
    __device__ static const double* cls(const DevOps& o) { return o.cls_dbl; }
    __device__ static const double* scal_f(const DevOps& o) { return o.scal_f; }
    __device__ static const double* scal_s(const DevOps& o) { return o.scal_s; }
    __device__ static const double* beta_f(const DevOps& o) { return o.beta_f; }
    __device__ static const double* beta_s(const DevOps& o) { return o.beta_s; }
    __device__ static const double* if_coef(const DevOps& o) { return o.if_coef; }
};
template <>
struct OpData<float> {
    __device__ static const float* cls(const DevOps& o) { return o.cls_f32; }
    __device__ static const float* scal_f(const DevOps& o) { return o.scal_f_f32; }
    __device__ static const float* scal_s(const DevOps& o) { return o.scal_s_f32; }
    __device__ static const float* beta_f(const DevOps& o) { return o.beta_f_f32; }
    __device__ static const float* beta_s(const DevOps& o) { return o.beta_s_f32; }
    __device__ static const float* if_coef(const DevOps& o) { return o.if_coef_f32; }
};

template <>
struct OpData<f2x> {
    __device__ static const f2x* cls(const DevOps& o) { return o.cls_x; }
    __device__ static const f2x* scal_f(const DevOps& o) { return o.scal_f_x; }
    __device__ static const f2x* scal_s(const DevOps& o) { return o.scal_s_x; }
    __device__ static const f2x* beta_f(const DevOps& o) { return o.beta_f_x; }
    __device__ static const f2x* beta_s(const DevOps& o) { return o.beta_s_x; }
    __device__ static const f2x* if_coef(const DevOps& o) { return o.if_coef_x; }
};

// d/dX of a polynomial in the scaled-monomial basis (exact, compile-time sparse).
template <class T, int K>
__device__ __forceinline__ void ddx(const T* u, T* out) {
#pragma unroll
    for (int i = 0; i < Dims<K>::n; ++i) {
        const int a = ea(i), b = eb(i);
        if (a + 1 + b <= K) {
            const int s = eidx(a + 1, b);
            out[i] = (a == 0) ? u[s] : mulc(float(a + 1), u[s]);
        } else {
            out[i] = T(0);
        }
    }
}
template <class T, int K>
__device__ __forceinline__ void ddy(const T* u, T* out) {
#pragma unroll
    for (int i = 0; i < Dims<K>::n; ++i) {
        const int a = ea(i), b = eb(i);
        if (a + b + 1 <= K) {
            const int s = eidx(a, b + 1);
            out[i] = (b == 0) ? u[s] : mulc(float(b + 1), u[s]);
        } else {
            out[i] = T(0);
        }
    }
}
// out += d/dX u  (or d/dY u)
template <class T, int K>
__device__ __forceinline__ void add_ddx(const T* u, T* out) {
#pragma unroll
    for (int i = 0; i < Dims<K>::n; ++i) {
        const int a = ea(i), b = eb(i);
        if (a + 1 + b <= K) {
            const int s = eidx(a + 1, b);
            out[i] = (a == 0) ? out[i] + u[s] : fmac(float(a + 1), u[s], out[i]);
        }
    }
}
template <class T, int K>
__device__ __forceinline__ void add_ddy(const T* u, T* out) {
#pragma unroll
    for (int i = 0; i < Dims<K>::n; ++i) {
        const int a = ea(i), b = eb(i);
        if (a + b + 1 <= K) {
            const int s = eidx(a, b + 1);
            out[i] = (b == 0) ? out[i] + u[s] : fmac(float(b + 1), u[s], out[i]);
        }
    }
}

// ---- face policies ---------------------------------------------------------------
// GenericFace: any polygon face; normals and class matrices read at run time,
// every matrix entry used (no run-time tests on floating-point values).
// RectAxis<A>: the faces of an axis-aligned rectangle with one orientation,
// A = 0 horizontal (faces 0 bottom and 2 top, normal (0, s)), A = 1 vertical
// (faces 1 right and 3 left, normal (s, 0)); the sign s = +-1 is a run-time
// argument, the parity sparsity of Tr and Lift is compile-time and entries
// outside the pattern are never loaded.  One body per orientation, looped
// over its two faces, keeps the kernel's instruction footprint small.
// SquareAxis<A>: the faces of a square cell; their traces are Horner sums
// with compile-time coefficients (trace_square) and Tr is never read, and
// their lifting matrices also vanish where the exponent along the face
// exceeds the face coefficient's degree by 2 (checked when the class is
// built, up to k = 3).
// PolyAxis<A>: a horizontal or vertical face of any polygon; every Lift entry
// is used, but X^a Y^b traces to degree a only where Y is constant (b where X
// is), so half of Tr is empty, and one component of the flux is enough.
struct GenericFace {
    static constexpr bool axis = false;
    static constexpr bool rect = false;
    static constexpr bool square = false;
    static constexpr bool horiz = false;
    __host__ __device__ static constexpr bool tr_nz(int, int) { return true; }
    __host__ __device__ static constexpr bool lift_nz(int, int) { return true; }
};
template <int AX>
struct PolyAxis {
    static constexpr bool axis = true;
    static constexpr bool rect = false;
    static constexpr bool square = false;
    static constexpr bool horiz = AX == 0;
    __host__ __device__ static constexpr bool tr_nz(int l, int i) { return (horiz ? ea(i) : eb(i)) >= l; }
    __host__ __device__ static constexpr bool lift_nz(int, int) { return true; }
};
template <int AX>
struct RectAxis {
    static constexpr bool axis = true;
    static constexpr bool rect = true;
    static constexpr bool square = false;
    static constexpr bool horiz = AX == 0;
    __host__ __device__ static constexpr int e(int i) { return horiz ? ea(i) : eb(i); }
    __host__ __device__ static constexpr bool tr_nz(int l, int i) { return e(i) == l; }
    __host__ __device__ static constexpr bool lift_nz(int i, int l) { return ((e(i) + l) % 2) == 0; }
};
template <int AX>
struct SquareAxis : RectAxis<AX> {
    static constexpr bool square = true;
    __host__ __device__ static constexpr bool lift_nz(int i, int l) {
        return RectAxis<AX>::lift_nz(i, l) && RectAxis<AX>::e(i) - l != 2;
    }
};

// The FP64 kernel is bound by the FP64 pipe, and its arithmetic is arranged to
// issue the fewest instructions: tau multiplies a cell's lifted jumps once
// instead of every pair's sigma and delta, and axis-aligned faces of polygons
// have bodies of their own that skip the empty half of their trace matrices
// (k = 3 stages of 524,288 cells: hanging nodes 754 -> 630 us, triangles
// 857 -> 752; the 680 x 340 hybrid mesh 324 -> 305).  The other types are bound
// by memory and latency and lost 5 to 10 % to the longer code and the extra
// accumulators, so they keep the compact form.
template <class T>
struct Fp64Form {
    static constexpr bool value = std::is_same<T, double>::value;
};

// Class matrices of the double-float kernel are read from a per-warp copy in
// shared memory (its many FP32 instructions per matrix entry would otherwise
// wait on L1 misses: the streamed state and traces evict the class rows); the
// FP64 and FP32 kernels read them through the read-only data path.
template <class T>
struct ClsSmem {
    static constexpr bool value = false;
};
template <>
struct ClsSmem<f2x> {
    static constexpr bool value = true;
};
template <class T>
__device__ __forceinline__ void cls_row(const T* p, T* o) {
    if constexpr (ClsSmem<T>::value) {
        const float4 v = *reinterpret_cast<const float4*>(p);   // two pairs
        o[0] = T(v.x, v.y);
        o[1] = T(v.z, v.w);
    } else {
        Vec16<T>::load(p, o);
    }
}
template <class T>
__device__ __forceinline__ T cls_val(const T* p) {
    if constexpr (ClsSmem<T>::value) return *p;
    else return __ldg(p);
}

// y[l] = sum_i Tr[l][i] x[i] over the policy's pattern.  Each row is read in
// 16-byte chunks; a chunk with no entry in the pattern is not loaded.
template <class T, int K, class P>
__device__ __forceinline__ void trace_apply(const T* __restrict__ Tr, const T* x, T* y) {
    constexpr int n = Dims<K>::n, f = Dims<K>::f, nP = Dims<K>::nP, w = Vec16<T>::w;
#pragma unroll
    for (int l = 0; l < f; ++l) {
        T row[nP];
#pragma unroll
        for (int c0 = 0; c0 < nP; c0 += w) {
            bool need = false;
#pragma unroll
            for (int e = 0; e < w; ++e) need = need || (c0 + e < n && P::tr_nz(l, c0 + e));
            if (need) cls_row<T>(Tr + l * nP + c0, row + c0);
        }
        T acc = T(0);
#pragma unroll
        for (int i = 0; i < n; ++i)
            if (P::tr_nz(l, i)) acc = fma(row[i], x[i], acc);
        y[l] = acc;
    }
}
// Traces on a square's face with outward normal sign sg (faces 0 and 3:
// -1, faces 1 and 2: +1): the monomial with exponent l along the face and m
// across it traces to s_t^l (sg rho0)^m psi_l, s_t = -sg on horizontal and
// sg on vertical faces, so y[l] = s_t^l sum_m (sg rho0)^m x[(l, m)] by
// Horner's rule (K - l multiply-adds).
// sg * rho0 in T; the double-float split is formed at compile time (a
// run-time split would issue FP64 instructions on the slow FP64 pipe)
template <class T>
__device__ __forceinline__ T signed_face_rho(int sg) {
    return T(sg > 0 ? FACE_RHO : -FACE_RHO);
}
template <>
__device__ __forceinline__ f2x signed_face_rho<f2x>(int sg) {
    constexpr float hi = (float)FACE_RHO;
    constexpr float lo = (float)(FACE_RHO - (double)hi);
    return sg > 0 ? f2x(hi, lo) : f2x(-hi, -lo);
}
template <class T, int K, bool HORIZ>
__device__ __forceinline__ void trace_square(const T* x, T* y, int sg) {
    const T c = signed_face_rho<T>(sg);
    const bool flip = HORIZ ? sg > 0 : sg < 0;   // s_t = -1
#pragma unroll
    for (int l = 0; l <= K; ++l) {
        T acc = x[HORIZ ? eidx(l, K - l) : eidx(K - l, l)];
#pragma unroll
        for (int m = K - l - 1; m >= 0; --m) acc = fma(c, acc, x[HORIZ ? eidx(l, m) : eidx(m, l)]);
        y[l] = ((l & 1) && flip) ? -acc : acc;
    }
}
template <class T, int K, class P>
__device__ __forceinline__ void face_trace_apply(const T* __restrict__ Tr, const T* x, T* y, int sg) {
    if constexpr (P::square) trace_square<T, K, P::horiz>(x, y, sg);
    else trace_apply<T, K, P>(Tr, x, y);
}
// y[i] = sum_l L[i][l] j[l] over the policy's pattern (rows of fP entries).
template <class T, int K, class P>
__device__ __forceinline__ void lift_apply(const T* __restrict__ L, const T* j, T* y) {
    constexpr int n = Dims<K>::n, f = Dims<K>::f, fP = Dims<K>::fP, w = Vec16<T>::w;
#pragma unroll
    for (int i = 0; i < n; ++i) {
        T row[fP];
#pragma unroll
        for (int c0 = 0; c0 < fP; c0 += w) {
            bool need = false;
#pragma unroll
            for (int e = 0; e < w; ++e) need = need || (c0 + e < f && P::lift_nz(i, c0 + e));
            if (need) cls_row<T>(L + i * fP + c0, row + c0);
        }
        T acc = T(0);
#pragma unroll
        for (int l = 0; l < f; ++l)
            if (P::lift_nz(i, l)) acc = fma(row[l], j[l], acc);
        y[i] = acc;
    }
}
// Rectangle faces: one body per orientation looped over its two faces
// (compact code: the double-float kernel is bound by instruction fetch
// otherwise), or the four faces unrolled with constant signs (the FP64
// kernel schedules better fully unrolled); per arithmetic and k from the
// tuning table.

// Where a stage thread keeps its 3n (fluid) or 5n (solid) accumulators.  In
// registers they do not fit the 64-register budget of 8 resident blocks and
// spill to local memory, whose footprint (over 400 bytes a thread) exceeds
// L1.  With AccSmem the block's dynamic shared memory holds them instead,
// thread-major with an odd stride in elements (no bank conflicts).  That made
// the FP32 kernel about 20 % faster at k = 3 and the double-float one 7 % at
// k = 2.  FP64 is indifferent (k = 2, 1024 x 512: 224.0 us either way; k = 3 at
// 4 blocks, 680 x 340 hybrid: 275.6 us against 275.7 in registers), and
// double-float k = 3 gains nothing (4 blocks).
template <class T>
struct Tuned;
template <>
struct Tuned<double> {
    static constexpr StageTuning t = TUNED_F64;
};
template <>
struct Tuned<float> {
    static constexpr StageTuning t = TUNED_F32;
};
template <>
struct Tuned<f2x> {
    static constexpr StageTuning t = TUNED_F2X;
};
template <class T, int K>
struct RectLoop {
    static constexpr bool value = Tuned<T>::t.rect_loop[K - 1] != 0;
};
template <class T, int K>
struct AccSmem {
    static constexpr bool value = Tuned<T>::t.acc_smem[K - 1] != 0;
};
template <int K>
__host__ __device__ constexpr int acc_stride() {
    return (5 * Dims<K>::n) | 1;
}

// y += s * x for a run-time sign s = +-1
template <int NN, class T>
__device__ __forceinline__ void add_signed(const T* x, T* y, int s) {
#pragma unroll
    for (int i = 0; i < NN; ++i) y[i] += (s > 0) ? x[i] : -x[i];
}

template <int NV, class T>
__device__ __forceinline__ void load_state(const T* src, int N, int q, int first, T* u) {
#pragma unroll
    for (int i = 0; i < NV; ++i) u[i] = src[(size_t)(first + i) * N + q];
}

// ERK targets: dst = src + coef * scale_g * k, where g = GRP(i) picks the
// per-cell material factor of value i (the inverse mass, folded into the
// target coefficient).  Target 0 is kept in `k` (overwritten).  `off` is the
// offset of this shot's domain block.
//
// The sources are read TARGET_BATCH at a time before any of the batch is
// stored: a target may be its own source (the ERK accumulator), so the compiler
// keeps every later load behind every earlier store, and value by value the
// targets were 100 memory round trips in a row for a k = 3 solid cell.  Stage
// kernel, us, by batch 1 | 5 | 10 | 16 | 25: FP32, 16 shots of the 680 x 340
// k = 3 hybrid mesh 1174 | 892 | 866 | 869 | 908; FP32, 21 shots of the 331 x 167
// k = 2 hanging mesh 318 | 288 | 283 | 279 | 292; double-float, 1024 x 512,
// k = 2: 210 | - | 172 | 174 (15); FP64 the same: 247 | 237 (3) | 238.
constexpr int TARGET_BATCH = 10;
template <int NV, class GRP, class T>
__device__ __forceinline__ void write_targets(const StageArgsT<T>& A, int N, size_t off, int q, T* k, const T* sc) {
    constexpr int B = TARGET_BATCH;
#pragma unroll 1
    for (int t = A.n_tgt - 1; t >= 0; --t) {
        const TargetT<T> G = A.tgt[t];
        const T c[3] = {G.coef * sc[0], G.coef * sc[1], G.coef * sc[2]};
        T* dst = G.dst + off;
        const T* src = G.src + off;
        const bool add = G.src != nullptr;
#pragma unroll
        for (int i0 = 0; i0 < NV; i0 += B) {
            T s[B];
            if (add) {
#pragma unroll
                for (int b = 0; b < B; ++b)
                    if (i0 + b < NV) s[b] = src[(size_t)(i0 + b) * N + q];
            }
#pragma unroll
            for (int b = 0; b < B; ++b) {
                const int i = i0 + b;
                if (i >= NV) continue;
                const T v = norm(add ? fma(c[GRP::g(i)], k[i], s[b]) : c[GRP::g(i)] * k[i]);
                dst[(size_t)i * N + q] = v;
                if (t == 0) k[i] = v;
            }
        }
    }
}
template <int n>
struct FluidGroups {   // [m_x, m_y | p]
    __host__ __device__ static constexpr int g(int i) { return i < 2 * n ? 0 : 1; }
};
template <int n>
struct SolidGroups {   // [s_xx, s_yy | s_xy | v_x, v_y]
    __host__ __device__ static constexpr int g(int i) { return i < 2 * n ? 0 : (i < 3 * n ? 1 : 2); }
};

// Per-thread view of one (cell, shot): class layout and this shot's buffers.
template <class T>
struct CellCtx {
    int q, lq, nF, npad, sbase, N, SF, SS, FS;
    uint32_t hor, ver; // axis-aligned faces (CI_HOR, CI_VER)
    const T* cd;       // class face blocks
    T tau;
    const T* trf_in;   // this shot's trace buffers (fluid part, solid part)
    const T* trs_in;
    T* trf_out;
    T* trs_out;
};

// The faces of a polygon.  FP64: horizontal ones, then vertical ones (each with
// the sign of its normal), then the others; the order is part of the arithmetic,
// and the team form adds the faces in the same one.  Other types: in local order
// through the general body.
template <class T, class H, class V, class O>
__device__ __forceinline__ void for_faces(const CellCtx<T>& c, H hor, V ver, O other) {
    if constexpr (Fp64Form<T>::value) {
#pragma unroll 1
        for (uint32_t m = c.hor; m; m &= m - 1) {
            const int j = __ffs(m) - 1;
            hor(j, is_negative(cls_val(c.cd + j * c.FS + 1)) ? -1 : 1);
        }
#pragma unroll 1
        for (uint32_t m = c.ver; m; m &= m - 1) {
            const int j = __ffs(m) - 1;
            ver(j, is_negative(cls_val(c.cd + j * c.FS)) ? -1 : 1);
        }
        const uint32_t done = c.hor | c.ver;
#pragma unroll 1
        for (int j = 0; j < c.nF; ++j)
            if (!((done >> j) & 1)) other(j);
    } else {
#pragma unroll 1
        for (int j = 0; j < c.nF; ++j) other(j);
    }
}

// ---- L2 prefetch hints -------------------------------------------------------------
// A stage thread reads its cell's state, its faces' own traces, its
// neighbours' traces and the targets' sources in about twenty dependent
// rounds, and with 64 registers it cannot hold more of them in flight.
// Prefetch hints take no register and bring the lines of later rounds into
// L2 early.  Mask bits: 1 state, 2 own traces and face tables, 4 neighbour
// traces, 8 target sources, all at the start of the cell; 16 target sources
// and 32 neighbour traces just before the face loop.  Stage kernel, us, by mask:
// FP32, 16 shots of the 680 x 340 k = 3 hybrid mesh 0: 944, 34: 902, 51: 843;
// double-float, 1024 x 512, k = 2, 0: 169.9, 34: 169.4, 50: 172, 51: 174;
// FP64 the same 0: 225, 34: 230, 50: 236 (its pipe binds, and the hints are
// instructions).  Register accumulators (spilled) lost with every mask.
template <class T, int K>
struct L2Prefetch {
    static constexpr int mask = Tuned<T>::t.prefetch[K - 1];
};

__device__ __forceinline__ void pf_l2(const void* p) { asm volatile("prefetch.L2 [%0];" ::"l"(p)); }

// The warp's 32-element runs base + a * stride (a < narr), spread over the
// lanes: every 128-byte line a run touches, unaligned runs included.
template <class E>
__device__ __forceinline__ void pf_runs(const E* base, size_t stride, int narr, int lane) {
    constexpr int BYTES = 32 * (int)sizeof(E), LINES = BYTES / 128 + 1;
    for (int e = lane; e < narr * LINES; e += 32) {
        const int a = e / LINES, m = e - a * LINES;
        pf_l2(reinterpret_cast<const char*>(base + (size_t)a * stride) + min(m * 128, BYTES - 1));
    }
}

// WHERE 0: at the start of the cell; 1: before the face loop.  NV state
// values per cell, NW published traces per face slot (w first, then omega).
template <class T, int K, int NV, int NW, int WHERE, bool TARGETS>
__device__ __forceinline__ void prefetch_cell(const StageArgsT<T>& A, const CellCtx<T>& c, size_t soff, const T* tr,
                                              int S, const int* nbt, const T* bet, int nfaces) {
    constexpr int PF = L2Prefetch<T, K>::mask;
    const int lane = c.q & 31;
    if constexpr (WHERE == 0 && (PF & 1)) pf_runs(A.inp + soff + (c.q - lane), c.N, NV, lane);
    if constexpr (WHERE == 0 && (PF & 2)) {
        for (int j = 0; j < nfaces; ++j) {
            const int s0 = c.sbase + j * c.npad + c.lq - lane;
            pf_runs(tr + (size_t)NW * S + s0, S, NW, lane);
            pf_runs(nbt + s0, 0, 1, lane);
            pf_runs(bet + s0, 0, 1, lane);
        }
    }
    if constexpr ((WHERE == 0 && (PF & 4)) || (WHERE == 1 && (PF & 32))) {
        for (int j = 0; j < nfaces; ++j) {
            const int nb = __ldg(nbt + c.sbase + j * c.npad + c.lq);
            if (nb >= 0)
                for (int l = 0; l < NW; ++l) pf_l2(tr + (size_t)l * S + nb);
        }
    }
    if constexpr (TARGETS && ((WHERE == 0 && (PF & 8)) || (WHERE == 1 && (PF & 16)))) {
        for (int t = 0; t < A.n_tgt; ++t)
            if (A.tgt[t].src) pf_runs(A.tgt[t].src + soff + (c.q - lane), c.N, NV, lane);
    }
}

// ---- point-source wavelets ----------------------------------------------------------
// Ricker wavelet amp (1 - 2 a^2) exp(-a^2), a = pi f0 (t - t0), at the stage
// time.  With a device clock (graph replay) the time is (t0 + n dt) + c dt
// formed with rounded operations in the host's order, and the wavelet is
// evaluated here; otherwise the host's values are used.
__device__ __forceinline__ double stage_time(const StageClock* clk, double dt, double c) {
    const double tn = __dadd_rn(clk->t0, __dmul_rn((double)clk->step, dt));
    return __dadd_rn(tn, __dmul_rn(c, dt));
}
__device__ __forceinline__ double ricker_dev(double t, double f0, double t0, double amp) {
    const double a = __dmul_rn(__dmul_rn(M_PI, f0), __dadd_rn(t, -t0));
    const double a2 = __dmul_rn(a, a);
    return __dmul_rn(__dmul_rn(amp, __dadd_rn(1.0, -__dmul_rn(2.0, a2))), exp(-a2));
}
template <class T>
__device__ __forceinline__ T src_value(const StageArgsT<T>& A, int s) {
    if (!A.clock) return A.src_w[s];
    return T(ricker_dev(stage_time(A.clock, A.dt, A.c_stage), A.src_f0[s], A.src_t0[s], A.src_amp[s]));
}
template <class T>
__device__ __forceinline__ T shot_src_value(const StageArgsT<T>& A) {
    if (!A.clock) return A.shot_src_w;
    return T(ricker_dev(stage_time(A.clock, A.dt, A.c_stage), A.shot_f0, A.shot_t0, A.shot_amp));
}

// ---- adjoint gradients (MODE_GRAD) ---------------------------------------------------
// A cell's sums of products: FP64 for FP64 values; for FP32 values double-float
// (48 bits, on the FP32 pipes: an FP64 sum of FP32 products would spend most of its
// time in conversions on the FP64 pipe) of values that are first divided by a
// power of two near their largest (Range), which is put back in FP64: a pair has
// FP32's exponents, and the product of two FP32 values needs FP64's.
template <class T>
struct Wide {
    using type = double;
};
template <>
struct Wide<float> {
    using type = f2x;
};
// The largest magnitude of the values shown to it as a power of two: factor()
// brings them to 4 or less (below 2^-125, to 2 or less), exponent() undoes that.
template <class T>
struct Range;
template <>
struct Range<double> {   // FP64 products stay in range unscaled
    __device__ void add(double) {}
    __device__ double factor() const { return 1.0; }
    __device__ int exponent() const { return 0; }
};
template <>
struct Range<float> {
    uint32_t m = 0;
    __device__ void add(float x) { m = max(m, __float_as_uint(x) & 0x7fffffffu); }
    __device__ int biased() const { return min(max((int)(m >> 23), 1), 253); }
    __device__ float factor() const { return __uint_as_float((uint32_t)(254 - biased()) << 23); }
    __device__ int exponent() const { return biased() - 127; }
};
// x[0..N) divided by a power of two near the largest; returns its exponent
template <int N, class T>
__device__ __forceinline__ int to_unit(T* x) {
    Range<T> r;
#pragma unroll
    for (int i = 0; i < N; ++i) r.add(x[i]);
    const T s = r.factor();
#pragma unroll
    for (int i = 0; i < N; ++i) x[i] *= s;
    return r.exponent();
}
// x 2^e, |e| < 512, for x zero, not finite, or a double-float value (no FP64 instruction)
__device__ __forceinline__ double times_pow2(double x, int e) {
    const int h = __double2hiint(x);
    const uint32_t b = ((uint32_t)h >> 20) & 0x7ffu;
    return b - 1u < 0x7feu ? __hiloint2double(h + e * (1 << 20), __double2loint(x)) : x;
}
__device__ __forceinline__ double leading(double x) { return x; }
__device__ __forceinline__ float leading(f2x x) { return x.hi; }
__device__ __forceinline__ double widen(double x) { return x; }
__device__ __forceinline__ f2x widen(float x) { return f2x(x, 0.0f); }
template <class T>
struct WideData;   // operator data in the wide type
template <>
struct WideData<double> {
    __device__ static const double* beta_f(const DevOps& o) { return o.beta_f; }
    __device__ static const double* beta_s(const DevOps& o) { return o.beta_s; }
    __device__ static const double* cls(const DevOps& o) { return o.cls_dbl; }
};
template <>
struct WideData<float> {
    __device__ static const f2x* beta_f(const DevOps& o) { return o.beta_f_x; }
    __device__ static const f2x* beta_s(const DevOps& o) { return o.beta_s_x; }
    __device__ static const f2x* cls(const DevOps& o) { return o.cls_x; }
};

// M0's parity pattern on rectangles: it couples equal parities of both exponents.
__host__ __device__ constexpr bool mass_nz(int i, int j) {
    return ((ea(i) + ea(j)) & 1) == 0 && ((eb(i) + eb(j)) & 1) == 0;
}
// y = M0 x with the class mass matrix (stored n x n, rows unpadded), in the
// wide type: mu = S M z is a difference of large terms where M0 is badly
// conditioned, so FP32 matrix entries or sums would cost the FP32 gradient
// about a factor of two in accuracy.
template <class T, int K, bool RECT, class W>
__device__ __forceinline__ void mass_apply(const W* __restrict__ M0, const T* x, W* y) {
    constexpr int n = Dims<K>::n;
#pragma unroll
    for (int i = 0; i < n; ++i) {
        W s(0);
#pragma unroll
        for (int j = 0; j < n; ++j)
            if (!RECT || mass_nz(i, j)) s = fma(__ldg(M0 + i * n + j), widen(x[j]), s);
        y[i] = s;
    }
}
template <class T, int K, class W>
__device__ __forceinline__ void mass_apply(const W* __restrict__ M0, bool rect, const T* x, W* y) {
    if (rect) mass_apply<T, K, true>(M0, x, y);
    else mass_apply<T, K, false>(M0, x, y);
}
template <class T, int K, class W>
__device__ __forceinline__ W coef_dot(const T* x, const W* y) {
    W s(0);
#pragma unroll
    for (int i = 0; i < Dims<K>::n; ++i) s = fma(widen(x[i]), y[i], s);
    return s;
}

// sum over NC fields of z^T M0 g of a cell (z with stride N): the source cells
// of the wavelet gradient only.
template <class T, int K, int NC>
__device__ __noinline__ double wide_form(const DevOps& op, const int* ci, const T* z, int N, const T* g) {
    using W = typename Wide<T>::type;
    constexpr int n = Dims<K>::n;
    const W* M0 = WideData<T>::cls(op) + __ldg(ci + CI_DOFF);
    Range<T> rz, rg;
    for (int i = 0; i < NC * n; ++i) {
        rz.add(z[(size_t)i * N]);
        rg.add(g[i]);
    }
    W acc(0);
    for (int e = 0; e < NC; ++e)
        for (int i = 0; i < n; ++i) {
            W y(0);
            for (int j = 0; j < n; ++j) y = fma(M0[i * n + j], widen(z[(size_t)(e * n + j) * N] * rz.factor()), y);
            acc = fma(y, widen(g[e * n + i] * rg.factor()), acc);
        }
    return times_pow2(to_f64(acc), rz.exponent() + rg.exponent());
}

// The integral over a face of unit length of the product of two functions
// given by their face coefficients:
// (psi_l, psi_m) = rho0^(l+m) / (l+m+1) on a face of unit length for even
// l + m, else 0 (constants of the unrolled sums).
__host__ __device__ constexpr double face_gram(int l, int m) {
    if ((l + m) & 1) return 0.0;
    double r = 1.0;
    for (int e = 0; e < l + m; ++e) r *= FACE_RHO;
    return r / (l + m + 1);
}
// a gram entry in the wide type; called with unrolled constants, so that the
// double-float split is folded and issues no FP64 instruction
template <class W>
__device__ __forceinline__ W gram_const(double v) {
    return W(v);
}
template <int K, class W>
__device__ __forceinline__ W face_inner(const W* a, const W* b, W acc) {
    constexpr int f = Dims<K>::f;
#pragma unroll
    for (int l = 0; l < f; ++l) {
        W t = l == 0 ? b[l] : gram_const<W>(face_gram(l, l)) * b[l];   // (psi_0, psi_0) = 1
#pragma unroll
        for (int m = 0; m < f; ++m)
            if (m != l && ((l + m) & 1) == 0) t = fma(gram_const<W>(face_gram(l, m)), b[m], t);
        acc = fma(a[l], t, acc);
    }
    return acc;
}

// Jump of the primal trace on local face j in the wide type, from the
// published traces tr (fluid part then solid part) and interface
// coefficients `co6`; NC = 1 component in a fluid cell, 2 in a solid cell.
// Returns the exponent of the power of two that jmp is divided by (Range).
template <class T, int K, int NC, class W>
__device__ __forceinline__ int wide_jump(const DevOps& op, const T* tr, const double* co6, int slot, int nb, W* jmp) {
    constexpr int f = Dims<K>::f;
    const size_t S = NC == 1 ? op.SF : op.SS;
    const T* trf = tr;
    const T* trs = tr + (size_t)2 * f * op.SF;
    const T* own = NC == 1 ? trf : trs;
    Range<T> range;
    T om[NC * f];
#pragma unroll
    for (int i = 0; i < NC * f; ++i) range.add(om[i] = own[(NC * f + i) * S + slot]);
    auto start = [&](T s) {
#pragma unroll
        for (int i = 0; i < NC * f; ++i) jmp[i] = widen(om[i] * s);
        return s;
    };
    if (nb >= 0) {
        const W be = __ldg((NC == 1 ? WideData<T>::beta_f(op) : WideData<T>::beta_s(op)) + slot);
        T w[NC * f];
#pragma unroll
        for (int i = 0; i < NC * f; ++i) range.add(leading(be) * (w[i] = own[i * S + nb]));
        const T s = start(range.factor());
#pragma unroll
        for (int i = 0; i < NC * f; ++i) jmp[i] = ((i % f) & 1) ? fma(-be, widen(w[i] * s), jmp[i]) : fma(be, widen(w[i] * s), jmp[i]);
    } else if (nb < NB_BOUNDARY) {
        const int r = -2 - nb;
        const int no = __ldg(op.if_nb + r);
        const double* co = co6 + 6 * r;
        if constexpr (NC == 1) {
            const W bx(__ldg(co + 1)), by(__ldg(co + 2));
            T wx[f], wy[f];
#pragma unroll
            for (int l = 0; l < f; ++l) {
                range.add(leading(bx) * (wx[l] = trs[(size_t)l * op.SS + no]));
                range.add(leading(by) * (wy[l] = trs[(size_t)(f + l) * op.SS + no]));
            }
            const T s = start(range.factor());
#pragma unroll
            for (int l = 0; l < f; ++l) {
                const W ws = fma(bx, widen(wx[l] * s), by * widen(wy[l] * s));
                jmp[l] = (l & 1) ? jmp[l] - ws : jmp[l] + ws;
            }
        } else {
            const W b0(__ldg(co + 4)), b1(__ldg(co + 5));
            T wf[f];
#pragma unroll
            for (int l = 0; l < f; ++l) {
                wf[l] = trf[(size_t)l * op.SF + no];
                range.add(leading(b0) * wf[l]);
                range.add(leading(b1) * wf[l]);
            }
            const T s = start(range.factor());
#pragma unroll
            for (int l = 0; l < f; ++l) {
                const W w = widen(wf[l] * s);
                jmp[l] = (l & 1) ? fma(-b0, w, jmp[l]) : fma(b0, w, jmp[l]);
                jmp[f + l] = (l & 1) ? fma(-b1, w, jmp[f + l]) : fma(b1, w, jmp[f + l]);
            }
        }
    } else {
        start(range.factor());
    }
    return range.exponent();
}

// Stabilisation-weight part of one backward stage: gstab += w sum_F |F|/h
// (jump of Y, jump of z)_F over the cell's faces.
template <class T, int K, int NC>
__device__ __forceinline__ void tau_grad(const StageArgsT<T>& A, const GradArgsT<T>& G, const CellCtx<T>& c,
                                         const int* ci, int g) {
    using W = typename Wide<T>::type;
    constexpr int f = Dims<K>::f, FS = Dims<K>::FS;
    const DevOps& op = A.op;
    const double* cd = op.cls_dbl + __ldg(ci + CI_DOFF) + Dims<K>::M0P;
    double acc = 0.0;
#pragma unroll 1
    for (int j = 0; j < c.nF; ++j) {
        const int slot = c.sbase + j * c.npad + c.lq;
        const int nb = __ldg((NC == 1 ? op.nb_f : op.nb_s) + slot);
        W jy[NC * f], jz[NC * f];
        const int ey = wide_jump<T, K, NC, W>(op, A.tr_in, op.if_coef, slot, nb, jy);
        const int ez = wide_jump<T, K, NC, W>(op, G.tr_z, G.if_coef_z, slot, nb, jz);
        W sum(0);
#pragma unroll
        for (int e = 0; e < NC; ++e) sum = face_inner<K, W>(jy + e * f, jz + e * f, sum);
        acc = fma(__ldg(cd + j * FS + 2), times_pow2(to_f64(sum), ey + ez), acc);   // |F| / h
    }
    G.gstab[g] = fma(G.w, acc, G.gstab[g]);
}

// Gradients of one fluid cell: U holds the raw rates [grad p (2), div m].
// With mu = w S M z, mu^T raw is a sum of z^T M0 raw per field.
template <class T, int K>
__device__ __forceinline__ void fluid_grad(const StageArgsT<T>& A, const GradArgsT<T>& G, const CellCtx<T>& c,
                                           const int* ci, bool rect, const T* U) {
    constexpr int n = Dims<K>::n;
    using W = typename Wide<T>::type;
    const int q = c.q;
    const W* M0 = WideData<T>::cls(A.op) + __ldg(ci + CI_DOFF);
    double qf[3];
#pragma unroll
    for (int fld = 0; fld < 3; ++fld) {
        T u[n], z[n];
        W y[n];
#pragma unroll
        for (int i = 0; i < n; ++i) u[i] = U[fld * n + i];
        const int eu = to_unit<n>(u);
        mass_apply<T, K>(M0, rect, u, y);
        load_state<n>(G.z, c.N, q, fld * n, z);
        const int ez = to_unit<n>(z);
        qf[fld] = times_pow2(to_f64(coef_dot<T, K, W>(z, y)), eu + ez);
    }
    const double cm = G.mass_f[q], cp = G.mass_f[c.N + q];
    G.grad_f[q] = fma(-G.w * cm, qf[0] + qf[1], G.grad_f[q]);
    G.grad_f[c.N + q] = fma(G.w * cp, qf[2], G.grad_f[c.N + q]);
    if (G.wgrad)
        for (int s = 0; s < A.n_src; ++s)
            if (A.src_dom[s] == 0 && A.src_q[s] == q)
                G.wgrad[s] = G.w * cp * wide_form<T, K, 1>(A.op, ci, G.z + (size_t)2 * n * c.N + q, c.N,
                                                           A.src_g + (size_t)s * 2 * n);
}

// Gradients of one solid cell: U holds the raw rates [e_xx, e_yy, e_xy, div s (2)].
template <class T, int K>
__device__ __forceinline__ void solid_grad(const StageArgsT<T>& A, const GradArgsT<T>& G, const CellCtx<T>& c,
                                           const int* ci, bool rect, const T* U) {
    constexpr int n = Dims<K>::n;
    using W = typename Wide<T>::type;
    const int q = c.q;
    const size_t N = c.N;
    const W* M0 = WideData<T>::cls(A.op) + __ldg(ci + CI_DOFF);
    const T* zb = G.z + (size_t)3 * n * A.op.Nf;
    double q00, q01, q10, q11;   // q_ab = z_a^T M0 raw_b
    {
        T u[n], z[n];
        W y0[n], y1[n];
#pragma unroll
        for (int i = 0; i < n; ++i) u[i] = U[i];
        const int e0 = to_unit<n>(u);
        mass_apply<T, K>(M0, rect, u, y0);
#pragma unroll
        for (int i = 0; i < n; ++i) u[i] = U[n + i];
        const int e1 = to_unit<n>(u);
        mass_apply<T, K>(M0, rect, u, y1);
        load_state<n>(zb, c.N, q, 0, z);
        int ez = to_unit<n>(z);
        q00 = times_pow2(to_f64(coef_dot<T, K, W>(z, y0)), ez + e0);
        q01 = times_pow2(to_f64(coef_dot<T, K, W>(z, y1)), ez + e1);
        load_state<n>(zb, c.N, q, n, z);
        ez = to_unit<n>(z);
        q10 = times_pow2(to_f64(coef_dot<T, K, W>(z, y0)), ez + e0);
        q11 = times_pow2(to_f64(coef_dot<T, K, W>(z, y1)), ez + e1);
    }
    double qs[3];
#pragma unroll
    for (int fld = 2; fld < 5; ++fld) {
        T u[n], z[n];
        W y[n];
#pragma unroll
        for (int i = 0; i < n; ++i) u[i] = U[fld * n + i];
        const int eu = to_unit<n>(u);
        mass_apply<T, K>(M0, rect, u, y);
        load_state<n>(zb, c.N, q, fld * n, z);
        const int ez = to_unit<n>(z);
        qs[fld - 2] = times_pow2(to_f64(coef_dot<T, K, W>(z, y)), eu + ez);
    }
    const double q22 = qs[0], qv = qs[1] + qs[2];
    const double d0 = G.mass_s[q], d1 = G.mass_s[N + q], d2 = G.mass_s[2 * N + q], rv = G.mass_s[3 * N + q];
    const double c1 = A.op.scal_s[SS_C1 * N + q], r = A.op.scal_s[SS_R * N + q];
    // mu_xx = -(d0 z_xx + d1 z_yy), mu_yy = -(d1 z_xx + d0 z_yy), mu_xy = -d2 z_xy (times M0 and w)
    const double xx_xx = d0 * q00 + d1 * q10, xx_yy = d0 * q01 + d1 * q11;
    const double yy_xx = d1 * q00 + d0 * q10, yy_yy = d1 * q01 + d0 * q11;
    const double w = G.w;
    G.grad_s[q] = fma(-w, xx_xx + r * xx_yy + yy_yy + r * yy_xx, G.grad_s[q]);          // d/dc1
    G.grad_s[N + q] = fma(-w * c1, xx_yy + yy_xx, G.grad_s[N + q]);                     // d/dr
    G.grad_s[2 * N + q] = fma(-w * d2, q22, G.grad_s[2 * N + q]);               // d/dc3
    G.grad_s[3 * N + q] = fma(w * rv, qv, G.grad_s[3 * N + q]);                 // d/d(1/(rho h))
    if (G.wgrad)
        for (int s = 0; s < A.n_src; ++s)
            if (A.src_dom[s] == 1 && A.src_q[s] == q)
                G.wgrad[s] = w * rv * wide_form<T, K, 2>(A.op, ci, zb + (size_t)3 * n * N + q, c.N,
                                                         A.src_g + (size_t)s * 2 * n);
}

// ---- fluid cells -------------------------------------------------------------------
// Lift the face jump of one face into the raw rate accumulators
// (kmx, kmy: grad p part; kp: div m part, tau folded).
// The jump p_F - p|_F on local face j (face-basis coefficients, the cell's
// orientation): own omega plus the neighbour's w (interior), or the
// interface combination of the solid neighbour's traces.
template <class T, int K>
__device__ __forceinline__ void fluid_face_jump(const StageArgsT<T>& A, const CellCtx<T>& c, int j, T* jmp) {
    constexpr int f = Dims<K>::f;
    const DevOps& op = A.op;
    const int slot = c.sbase + j * c.npad + c.lq;
    const int nb = __ldg(op.nb_f + slot);
#pragma unroll
    for (int l = 0; l < f; ++l) jmp[l] = c.trf_in[(size_t)(f + l) * c.SF + slot];
    if (nb >= 0) {
        const T be = __ldg(OpData<T>::beta_f(op) + slot);
#pragma unroll
        for (int l = 0; l < f; ++l) {
            const T w = c.trf_in[(size_t)l * c.SF + nb];
            jmp[l] = (l & 1) ? fma(-be, w, jmp[l]) : fma(be, w, jmp[l]);
        }
    } else if (nb < NB_BOUNDARY) {
        const int r = -2 - nb;
        const int ns = __ldg(op.if_nb + r);
        const T* co = OpData<T>::if_coef(op) + 6 * r;
        const T bx = __ldg(co + 1), by = __ldg(co + 2);
#pragma unroll
        for (int l = 0; l < f; ++l) {
            const T ws = fma(bx, c.trs_in[(size_t)l * c.SS + ns], by * c.trs_in[(size_t)(f + l) * c.SS + ns]);
            jmp[l] = (l & 1) ? jmp[l] - ws : jmp[l] + ws;
        }
    }
}

// Both faces of one orientation of a rectangle (AX = 0: faces 0 and 2,
// normals -/+ e_y; AX = 1: faces 1 and 3, normals +/- e_x), lifted with the
// first face's matrix L.  The mirror through the centroid maps face AX to
// face AX + 2 with Lift_{AX+2} = P L F (P: (-1)^(exponent along the normal)
// on the rows, F: (-1)^l on the face coefficients; checked when the class is
// built).  With s the first face's normal sign, jb, jp the two jumps and
// jh = F jp, sigma = jb + jh and delta = jb - jh:
//     normal accumulator  += s L delta (rows with P = +1), s L sigma (P = -1)
//     jump accumulator    += L sigma (P = +1), L delta (P = -1)
// Each lifted row is accumulated straight into its target: 2f + 2 nnz(L)
// operations per pair instead of 2 (nnz(L) + 2n) for two separate lifts.  tau
// multiplies the jump accumulator once per cell in FP64 (Fp64Form); the other
// types scale sigma and delta and accumulate into the rate.
template <class T, int K, int AX, bool SQ = false>
__device__ __forceinline__ void lift_pair(const T* __restrict__ L, const T* jb, const T* jp, T tau, T* ke, T* ks) {
    constexpr int n = Dims<K>::n, f = Dims<K>::f, fP = Dims<K>::fP, w = Vec16<T>::w;
    using P = typename std::conditional<SQ, SquareAxis<AX>, RectAxis<AX>>::type;
    constexpr bool neg = AX == 0;   // face 0 has normal -e_y, face 1 +e_x
    T sg[f], dl[f], ts[f], td[f];   // sigma, delta; what the jump accumulator takes
#pragma unroll
    for (int l = 0; l < f; ++l) {
        const T jh = (l & 1) ? -jp[l] : jp[l];
        sg[l] = jb[l] + jh;
        dl[l] = jb[l] - jh;
        ts[l] = Fp64Form<T>::value ? sg[l] : mul_rn(tau, sg[l]);
        td[l] = Fp64Form<T>::value ? dl[l] : mul_rn(tau, dl[l]);
    }
#pragma unroll
    for (int i = 0; i < n; ++i) {
        const int en = AX == 0 ? eb(i) : ea(i);   // exponent along the normal
        const bool even = (en & 1) == 0;
        T row[fP];
#pragma unroll
        for (int c0 = 0; c0 < fP; c0 += w) {
            bool need = false;
#pragma unroll
            for (int e = 0; e < w; ++e) need = need || (c0 + e < f && P::lift_nz(i, c0 + e));
            if (need) cls_row<T>(L + i * fP + c0, row + c0);
        }
        T e = ke[i], k = ks[i];
#pragma unroll
        for (int l = 0; l < f; ++l)
            if (P::lift_nz(i, l)) {
                const T a = even ? dl[l] : sg[l];
                e = neg ? fma(-row[l], a, e) : fma(row[l], a, e);
                k = fma(row[l], even ? ts[l] : td[l], k);
            }
        ke[i] = e;
        ks[i] = k;
    }
}

template <class T, int K, int AX, bool SQ = false>
__device__ __forceinline__ void fluid_pair_rate(const StageArgsT<T>& A, const CellCtx<T>& c, T* kmx, T* kmy, T* ks) {
    constexpr int f = Dims<K>::f, FS = Dims<K>::FS;
    T jb[f], jp[f];
    fluid_face_jump<T, K>(A, c, AX, jb);
    fluid_face_jump<T, K>(A, c, AX + 2, jp);
    lift_pair<T, K, AX, SQ>(c.cd + AX * FS + Dims<K>::LI, jb, jp, c.tau, AX == 0 ? kmy : kmx, ks);
}

template <class T, int K, class P>
__device__ __forceinline__ void fluid_face_rate(const StageArgsT<T>& A, const CellCtx<T>& c, int j, int sg, T* kmx,
                                                T* kmy, T* kp) {
    constexpr int n = Dims<K>::n, f = Dims<K>::f, FS = Dims<K>::FS;
    const DevOps& op = A.op;
    const T* fm = c.cd + j * FS;
    T jmp[f];
    fluid_face_jump<T, K>(A, c, j, jmp);
    T lv[n];
    lift_apply<T, K, P>(fm + Dims<K>::LI, jmp, lv);
    if constexpr (P::axis) {
        add_signed<n>(lv, P::horiz ? kmy : kmx, sg);
    } else {
        const T nx = cls_val(fm), ny = cls_val(fm + 1);
#pragma unroll
        for (int i = 0; i < n; ++i) {
            kmx[i] = fma(nx, lv[i], kmx[i]);
            kmy[i] = fma(ny, lv[i], kmy[i]);
        }
    }
#pragma unroll
    for (int i = 0; i < n; ++i) kp[i] = fma(c.tau, lv[i], kp[i]);
}

// Publish w = tau p|_F - (m.n)|_F and omega = alpha w - p|_F for one face.
template <class T, int K, class P>
__device__ __forceinline__ void fluid_face_trace(const StageArgsT<T>& A, const CellCtx<T>& c, int j, int sg,
                                                 const T* U) {
    constexpr int n = Dims<K>::n, f = Dims<K>::f, FS = Dims<K>::FS;
    const DevOps& op = A.op;
    const T* fm = c.cd + j * FS;
    const T* Tr = fm + Dims<K>::TR;
    const T* mx = U;
    const T* my = U + n;
    const T* p = U + 2 * n;
    T tp[f], tm[f];
    face_trace_apply<T, K, P>(Tr, p, tp, sg);
    if constexpr (P::axis) {
        face_trace_apply<T, K, P>(Tr, P::horiz ? my : mx, tm, sg);
    } else {
        const T nx = cls_val(fm), ny = cls_val(fm + 1);
        if constexpr (Fp64Form<T>::value) {   // two traces (2 f n + 2 f operations) against 2 n + f n for m.n first:
            T t1[f];                          // more here, but the team form, which shares it, takes coefficient by
            face_trace_apply<T, K, P>(Tr, mx, tm, sg);   // coefficient and would form m.n f times
            face_trace_apply<T, K, P>(Tr, my, t1, sg);
#pragma unroll
            for (int l = 0; l < f; ++l) tm[l] = fma(nx, tm[l], mul_rn(ny, t1[l]));
        } else {
            T mn[n];
#pragma unroll
            for (int i = 0; i < n; ++i) mn[i] = fma(nx, mx[i], mul_rn(ny, my[i]));
            face_trace_apply<T, K, P>(Tr, mn, tm, sg);
        }
    }
    const int sgn = P::axis ? sg : 1;   // axis-aligned: tm holds the unsigned trace
    const int slot = c.sbase + j * c.npad + c.lq;
    const int nb = __ldg(op.nb_f + slot);
    const T al = (nb >= NB_BOUNDARY) ? __ldg(OpData<T>::beta_f(op) + slot) : __ldg(OpData<T>::if_coef(op) + 6 * (-2 - nb));
#pragma unroll
    for (int l = 0; l < f; ++l) {
        const T w = fma(c.tau, tp[l], (sgn > 0) ? -tm[l] : tm[l]);
        c.trf_out[(size_t)l * c.SF + slot] = norm(w);
        c.trf_out[(size_t)(f + l) * c.SF + slot] = norm(fma(al, w, -tp[l]));
    }
}

// The four faces of a rectangle: one body per orientation looped over its
// two faces (RectLoop), or unrolled with constant signs.
template <class T, int K, class PH, class PV>
__device__ __forceinline__ void fluid_rect_traces(const StageArgsT<T>& A, const CellCtx<T>& c, const T* U) {
    if constexpr (RectLoop<T, K>::value) {
#pragma unroll 1
        for (int h = 0; h < 2; ++h) fluid_face_trace<T, K, PH>(A, c, 2 * h, 2 * h - 1, U);
#pragma unroll 1
        for (int v = 0; v < 2; ++v) fluid_face_trace<T, K, PV>(A, c, 1 + 2 * v, 1 - 2 * v, U);
    } else {
        fluid_face_trace<T, K, PH>(A, c, 0, -1, U);
        fluid_face_trace<T, K, PV>(A, c, 1, 1, U);
        fluid_face_trace<T, K, PH>(A, c, 2, 1, U);
        fluid_face_trace<T, K, PV>(A, c, 3, -1, U);
    }
}

// FP64 rectangles: the rate of a primal field from its lifted jumps k (sum_F L j)
// and the divergence of its flux (a, b), the state's fields at rows fa and fb:
// k = tau k + da/dX + db/dY.  The flux is loaded here, after the faces, so that
// the face loop holds neither it nor its derivatives.
template <class T, int K>
__device__ __forceinline__ void fp64_rect_div(const T* inp, const CellCtx<T>& c, int fa, int fb, T* k) {
    constexpr int n = Dims<K>::n;
    T a[n], b[n], d[n];
    load_state<n>(inp, c.N, c.q, fa, a);
    load_state<n>(inp, c.N, c.q, fb, b);
    ddx<T, K>(a, d);
    add_ddy<T, K>(b, d);
#pragma unroll
    for (int i = 0; i < n; ++i) k[i] = fma(c.tau, k[i], d[i]);
}

template <class T, int K, int MODE>
__device__ __forceinline__ void fluid_cell(const StageArgsT<T>& A, int q, int shot, const T* cd_smem, T* acc_smem,
                                           const GradArgsT<T>* G = nullptr) {
    constexpr int n = Dims<K>::n, f = Dims<K>::f;
    const DevOps& op = A.op;
    const int cls = __ldg(op.warp_class + (q >> 5));
    const int* ci = op.cls_int + cls * CI_STRIDE;
    CellCtx<T> c;
    c.q = q;
    c.lq = q - __ldg(ci + CI_START);
    if (c.lq >= __ldg(ci + CI_COUNT)) return;   // class padding
    c.nF = __ldg(ci + CI_NF);
    c.npad = __ldg(ci + CI_NPAD);
    c.sbase = __ldg(ci + CI_SLOT);
    c.hor = (uint32_t)__ldg(ci + CI_HOR);
    c.ver = (uint32_t)__ldg(ci + CI_VER);
    c.FS = Dims<K>::FS;
    c.cd = ClsSmem<T>::value ? cd_smem : OpData<T>::cls(op) + __ldg(ci + CI_DOFF) + Dims<K>::M0P;
    c.N = op.Nf;
    c.SF = op.SF;
    c.SS = op.SS;
    c.tau = __ldg(OpData<T>::scal_f(op) + SF_TAU * c.N + q);
    const size_t toff = (size_t)shot * A.trace_stride;
    c.trf_in = A.tr_in + toff;
    c.trs_in = A.tr_in + toff + (size_t)2 * f * c.SF;
    c.trf_out = A.tr_out + toff;
    c.trs_out = A.tr_out + toff + (size_t)2 * f * c.SF;
    const size_t soff = (size_t)shot * A.state_stride;
    const int kind = __ldg(ci + CI_KIND);
    const bool rect = kind != KIND_GENERIC;
    T Ureg[AccSmem<T, K>::value ? 1 : 3 * n];
    T* U = AccSmem<T, K>::value ? acc_smem : Ureg;   // [m_x | m_y | p]
    if constexpr (MODE == MODE_TRACES) {
        load_state<3 * n>(A.inp + soff, c.N, q, 0, U);
    } else {
        T* kmx = U;
        T* kmy = U + n;
        T* kp = U + 2 * n;
        if constexpr (L2Prefetch<T, K>::mask != 0)
            prefetch_cell<T, K, 3 * n, f, 0, MODE != MODE_GRAD>(A, c, soff, c.trf_in, c.SF, op.nb_f,
                                                            OpData<T>::beta_f(op), rect ? 4 : c.nF);
        const bool late = Fp64Form<T>::value && rect;   // div m after the faces, see fp64_rect_div
        {
            T u[n];
            load_state<n>(A.inp + soff, c.N, q, 2 * n, u);      // p
            ddx<T, K>(u, kmx);
            ddy<T, K>(u, kmy);
            if (!late) {
                load_state<n>(A.inp + soff, c.N, q, 0, u);      // m_x
                ddx<T, K>(u, kp);
                load_state<n>(A.inp + soff, c.N, q, n, u);      // m_y
                add_ddy<T, K>(u, kp);
            }
        }
        if constexpr (L2Prefetch<T, K>::mask != 0)
            prefetch_cell<T, K, 3 * n, f, 1, MODE != MODE_GRAD>(A, c, soff, c.trf_in, c.SF, op.nb_f,
                                                            OpData<T>::beta_f(op), rect ? 4 : c.nF);
        if (rect) {
            // faces 0 (s = -1) and 2 (s = +1) are horizontal, 1 (s = +1) and 3 (s = -1) vertical
            if constexpr (Fp64Form<T>::value) {
#pragma unroll
                for (int i = 0; i < n; ++i) kp[i] = T(0);
            }
            if (kind == KIND_SQUARE) {
                fluid_pair_rate<T, K, 0, true>(A, c, kmx, kmy, kp);   // faces 0 and 2
                fluid_pair_rate<T, K, 1, true>(A, c, kmx, kmy, kp);   // faces 1 and 3
            } else {
                fluid_pair_rate<T, K, 0>(A, c, kmx, kmy, kp);
                fluid_pair_rate<T, K, 1>(A, c, kmx, kmy, kp);
            }
            if constexpr (Fp64Form<T>::value) fp64_rect_div<T, K>(A.inp + soff, c, 0, n, kp);
        } else {
            for_faces(c, [&](int j, int sg) { fluid_face_rate<T, K, PolyAxis<0>>(A, c, j, sg, kmx, kmy, kp); },
                      [&](int j, int sg) { fluid_face_rate<T, K, PolyAxis<1>>(A, c, j, sg, kmx, kmy, kp); },
                      [&](int j) { fluid_face_rate<T, K, GenericFace>(A, c, j, 1, kmx, kmy, kp); });
        }
        const T Am = __ldg(OpData<T>::scal_f(op) + SF_AM * c.N + q), Ap = __ldg(OpData<T>::scal_f(op) + SF_AP * c.N + q);
        // Point sources: the stored vector is kappa/h^2 M0^-1 phi(x_s); the
        // raw rate is multiplied by A_p = kappa/h in the targets.
        for (int s = 0; s < A.n_src; ++s) {
            if (A.src_dom[s] == 0 && A.src_q[s] == q) {
                const T w = src_value(A, s) / Ap;
                const T* g = A.src_g + (size_t)s * 2 * n;
#pragma unroll
                for (int i = 0; i < n; ++i) kp[i] = fma(w, g[i], kp[i]);
            }
        }
        if (A.shot_src_q && A.shot_src_dom[shot] == 0 && A.shot_src_q[shot] == q) {
            const T w = shot_src_value(A) / Ap;
            const T* g = A.shot_src_g + (size_t)shot * 2 * n;
#pragma unroll
            for (int i = 0; i < n; ++i) kp[i] = fma(w, g[i], kp[i]);
        }
        if constexpr (MODE == MODE_GRAD) {
            fluid_grad<T, K>(A, *G, c, ci, rect, U);
            return;
        }
        const T sc[3] = {Am, Ap, T(0)};
        write_targets<3 * n, FluidGroups<n>>(A, c.N, soff, q, U, sc);
        if constexpr (MODE == MODE_APPLY) return;
    }
    if (kind == KIND_SQUARE) {
        fluid_rect_traces<T, K, SquareAxis<0>, SquareAxis<1>>(A, c, U);
    } else if (rect) {
        fluid_rect_traces<T, K, RectAxis<0>, RectAxis<1>>(A, c, U);
    } else {
        for_faces(c, [&](int j, int sg) { fluid_face_trace<T, K, PolyAxis<0>>(A, c, j, sg, U); },
                  [&](int j, int sg) { fluid_face_trace<T, K, PolyAxis<1>>(A, c, j, sg, U); },
                  [&](int j) { fluid_face_trace<T, K, GenericFace>(A, c, j, 1, U); });
    }
}

// ---- solid cells -------------------------------------------------------------------
// The velocity jump v_F - v|_F on local face j (components x, y).
template <class T, int K>
__device__ __forceinline__ void solid_face_jump(const StageArgsT<T>& A, const CellCtx<T>& c, int j, T* jx, T* jy) {
    constexpr int f = Dims<K>::f;
    const DevOps& op = A.op;
    const int slot = c.sbase + j * c.npad + c.lq;
    const int nb = __ldg(op.nb_s + slot);
#pragma unroll
    for (int l = 0; l < f; ++l) {
        jx[l] = c.trs_in[(size_t)(2 * f + l) * c.SS + slot];
        jy[l] = c.trs_in[(size_t)(3 * f + l) * c.SS + slot];
    }
    if (nb >= 0) {
        const T be = __ldg(OpData<T>::beta_s(op) + slot);
#pragma unroll
        for (int l = 0; l < f; ++l) {
            const T wx = c.trs_in[(size_t)l * c.SS + nb];
            const T wy = c.trs_in[(size_t)(f + l) * c.SS + nb];
            jx[l] = (l & 1) ? fma(-be, wx, jx[l]) : fma(be, wx, jx[l]);
            jy[l] = (l & 1) ? fma(-be, wy, jy[l]) : fma(be, wy, jy[l]);
        }
    } else if (nb < NB_BOUNDARY) {
        const int r = -2 - nb;
        const int nfs = __ldg(op.if_nb + r);
        const T* co = OpData<T>::if_coef(op) + 6 * r;
        const T b0 = __ldg(co + 4), b1 = __ldg(co + 5);
#pragma unroll
        for (int l = 0; l < f; ++l) {
            const T wf = c.trf_in[(size_t)l * c.SF + nfs];
            jx[l] = (l & 1) ? fma(-b0, wf, jx[l]) : fma(b0, wf, jx[l]);
            jy[l] = (l & 1) ? fma(-b1, wf, jy[l]) : fma(b1, wf, jy[l]);
        }
    }
}

// Lift one face's velocity jump into the raw accumulators: e (strain rate,
// symmetric-gradient part) and kv (div s part, tau folded).
template <class T, int K, class P>
__device__ __forceinline__ void solid_face_rate(const StageArgsT<T>& A, const CellCtx<T>& c, int j, int sg, T* exx,
                                                T* eyy, T* exy, T* kvx, T* kvy) {
    constexpr int n = Dims<K>::n, f = Dims<K>::f, FS = Dims<K>::FS;
    const DevOps& op = A.op;
    const T* fm = c.cd + j * FS;
    T jx[f], jy[f];
    solid_face_jump<T, K>(A, c, j, jx, jy);
    const T* L = fm + Dims<K>::LI;
    T lx[n], ly[n];
    lift_apply<T, K, P>(L, jx, lx);
    lift_apply<T, K, P>(L, jy, ly);
    if constexpr (P::axis) {
        if constexpr (P::horiz) {
            add_signed<n>(ly, eyy, sg);
            add_signed<n>(lx, exy, sg);
        } else {
            add_signed<n>(lx, exx, sg);
            add_signed<n>(ly, exy, sg);
        }
    } else {
        const T nx = cls_val(fm), ny = cls_val(fm + 1);
#pragma unroll
        for (int i = 0; i < n; ++i) {
            exx[i] = fma(nx, lx[i], exx[i]);
            eyy[i] = fma(ny, ly[i], eyy[i]);
            exy[i] = fma(nx, ly[i], fma(ny, lx[i], exy[i]));
        }
    }
#pragma unroll
    for (int i = 0; i < n; ++i) {
        kvx[i] = fma(c.tau, lx[i], kvx[i]);
        kvy[i] = fma(c.tau, ly[i], kvy[i]);
    }
}

// Both faces of one rectangle orientation (see lift_pair): horizontal faces
// feed e_yy (y component) and e_xy (x component), vertical ones e_xx (x) and
// e_xy (y); tau times both components feeds kv.
template <class T, int K, int AX, bool SQ = false>
__device__ __forceinline__ void solid_pair_rate(const StageArgsT<T>& A, const CellCtx<T>& c, T* exx, T* eyy, T* exy,
                                                T* kvx, T* kvy) {
    constexpr int f = Dims<K>::f, FS = Dims<K>::FS;
    T bx[f], by[f], px[f], py[f];
    solid_face_jump<T, K>(A, c, AX, bx, by);
    solid_face_jump<T, K>(A, c, AX + 2, px, py);
    const T* L = c.cd + AX * FS + Dims<K>::LI;
    lift_pair<T, K, AX, SQ>(L, bx, px, c.tau, AX == 0 ? exy : exx, kvx);
    lift_pair<T, K, AX, SQ>(L, by, py, c.tau, AX == 0 ? eyy : exy, kvy);
}

// FP64: both components of one orientation's jumps lifted together, so that
// four consecutive multiply-adds share the matrix entry.  The FP64 pipe takes 16
// cycles for an instruction that shares a register operand with the one before
// it and 19 otherwise (measured per SM).
template <class T, int K, int AX, bool SQ>
__device__ __forceinline__ void fp64_solid_pair(const StageArgsT<T>& A, const CellCtx<T>& c, T* ex, T* ey, T* kvx,
                                                T* kvy) {
    constexpr int n = Dims<K>::n, f = Dims<K>::f, fP = Dims<K>::fP, FS = Dims<K>::FS, w = Vec16<T>::w;
    using P = typename std::conditional<SQ, SquareAxis<AX>, RectAxis<AX>>::type;
    constexpr bool neg = AX == 0;
    const T* L = c.cd + AX * FS + Dims<K>::LI;
    T sx[f], sy[f], dx[f], dy[f];   // sigma, delta of both components
    {
        T bx[f], by[f], px[f], py[f];
        solid_face_jump<T, K>(A, c, AX, bx, by);
        solid_face_jump<T, K>(A, c, AX + 2, px, py);
#pragma unroll
        for (int l = 0; l < f; ++l) {
            const T hx = (l & 1) ? -px[l] : px[l], hy = (l & 1) ? -py[l] : py[l];
            sx[l] = bx[l] + hx;
            dx[l] = bx[l] - hx;
            sy[l] = by[l] + hy;
            dy[l] = by[l] - hy;
        }
    }
#pragma unroll
    for (int i = 0; i < n; ++i) {
        const bool even = ((AX == 0 ? eb(i) : ea(i)) & 1) == 0;
        T row[fP];
#pragma unroll
        for (int c0 = 0; c0 < fP; c0 += w) {
            bool need = false;
#pragma unroll
            for (int e = 0; e < w; ++e) need = need || (c0 + e < f && P::lift_nz(i, c0 + e));
            if (need) cls_row<T>(L + i * fP + c0, row + c0);
        }
        T e0 = ex[i], e1 = ey[i], k0 = kvx[i], k1 = kvy[i];
#pragma unroll
        for (int l = 0; l < f; ++l)
            if (P::lift_nz(i, l)) {
                const T a0 = even ? dx[l] : sx[l], a1 = even ? dy[l] : sy[l];
                e0 = neg ? fma(-row[l], a0, e0) : fma(row[l], a0, e0);
                e1 = neg ? fma(-row[l], a1, e1) : fma(row[l], a1, e1);
                k0 = fma(row[l], even ? sx[l] : dx[l], k0);
                k1 = fma(row[l], even ? sy[l] : dy[l], k1);
            }
        ex[i] = e0;
        ey[i] = e1;
        kvx[i] = k0;
        kvy[i] = k1;
    }
}

// Publish w = tau v|_F - (s n)|_F and omega = alpha w - v|_F for one face.
template <class T, int K, class P>
__device__ __forceinline__ void solid_face_trace(const StageArgsT<T>& A, const CellCtx<T>& c, int j, int sg,
                                                 const T* U) {
    constexpr int n = Dims<K>::n, f = Dims<K>::f, FS = Dims<K>::FS;
    const DevOps& op = A.op;
    const T* fm = c.cd + j * FS;
    const T* Tr = fm + Dims<K>::TR;
    const T* sxx = U;
    const T* syy = U + n;
    const T* sxy = U + 2 * n;
    const T* vx = U + 3 * n;
    const T* vy = U + 4 * n;
    T tvx[f], tvy[f], tsx[f], tsy[f];
    face_trace_apply<T, K, P>(Tr, vx, tvx, sg);
    face_trace_apply<T, K, P>(Tr, vy, tvy, sg);
    if constexpr (P::axis) {
        // s n = (nx s_xx + ny s_xy, nx s_xy + ny s_yy) with one of nx, ny = +-1
        if constexpr (!P::horiz) {
            face_trace_apply<T, K, P>(Tr, sxx, tsx, sg);
            face_trace_apply<T, K, P>(Tr, sxy, tsy, sg);
        } else {
            face_trace_apply<T, K, P>(Tr, sxy, tsx, sg);
            face_trace_apply<T, K, P>(Tr, syy, tsy, sg);
        }
    } else {
        const T nx = cls_val(fm), ny = cls_val(fm + 1);
        if constexpr (Fp64Form<T>::value) {   // see fluid_face_trace
            T txy[f];
            face_trace_apply<T, K, P>(Tr, sxx, tsx, sg);
            face_trace_apply<T, K, P>(Tr, syy, tsy, sg);
            face_trace_apply<T, K, P>(Tr, sxy, txy, sg);
#pragma unroll
            for (int l = 0; l < f; ++l) {
                tsx[l] = fma(nx, tsx[l], mul_rn(ny, txy[l]));
                tsy[l] = fma(nx, txy[l], mul_rn(ny, tsy[l]));
            }
        } else {
            T snx[n], sny[n];
#pragma unroll
            for (int i = 0; i < n; ++i) {
                snx[i] = fma(nx, sxx[i], mul_rn(ny, sxy[i]));
                sny[i] = fma(nx, sxy[i], mul_rn(ny, syy[i]));
            }
            face_trace_apply<T, K, P>(Tr, snx, tsx, sg);
            face_trace_apply<T, K, P>(Tr, sny, tsy, sg);
        }
    }
    const int sgn = P::axis ? sg : 1;
    const int slot = c.sbase + j * c.npad + c.lq;
    const int nb = __ldg(op.nb_s + slot);
    T* TWS = c.trs_out;
    if (nb >= NB_BOUNDARY) {
        const T be = __ldg(OpData<T>::beta_s(op) + slot);
#pragma unroll
        for (int l = 0; l < f; ++l) {
            const T wx = fma(c.tau, tvx[l], (sgn > 0) ? -tsx[l] : tsx[l]);
            const T wy = fma(c.tau, tvy[l], (sgn > 0) ? -tsy[l] : tsy[l]);
            TWS[(size_t)l * c.SS + slot] = norm(wx);
            TWS[(size_t)(f + l) * c.SS + slot] = norm(wy);
            TWS[(size_t)(2 * f + l) * c.SS + slot] = norm(fma(be, wx, -tvx[l]));
            TWS[(size_t)(3 * f + l) * c.SS + slot] = norm(fma(be, wy, -tvy[l]));
        }
    } else {
        const T* co = OpData<T>::if_coef(op) + 6 * (-2 - nb);
        const T a00 = __ldg(co), a01 = __ldg(co + 1), a10 = __ldg(co + 2), a11 = __ldg(co + 3);
#pragma unroll
        for (int l = 0; l < f; ++l) {
            const T wx = fma(c.tau, tvx[l], (sgn > 0) ? -tsx[l] : tsx[l]);
            const T wy = fma(c.tau, tvy[l], (sgn > 0) ? -tsy[l] : tsy[l]);
            TWS[(size_t)l * c.SS + slot] = norm(wx);
            TWS[(size_t)(f + l) * c.SS + slot] = norm(wy);
            TWS[(size_t)(2 * f + l) * c.SS + slot] = norm(fma(a00, wx, fma(a01, wy, -tvx[l])));
            TWS[(size_t)(3 * f + l) * c.SS + slot] = norm(fma(a10, wx, fma(a11, wy, -tvy[l])));
        }
    }
}

// The four faces of a rectangle: one body per orientation looped over its
// two faces (RectLoop), or unrolled with constant signs.
template <class T, int K, class PH, class PV>
__device__ __forceinline__ void solid_rect_traces(const StageArgsT<T>& A, const CellCtx<T>& c, const T* U) {
    if constexpr (RectLoop<T, K>::value) {
#pragma unroll 1
        for (int h = 0; h < 2; ++h) solid_face_trace<T, K, PH>(A, c, 2 * h, 2 * h - 1, U);
#pragma unroll 1
        for (int v = 0; v < 2; ++v) solid_face_trace<T, K, PV>(A, c, 1 + 2 * v, 1 - 2 * v, U);
    } else {
        solid_face_trace<T, K, PH>(A, c, 0, -1, U);
        solid_face_trace<T, K, PV>(A, c, 1, 1, U);
        solid_face_trace<T, K, PH>(A, c, 2, 1, U);
        solid_face_trace<T, K, PV>(A, c, 3, -1, U);
    }
}

template <class T, int K, int MODE>
__device__ __forceinline__ void solid_cell(const StageArgsT<T>& A, int q, int shot, const T* cd_smem, T* acc_smem,
                                           const GradArgsT<T>* G = nullptr) {
    constexpr int n = Dims<K>::n, f = Dims<K>::f;
    const DevOps& op = A.op;
    const int cls = __ldg(op.warp_class + op.n_warps_f + (q >> 5));
    const int* ci = op.cls_int + cls * CI_STRIDE;
    CellCtx<T> c;
    c.q = q;
    c.lq = q - __ldg(ci + CI_START);
    if (c.lq >= __ldg(ci + CI_COUNT)) return;
    c.nF = __ldg(ci + CI_NF);
    c.npad = __ldg(ci + CI_NPAD);
    c.sbase = __ldg(ci + CI_SLOT);
    c.hor = (uint32_t)__ldg(ci + CI_HOR);
    c.ver = (uint32_t)__ldg(ci + CI_VER);
    c.FS = Dims<K>::FS;
    c.cd = ClsSmem<T>::value ? cd_smem : OpData<T>::cls(op) + __ldg(ci + CI_DOFF) + Dims<K>::M0P;
    c.N = op.Ns;
    c.SF = op.SF;
    c.SS = op.SS;
    c.tau = __ldg(OpData<T>::scal_s(op) + SS_TAU * c.N + q);
    const size_t toff = (size_t)shot * A.trace_stride;
    c.trf_in = A.tr_in + toff;
    c.trs_in = A.tr_in + toff + (size_t)2 * f * c.SF;
    c.trf_out = A.tr_out + toff;
    c.trs_out = A.tr_out + toff + (size_t)2 * f * c.SF;
    const int kind = __ldg(ci + CI_KIND);
    const bool rect = kind != KIND_GENERIC;
    const size_t soff = (size_t)shot * A.state_stride + (size_t)3 * n * op.Nf;
    const T* inp = A.inp + soff;
    T Ureg[AccSmem<T, K>::value ? 1 : 5 * n];
    T* U = AccSmem<T, K>::value ? acc_smem : Ureg;   // [s_xx | s_yy | s_xy | v_x | v_y]
    if constexpr (MODE == MODE_TRACES) {
        load_state<5 * n>(inp, c.N, q, 0, U);
    } else {
        T* exx = U;
        T* eyy = U + n;
        T* exy = U + 2 * n;
        T* kvx = U + 3 * n;
        T* kvy = U + 4 * n;
        if constexpr (L2Prefetch<T, K>::mask != 0)
            prefetch_cell<T, K, 5 * n, 2 * f, 0, MODE != MODE_GRAD>(A, c, soff, c.trs_in, c.SS, op.nb_s,
                                                                OpData<T>::beta_s(op), rect ? 4 : c.nF);
        const bool late = Fp64Form<T>::value && rect;   // div s after the faces, see fp64_rect_div
        {
            T u[n];
            load_state<n>(inp, c.N, q, 3 * n, u);    // v_x
            ddx<T, K>(u, exx);
            ddy<T, K>(u, exy);
            load_state<n>(inp, c.N, q, 4 * n, u);    // v_y
            ddy<T, K>(u, eyy);
            add_ddx<T, K>(u, exy);
        }
        if (!late) {
            T u[n];
            load_state<n>(inp, c.N, q, 0, u);        // s_xx
            ddx<T, K>(u, kvx);
            load_state<n>(inp, c.N, q, n, u);        // s_yy
            ddy<T, K>(u, kvy);
            load_state<n>(inp, c.N, q, 2 * n, u);    // s_xy
            add_ddy<T, K>(u, kvx);
            add_ddx<T, K>(u, kvy);
        }
        if constexpr (L2Prefetch<T, K>::mask != 0)
            prefetch_cell<T, K, 5 * n, 2 * f, 1, MODE != MODE_GRAD>(A, c, soff, c.trs_in, c.SS, op.nb_s,
                                                                OpData<T>::beta_s(op), rect ? 4 : c.nF);
        if (rect) {
            if constexpr (Fp64Form<T>::value) {
#pragma unroll
                for (int i = 0; i < n; ++i) kvx[i] = kvy[i] = T(0);
                if (kind == KIND_SQUARE) {
                    fp64_solid_pair<T, K, 0, true>(A, c, exy, eyy, kvx, kvy);   // faces 0 and 2
                    fp64_solid_pair<T, K, 1, true>(A, c, exx, exy, kvx, kvy);   // faces 1 and 3
                } else {
                    fp64_solid_pair<T, K, 0, false>(A, c, exy, eyy, kvx, kvy);
                    fp64_solid_pair<T, K, 1, false>(A, c, exx, exy, kvx, kvy);
                }
                fp64_rect_div<T, K>(inp, c, 0, 2 * n, kvx);
                // the order of the sum matters for the bits: d/dY s_yy first, as in the general path
                {
                    T a[n], b[n], d[n];
                    load_state<n>(inp, c.N, q, n, a);
                    load_state<n>(inp, c.N, q, 2 * n, b);
                    ddy<T, K>(a, d);
                    add_ddx<T, K>(b, d);
#pragma unroll
                    for (int i = 0; i < n; ++i) kvy[i] = fma(c.tau, kvy[i], d[i]);
                }
            } else if (kind == KIND_SQUARE) {
                solid_pair_rate<T, K, 0, true>(A, c, exx, eyy, exy, kvx, kvy);   // faces 0 and 2
                solid_pair_rate<T, K, 1, true>(A, c, exx, eyy, exy, kvx, kvy);   // faces 1 and 3
            } else {
                solid_pair_rate<T, K, 0>(A, c, exx, eyy, exy, kvx, kvy);
                solid_pair_rate<T, K, 1>(A, c, exx, eyy, exy, kvx, kvy);
            }
        } else {
            for_faces(c, [&](int j, int sg) { solid_face_rate<T, K, PolyAxis<0>>(A, c, j, sg, exx, eyy, exy, kvx, kvy); },
                      [&](int j, int sg) { solid_face_rate<T, K, PolyAxis<1>>(A, c, j, sg, exx, eyy, exy, kvx, kvy); },
                      [&](int j) { solid_face_rate<T, K, GenericFace>(A, c, j, 1, exx, eyy, exy, kvx, kvy); });
        }
        // stress rate = C e = c1 [(e_xx + r e_yy), (e_yy + r e_xx)], c3 e_xy; c1, c3 folded into targets
        const T r = __ldg(OpData<T>::scal_s(op) + SS_R * c.N + q);
        if constexpr (MODE != MODE_GRAD) {
#pragma unroll
            for (int i = 0; i < n; ++i) {
                const T a = exx[i], b = eyy[i];
                exx[i] = fma(r, b, a);
                eyy[i] = fma(r, a, b);
            }
        }
        const T Av = __ldg(OpData<T>::scal_s(op) + SS_AV * c.N + q);
        for (int s = 0; s < A.n_src; ++s) {
            if (A.src_dom[s] == 1 && A.src_q[s] == q) {
                const T w = src_value(A, s) / Av;
                const T* g = A.src_g + (size_t)s * 2 * n;
#pragma unroll
                for (int i = 0; i < n; ++i) {
                    kvx[i] = fma(w, g[i], kvx[i]);
                    kvy[i] = fma(w, g[n + i], kvy[i]);
                }
            }
        }
        if (A.shot_src_q && A.shot_src_dom[shot] == 1 && A.shot_src_q[shot] == q) {
            const T w = shot_src_value(A) / Av;
            const T* g = A.shot_src_g + (size_t)shot * 2 * n;
#pragma unroll
            for (int i = 0; i < n; ++i) {
                kvx[i] = fma(w, g[i], kvx[i]);
                kvy[i] = fma(w, g[n + i], kvy[i]);
            }
        }
        if constexpr (MODE == MODE_GRAD) {
            solid_grad<T, K>(A, *G, c, ci, rect, U);
            return;
        }
        const T sc[3] = {__ldg(OpData<T>::scal_s(op) + SS_C1 * c.N + q), __ldg(OpData<T>::scal_s(op) + SS_C3 * c.N + q), Av};
        write_targets<5 * n, SolidGroups<n>>(A, c.N, soff, q, U, sc);
        if constexpr (MODE == MODE_APPLY) return;
    }
    if (kind == KIND_SQUARE) {
        solid_rect_traces<T, K, SquareAxis<0>, SquareAxis<1>>(A, c, U);
    } else if (rect) {
        solid_rect_traces<T, K, RectAxis<0>, RectAxis<1>>(A, c, U);
    } else {
        for_faces(c, [&](int j, int sg) { solid_face_trace<T, K, PolyAxis<0>>(A, c, j, sg, U); },
                  [&](int j, int sg) { solid_face_trace<T, K, PolyAxis<1>>(A, c, j, sg, U); },
                  [&](int j) { solid_face_trace<T, K, GenericFace>(A, c, j, 1, U); });
    }
}

// Resident blocks per SM asked of the register allocator (128 threads a
// block): 2 blocks allow 255 registers, 3 allow 168, 4 allow 128, 5 allow 96,
// 6 allow 80, 8 allow 64.  The kernels wait for loads, so occupancy pays until
// the registers no longer hold a batch of them (write_targets): us a stage by
// blocks, FP32 k = 3 (16 hybrid shots) 8: 866, 6: 849, 5: 862, 4: 903; FP32 k = 2
// (21 hanging shots) 12: 309, 10: 283, 8: 260, 6: 260, 5: 277; double-float k = 2
// (1024 x 512) 6: 177, 5: 172, 4: 182; FP64 k = 2 8: 225, 6: 224, 5: 225; FP64
// k = 3 (680 x 340 hybrid) 8: 291, 6: 286, 5: 284, 4: 276, 3: 276.  Where the accumulators sit in
// shared memory (AccSmem) it may cap the resident blocks below this count.
template <class T, int K>
struct MinBlocks {
    static constexpr int value = Tuned<T>::t.min_blocks[K - 1];
};

// Dynamic shared memory of a stage block of `threads` threads: the per-warp
// class copies (max_nf face blocks of Dims<K>::FS values per warp) when
// ClsSmem<T>, and the accumulators when AccSmem<T, K>.
template <class T, int K>
__host__ __device__ size_t stage_cls_smem_bytes(int max_nf, int threads) {
    return ClsSmem<T>::value ? sizeof(T) * (threads / 32) * (size_t)max_nf * Dims<K>::FS : 0;
}
template <class T, int K>
size_t stage_smem_bytes(int max_nf, int threads) {
    return stage_cls_smem_bytes<T, K>(max_nf, threads) + (AccSmem<T, K>::value ? sizeof(T) * threads * acc_stride<K>() : 0);
}

// Grid: x over the padded cells of both domains (fluid warps, then solid
// warps; a warp lies in one class), y over shots; 128 threads.
template <class T, int K, int MODE>
__global__ void __launch_bounds__(128, MinBlocks<T, K>::value) stage_kernel(const StageArgsT<T> A) {
    // the last cells first: solid cells are the longer ones and should not make the tail
    const int gq = 32 * A.warp0 + (gridDim.x - 1 - blockIdx.x) * blockDim.x + threadIdx.x;
    const int shot = blockIdx.y;
    wait_for_predecessor();
    const T* cd = nullptr;
    extern __shared__ __align__(16) unsigned char stage_smem[];
    T* acc = nullptr;
    if constexpr (AccSmem<T, K>::value)
        acc = reinterpret_cast<T*>(stage_smem + stage_cls_smem_bytes<T, K>(A.op.max_nf, blockDim.x)) + threadIdx.x * acc_stride<K>();
    if constexpr (ClsSmem<T>::value) {
        constexpr int FS = Dims<K>::FS;
        const int gw = gq >> 5;
        if (gw >= A.op.n_warps_f + A.op.n_warps_s) return;   // the whole warp is past the last class
        T* dst = reinterpret_cast<T*>(stage_smem) + (threadIdx.x >> 5) * A.op.max_nf * FS;
        const int* ci = A.op.cls_int + __ldg(A.op.warp_class + gw) * CI_STRIDE;
        const int nv = __ldg(ci + CI_NF) * FS * (int)sizeof(T) / 16;
        const float4* src =
            reinterpret_cast<const float4*>(OpData<T>::cls(A.op) + __ldg(ci + CI_DOFF) + Dims<K>::M0P);
        float4* d4 = reinterpret_cast<float4*>(dst);
        for (int e = threadIdx.x & 31; e < nv; e += 32) d4[e] = __ldg(src + e);
        __syncwarp();
        cd = dst;
    }
    if (gq < A.op.Nf)
        fluid_cell<T, K, MODE>(A, gq, shot, cd, acc);
    else if (gq < A.op.Nf + A.op.Ns)
        solid_cell<T, K, MODE>(A, gq - A.op.Nf, shot, cd, acc);
}

// The stabilisation-weight part of one cell's gradients.
template <class T, int K>
__device__ __forceinline__ void tau_cell(const StageArgsT<T>& A, const GradArgsT<T>& G, int gq) {
    const DevOps& op = A.op;
    const bool fl = gq < op.Nf;
    const int* ci = op.cls_int + __ldg(op.warp_class + (gq >> 5)) * CI_STRIDE;
    CellCtx<T> c;
    c.q = fl ? gq : gq - op.Nf;
    c.lq = c.q - __ldg(ci + CI_START);
    if (c.lq >= __ldg(ci + CI_COUNT)) return;
    c.nF = __ldg(ci + CI_NF);
    c.npad = __ldg(ci + CI_NPAD);
    c.sbase = __ldg(ci + CI_SLOT);
    if (fl) tau_grad<T, K, 1>(A, G, c, ci, gq);
    else tau_grad<T, K, 2>(A, G, c, ci, gq);
}

// One backward stage's gradients (MODE_GRAD): the stage kernel's rate of the
// forward stage value, taken straight into the gradient sums instead of being
// stored.  y = 0: the mass part, y = 1: the tau part, which share nothing but the
// traces they read; side by side they halve the chain of a thread and fill a
// grid of one wave (65,536 cells, k = 2: FP64 44.4 -> 42.8 us, FP32 30.1 -> 20.8; 42.9 and
// 21.6 since values are brought to unit size first, Range).
template <class T, int K>
__global__ void __launch_bounds__(128, MinBlocks<T, K>::value)
    grad_stage_kernel(const StageArgsT<T> A, const GradArgsT<T> G) {
    extern __shared__ __align__(16) unsigned char stage_smem[];
    const int gq = (gridDim.x - 1 - blockIdx.x) * blockDim.x + threadIdx.x;   // solid cells first, as stage_kernel
    wait_for_predecessor();
    if (gq >= A.op.Nf + A.op.Ns) return;
    if (blockIdx.y == 1) {
        tau_cell<T, K>(A, G, gq);
        return;
    }
    T* acc = nullptr;
    if constexpr (AccSmem<T, K>::value) acc = reinterpret_cast<T*>(stage_smem) + threadIdx.x * acc_stride<K>();
    if (gq < A.op.Nf) fluid_cell<T, K, MODE_GRAD>(A, gq, 0, nullptr, acc, &G);
    else solid_cell<T, K, MODE_GRAD>(A, gq - A.op.Nf, 0, nullptr, acc, &G);
}

#include "stage_team.cuh"

// Per function and device: the opt-in above 48 KB of dynamic shared memory
// (the largest size set is remembered), and the largest carveout where the
// accumulators live in shared memory, for the resident blocks that the
// register budget allows.  `Tag` makes one state per kernel.
template <class Tag, class F>
void stage_smem_attributes(F* kernel, size_t smem, bool carve) {
    static SmemOptIn state;
    int dev = 0;
    cudaGetDevice(&dev);
    state.require(
        dev, smem, carve,
        [&](size_t n) { cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)n); },
        [&] {
            cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout,
                                 (int)cudaSharedmemCarveoutMaxShared);
        });
}
template <class T, int K, int MODE>
struct StageTag {};

}  // namespace

namespace hho_stage {

// Threads of a stage block (the kernels use no block-wide barrier).  128 for
// large grids.  A grid of at most 20 warps per SM runs in one wave, where
// blocks of one warp spread the cells evenly over the SMs, while blocks of four
// leave some SMs with one more than others.  us a launch with 32 | 64 | 128 threads:
// 2048 warps, FP64, squares k = 2 32.3 | 34.8 | 39.9, triangles k = 3 102 | 112 | 126,
// FP32 triangles k = 3 14.8 | 15.5 | 16.9, gradients (k = 2) FP64 42.9 | 42.1 | 44.5, FP32
// 21.6 | 20.3 | 20.8; 4200 warps, FP64 squares k = 2 73.2 | 73.8 | 72.2; 8192 warps
// 121.1 | 121.1 | 121.3.
inline int stage_threads(int64_t warps) { return warps <= 20 * GB300_SMS ? 32 : 128; }

template <class T, int K, int MODE, int W>
struct TeamTag {};

// Where the team form (stage_team.cuh) is the faster one: up to so many groups
// of 32 cells (times shots), by arithmetic, degree, mode (stage, application,
// traces alone) and mesh (rectangles, or at least a quarter of the groups others:
// gen).  Up to 600 groups take W warps a block, more four (fewer idle warps, more
// blocks an SM) but for the 8-byte types at k = 3, whose ten rows fit ten warps.
// Both forms give the same bits, so the choice is free.  The lines lie where both
// forms, timed at 128 to 8192 groups of squares and of triangles, cross (us a
// launch on GB300, thread form / team form):
//                                 512 groups    1048          2048          4200
//   stage, squares    FP64 k = 1  11.3 / 9.7    13.4 / 14.6   18.2 / 23.0   36.9 / 46.8
//                     FP64 k = 2  18.6 / 17.3   21.9 / 27.2   32.5 / 44.9   72.9 / 92.2
//                     FP64 k = 3  29.7 / 21.6   37.0 / 37.0   58.0 / 74.2   118 / 147
//                     pairs k = 1 9.6 / 6.5     10.2 / 7.9    11.5 / 13.2   20.4 / 31.0
//                     pairs k = 2 19.6 / 8.3    20.1 / 12.6   22.9 / 23.5   53.9 / 57.6
//                     pairs k = 3 31.7 / 12.7   33.2 / 19.9   69.7 / 46.7   120 / 94.2
//                     FP32 k = 1  5.7 / 4.3     6.7 / 5.5     6.9 / 9.1     8.9 / 16.2
//                     FP32 k = 2  8.7 / 5.3     9.7 / 7.6     10.0 / 13.6   15.4 / 25.5
//                     FP32 k = 3  11.0 / 8.4    11.9 / 10.5   12.7 / 18.8   31.3 / 45.9
//   stage, triangles  FP64 k = 2  31.1 / 22.3   33.9 / 35.0   56.2 / 57.9   113 / 118
//                     FP64 k = 3  51.0 / 33.5   60.7 / 57.1   103 / 106     202 / 211
//                     pairs k = 3 49.9 / 15.0   52.0 / 24.9   92.4 / 48.0   134 / 97.5
//                     FP32 k = 3  13.1 / 8.8    12.6 / 11.0   15.0 / 19.9   33.7 / 43.5
//   traces, triangles FP64 k = 2  13.3 / 11.7   15.0 / 17.0   26.1 / 28.7   52.1 / 58.5
//                     pairs k = 3 21.8 / 9.8    30.8 / 15.6   39.5 / 32.3   56.4 / 61.5
//                     FP32 k = 3  4.8 / 6.6     5.0 / 7.6     6.1 / 11.9    11.3 / 24.5
//   application, tri. pairs k = 3 22.7 / 9.3    38.7 / 15.0   43.8 / 26.2   70.7 / 55.6
// and pairs at 16,384 | 33,000 groups: squares k = 2 179 / 194 | 332 / 376, k = 3 368 /
// 341 | 660 / 676; triangles k = 2 196 / 201 | 383 / 399, k = 3 456 / 357 | 894 / 715.
// (1216 groups are one wave of the four-warp team, eight blocks an SM.)  Large
// FP64 grids are bound by the FP64 pipe, and the thread form issues the fewer FP64
// instructions; large FP32 ones by memory, where its coalesced rows of one warp do
// as well with less code.
template <class T, int K>
struct TeamRule;
constexpr int TEAM_ALL = 1 << 30;
#define HHO_TEAM_RULE(T_, K_, W_, rect_, gen_, app_rect_, app_gen_, tr_rect_, tr_gen_)                      \
    template <>                                                                                             \
    struct TeamRule<T_, K_> {                                                                               \
        static constexpr int W = W_, rect = rect_, gen = gen_, app_rect = app_rect_, app_gen = app_gen_,     \
                             tr_rect = tr_rect_, tr_gen = tr_gen_;                                          \
    }
HHO_TEAM_RULE(double, 1, 8, 720, 1500, 1216, 1300, 400, 700);
HHO_TEAM_RULE(double, 2, 8, 650, 1000, 1100, 1216, 350, 680);
HHO_TEAM_RULE(double, 3, 10, 1050, 2000, 1216, 3500, 480, 850);
HHO_TEAM_RULE(f2x, 1, 8, 1300, 1900, 3700, 1500, 1216, 1216);
HHO_TEAM_RULE(f2x, 2, 8, 2000, 12000, 4000, 5500, 700, 1700);
HHO_TEAM_RULE(f2x, 3, 10, 24000, TEAM_ALL, 2900, 24000, 1300, 3500);
HHO_TEAM_RULE(float, 1, 8, 1216, 1216, 0, 0, 640, 600);
HHO_TEAM_RULE(float, 2, 8, 1216, 1216, 0, 0, 500, 300);
HHO_TEAM_RULE(float, 3, 10, 1216, 1216, 0, 0, 300, 250);
#undef HHO_TEAM_RULE

// Warps of a team block for this launch, 0 for the thread form.
template <class T, int K, int MODE>
int team_warps(const DevOps& op, int warps, int n_shots) {
    using R = TeamRule<T, K>;
    const int64_t cells = op.n_warps_f + op.n_warps_s, groups = (int64_t)warps * n_shots;
    const bool gen = 4 * (cells - op.n_warps_rect) >= cells;
    const int limit = MODE == MODE_TRACES  ? (gen ? R::tr_gen : R::tr_rect)
                      : MODE == MODE_APPLY ? (gen ? R::app_gen : R::app_rect)
                                           : (gen ? R::gen : R::rect);
    if (groups > limit || sizeof(T) * team_smem_elems<T, K>(op.max_nf) > 200 * 1024) return 0;
    return groups <= 600 || (K == 3 && sizeof(T) == 8) ? R::W : 4;
}

template <class T, int K, int MODE>
void launch_stage(const StageArgsT<T>& a, int n_shots, cudaStream_t s) {
    const int warps = a.n_warps ? a.n_warps : a.op.n_warps_f + a.op.n_warps_s;
    const int W = team_warps<T, K, MODE>(a.op, warps, n_shots);
    auto team = [&](auto wc) {
        constexpr int TW = decltype(wc)::value;
        const size_t smem = sizeof(T) * team_smem_elems<T, K>(a.op.max_nf);
        stage_smem_attributes<TeamTag<T, K, MODE, TW>>(team_kernel<T, K, MODE, TW>, smem, true);
        launch_dependent(team_kernel<T, K, MODE, TW>, dim3(warps, n_shots), 32 * TW, smem, s, a);
    };
    if (W == 4) return team(std::integral_constant<int, 4>());
    if (W) return team(std::integral_constant<int, TeamRule<T, K>::W>());
    const int cells = 32 * warps, threads = stage_threads((int64_t)warps * n_shots);
    const size_t smem = stage_smem_bytes<T, K>(a.op.max_nf, threads);
    stage_smem_attributes<StageTag<T, K, MODE>>(stage_kernel<T, K, MODE>, smem, AccSmem<T, K>::value);
    launch_dependent(stage_kernel<T, K, MODE>, dim3((cells + threads - 1) / threads, n_shots), threads, smem, s, a);
}

template <class T, int K>
void launch_grad(const StageArgsT<T>& a, const GradArgsT<T>& g, cudaStream_t s) {
    const int cells = a.op.Nf + a.op.Ns, threads = stage_threads(cells / 32);
    const size_t smem = stage_smem_bytes<T, K>(a.op.max_nf, threads);
    stage_smem_attributes<StageTag<T, K, MODE_GRAD>>(grad_stage_kernel<T, K>, smem, AccSmem<T, K>::value);
    launch_dependent(grad_stage_kernel<T, K>, dim3((cells + threads - 1) / threads, 2), threads, smem, s, a, g);
}

}  // namespace hho_stage
