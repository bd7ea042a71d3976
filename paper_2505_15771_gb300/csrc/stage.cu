// The time-stepping entry points on the stage kernels (stage_kernels.cuh): ERK
// plans, launch loops and graphs, the host-buffer and batched paths, receivers,
// energy, packing, the cost model, and the stage launchers of the adjoint and
// SDIRK drivers.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <functional>
#include <memory>
#include <type_traits>
#include <vector>

#include "basis.h"
#include "dependent_launch.cuh"
#include "f2x.cuh"
#include "hho_internal.h"
#include "host_buffers.h"
#include "host_pieces.h"
#include "stage_launch.h"

namespace {

// canonical (AoS, input cell order, FP64) <-> device layout (SoA by class, T);
// y = shot: canonical shot stride n_canon, state shot stride n_state.
// A block of 128 threads moves 32 consecutive device slots (a class run is
// padded to 32, so one domain) through shared memory: the device side in
// 32-element rows, the canonical side in the cells' own runs, which are
// adjacent where the class's cells are.  Bound by memory; one thread a cell
// walking its run took 152 us to unpack the 1024 x 512, k = 2 state (200 MB) and
// 2265 us for 16 FP32 shots of the 680 x 340, k = 3 hybrid mesh (2.2 GB).
constexpr int PACK_THREADS = 128;
template <class T, int NV, bool PACK>
__device__ __forceinline__ void pack_block(const int32_t* __restrict__ dev2orig, const int64_t* __restrict__ canon_off,
                                           int N, int q0, typename std::conditional<PACK, const double, double>::type* canon,
                                           typename std::conditional<PACK, T, const T>::type* st, T* run) {
    constexpr int LD = NV | 1;   // odd stride: a column of the tile has no bank conflicts
    __shared__ int64_t off[32];
    if (threadIdx.x < 32) {
        const int c = dev2orig[threadIdx.x];
        off[threadIdx.x] = c < 0 ? -1 : canon_off[c];
    }
    const int lane = threadIdx.x & 31, row0 = threadIdx.x >> 5;
    if constexpr (!PACK) {
#pragma unroll 8
        for (int i = row0; i < NV; i += PACK_THREADS / 32) run[lane * LD + i] = st[(size_t)i * N + q0 + lane];
    }
    __syncthreads();
#pragma unroll 8
    for (int e = threadIdx.x; e < 32 * NV; e += PACK_THREADS) {
        const int cell = e / NV, i = e - cell * NV;
        const int64_t o = off[cell];
        if constexpr (PACK) run[cell * LD + i] = o < 0 ? T(0) : from_f64<T>(canon[o + i]);
        else if (o >= 0) canon[o + i] = to_f64(run[cell * LD + i]);
    }
    if constexpr (PACK) {
        __syncthreads();
#pragma unroll 8
        for (int i = row0; i < NV; i += PACK_THREADS / 32) st[(size_t)i * N + q0 + lane] = run[lane * LD + i];
    }
}
template <class T, int K>
__global__ void __launch_bounds__(PACK_THREADS)
    pack_kernel(const int32_t* __restrict__ dev2orig, const int64_t* __restrict__ canon_off, int Nf, int Ns,
                int64_t n_canon, int64_t n_state, const double* __restrict__ canon, T* __restrict__ state) {
    constexpr int n = (K + 1) * (K + 2) / 2;
    __shared__ T run[32 * ((5 * n) | 1)];
    const int g = blockIdx.x * 32;
    const double* cv = canon + (size_t)blockIdx.y * n_canon;
    T* st = state + (size_t)blockIdx.y * n_state;
    if (g < Nf) pack_block<T, 3 * n, true>(dev2orig + g, canon_off, Nf, g, cv, st, run);
    else pack_block<T, 5 * n, true>(dev2orig + g, canon_off, Ns, g - Nf, cv, st + (size_t)3 * n * Nf, run);
}
template <class T, int K>
__global__ void __launch_bounds__(PACK_THREADS)
    unpack_kernel(const int32_t* __restrict__ dev2orig, const int64_t* __restrict__ canon_off, int Nf, int Ns,
                  int64_t n_canon, int64_t n_state, const T* __restrict__ state, double* __restrict__ canon) {
    constexpr int n = (K + 1) * (K + 2) / 2;
    __shared__ T run[32 * ((5 * n) | 1)];
    const int g = blockIdx.x * 32;
    double* cv = canon + (size_t)blockIdx.y * n_canon;
    const T* st = state + (size_t)blockIdx.y * n_state;
    if (g < Nf) pack_block<T, 3 * n, false>(dev2orig + g, canon_off, Nf, g, cv, st, run);
    else pack_block<T, 5 * n, false>(dev2orig + g, canon_off, Ns, g - Nf, cv, st + (size_t)3 * n * Nf, run);
}
template <class T, int K>
void launch_pack(const hho_ops* ops, int n_shots, const double* canon, T* state, cudaStream_t st) {
    const dim3 grid((ops->dev.Nf + ops->dev.Ns) / 32, n_shots);
    pack_kernel<T, K><<<grid, PACK_THREADS, 0, st>>>(ops->d_dev2orig, ops->d_canon_off, ops->dev.Nf, ops->dev.Ns,
                                                     ops->n_canonical, ops->n_state, canon, state);
}
template <class T, int K>
void launch_unpack(const hho_ops* ops, int n_shots, const T* state, double* canon, cudaStream_t st) {
    const dim3 grid((ops->dev.Nf + ops->dev.Ns) / 32, n_shots);
    unpack_kernel<T, K><<<grid, PACK_THREADS, 0, st>>>(ops->d_dev2orig, ops->d_canon_off, ops->dev.Nf, ops->dev.Ns,
                                                       ops->n_canonical, ops->n_state, state, canon);
}
template <class T>
void launch_pack(const hho_ops* ops, int n_shots, const double* canon, void* state, cudaStream_t st) {
    if (ops->k == 1) launch_pack<T, 1>(ops, n_shots, canon, (T*)state, st);
    else if (ops->k == 2) launch_pack<T, 2>(ops, n_shots, canon, (T*)state, st);
    else launch_pack<T, 3>(ops, n_shots, canon, (T*)state, st);
}
template <class T>
void launch_unpack(const hho_ops* ops, int n_shots, const void* state, double* canon, cudaStream_t st) {
    if (ops->k == 1) launch_unpack<T, 1>(ops, n_shots, (const T*)state, canon, st);
    else if (ops->k == 2) launch_unpack<T, 2>(ops, n_shots, (const T*)state, canon, st);
    else launch_unpack<T, 3>(ops, n_shots, (const T*)state, canon, st);
}

// Canonical vector in host memory (pinned, mapped into the device's address
// space) <-> device-layout state of type T.  A block of 64 threads takes 64
// consecutive canonical cells, whose values form one contiguous run: the run
// crosses the host link in coalesced 8-byte accesses (eight in flight per
// thread) and is reordered through shared memory, one thread per cell on the
// device side.  Padding slots of the state are not touched.
template <class T>
__global__ void __launch_bounds__(STAGED_CELLS) pack_host_kernel(const int32_t* __restrict__ cell_dom,
                                                                 const int32_t* __restrict__ cell_pos,
                                                                 const int64_t* __restrict__ canon_off, int nc,
                                                                 int64_t n_canon, int Nf, int Ns, int n,
                                                                 const double* __restrict__ canon,
                                                                 T* __restrict__ state, int block0) {
    extern __shared__ double run[];
    const int c0 = (block0 + blockIdx.x) * STAGED_CELLS;
    const int c1 = min(c0 + STAGED_CELLS, nc);
    const int64_t e0 = canon_off[c0];
    const int len = (int)((c1 < nc ? canon_off[c1] : n_canon) - e0);
    constexpr int U = 8;
    for (int b = 0; b < len; b += U * STAGED_CELLS) {
        double v[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int e = b + u * STAGED_CELLS + threadIdx.x;
            v[u] = e < len ? canon[e0 + e] : 0.0;
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int e = b + u * STAGED_CELLS + threadIdx.x;
            if (e < len) run[e] = v[u];
        }
    }
    __syncthreads();
    const int c = c0 + threadIdx.x;
    if (c >= c1) return;
    const bool fl = cell_dom[c] == 0;
    const int q = cell_pos[c];
    const int N = fl ? Nf : Ns;
    T* st = state + (fl ? 0 : (size_t)3 * n * Nf);
    const double* v = run + (canon_off[c] - e0);
    const int nv = (fl ? 3 : 5) * n;
    for (int i = 0; i < nv; ++i) st[(size_t)i * N + q] = from_f64<T>(v[i]);
}
template <class T>
__global__ void __launch_bounds__(STAGED_CELLS) unpack_host_kernel(const int32_t* __restrict__ cell_dom,
                                                                   const int32_t* __restrict__ cell_pos,
                                                                   const int64_t* __restrict__ canon_off, int nc,
                                                                   int64_t n_canon, int Nf, int Ns, int n,
                                                                   const T* __restrict__ state,
                                                                   double* __restrict__ canon, int block0) {
    extern __shared__ double run[];
    const int c0 = (block0 + blockIdx.x) * STAGED_CELLS;
    const int c1 = min(c0 + STAGED_CELLS, nc);
    const int64_t e0 = canon_off[c0];
    const int len = (int)((c1 < nc ? canon_off[c1] : n_canon) - e0);
    const int c = c0 + threadIdx.x;
    if (c < c1) {
        const bool fl = cell_dom[c] == 0;
        const int q = cell_pos[c];
        const int N = fl ? Nf : Ns;
        const T* st = state + (fl ? 0 : (size_t)3 * n * Nf);
        double* v = run + (canon_off[c] - e0);
        const int nv = (fl ? 3 : 5) * n;
        for (int i = 0; i < nv; ++i) v[i] = to_f64(st[(size_t)i * N + q]);
    }
    __syncthreads();
    for (int e = threadIdx.x; e < len; e += STAGED_CELLS) canon[e0 + e] = run[e];
}

// Energy 1/2 U^T M U (Sec. 5.1) with M = h^2 (material) x M0_ref per cell.
template <int K>
__global__ void __launch_bounds__(256) energy_kernel(DevOps op, const double* __restrict__ state,
                                                    const double* __restrict__ mass_f,
                                                    const double* __restrict__ mass_s, double* partial) {
    constexpr int n = (K + 1) * (K + 2) / 2;
    const int g = blockIdx.x * blockDim.x + threadIdx.x;
    double e = 0.0;
    if (g < op.Nf + op.Ns) {
        const bool fl = g < op.Nf;
        const int q = fl ? g : g - op.Nf;
        const int cls = op.warp_class[(fl ? 0 : op.n_warps_f) + (q >> 5)];
        const int* ci = op.cls_int + cls * CI_STRIDE;
        if (q - ci[CI_START] < ci[CI_COUNT]) {
            const double* M0 = op.cls_dbl + ci[CI_DOFF];
            const int N = fl ? op.Nf : op.Ns;
            const double* st = state + (fl ? 0 : (size_t)3 * n * op.Nf);
            auto quad = [&](int fa, int fb) {
                double s = 0.0;
                for (int i = 0; i < n; ++i) {
                    double r = 0.0;
                    for (int j = 0; j < n; ++j) r = fma(M0[i * n + j], st[(size_t)(fb * n + j) * N + q], r);
                    s = fma(st[(size_t)(fa * n + i) * N + q], r, s);
                }
                return s;
            };
            if (fl) {
                e = 0.5 * (mass_f[q] * (quad(0, 0) + quad(1, 1)) + mass_f[N + q] * quad(2, 2));
            } else {
                const double d0 = mass_s[q], d1 = mass_s[N + q], d2 = mass_s[2 * N + q], r = mass_s[3 * N + q];
                e = 0.5 * (d0 * (quad(0, 0) + quad(1, 1)) + 2.0 * d1 * quad(0, 1) + d2 * quad(2, 2) +
                           r * (quad(3, 3) + quad(4, 4)));
            }
        }
    }
    for (int o = 16; o > 0; o >>= 1) e += __shfl_down_sync(0xffffffffu, e, o);
    __shared__ double ws[8];
    if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = e;
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += ws[w];
        partial[blockIdx.x] = s;
    }
}

__global__ void sum_kernel(const double* __restrict__ partial, int np, double* out) {
    __shared__ double sh[256];
    double s = 0.0;
    for (int i = threadIdx.x; i < np; i += blockDim.x) s += partial[i];
    sh[threadIdx.x] = s;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if ((int)threadIdx.x < o) sh[threadIdx.x] += sh[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) out[0] = sh[0];
}

// Receivers: fluid [p, m_x, m_y, 0, 0]; solid [v_x, v_y, s_xx, s_yy, s_xy];
// interface [p_F, v_Fx, v_Fy, 0, 0] from the pointwise face solve.
// Eight lanes a receiver (y = shot), a field each: a lane issues its loads together
// and adds the field's coefficients up, and the pointwise solve goes through
// shuffles.  The chain of loads is two long, and FP64 instructions, 64 cycles each
// to a warp, are issued for all fields and four receivers at once.  Few
// receivers: blocks of one warp, so that they spread over the SMs.  us for 8 |
// 1000 | 20,000 | 100,000 receivers, k = 2: one thread a receiver 8.2 | 14.7 | 16.7 |
// 27.0, one block a receiver 6.8 | 6.7 | 21.4 | 101.5, this form 6.8 | 6.6 | 9.7 | 27.5.
// State shot stride n_state, output shot stride 5 n_rec; with a device clock (graph
// replay) out is the trace base, offset by the step, and the last block to have
// read the step advances it.
constexpr int REC_LANES = 8;   // three fields of the fluid cell, five of the solid cell
constexpr int REC_MAX_N = 10;
template <class T, class TO = T>
__global__ void __launch_bounds__(128)
    record_kernel(DevOps op, int n_rec, const int32_t* __restrict__ ri, const double* __restrict__ rd, const T* state,
                  int64_t n_state, TO* out, StageClock* clock = nullptr) {
    const int n = op.n, t = threadIdx.x % REC_LANES;
    const int at = blockIdx.x * (blockDim.x / REC_LANES) + threadIdx.x / REC_LANES;
    const int r = min(at, n_rec - 1);   // lanes past the last receiver follow it and store nothing
    const double* d = rd + (size_t)r * (2 * n + 15);
    const int kind = ri[4 * r], q = ri[4 * r + (t < 3 ? 1 : 2)];
    const bool use = kind == 2 || (t >= 3) == (kind == 1);
    const double* phi = kind == 2 && t >= 3 ? d + n : d;
    release_successor();
    wait_for_predecessor();
    const size_t N = t < 3 ? op.Nf : op.Ns;
    const T* field = state + (size_t)blockIdx.y * n_state + (t < 3 ? (size_t)t * n * N : (size_t)3 * n * op.Nf + (size_t)(t - 3) * n * N);
    T val[REC_MAX_N];
#pragma unroll
    for (int j = 0; j < REC_MAX_N; ++j)
        if (use && j < n) val[j] = field[j * N + q];
    if (clock) {
        __shared__ int64_t step;
        if (threadIdx.x == 0) {
            step = *(volatile int64_t*)&clock->step;
            __threadfence();   // the read comes before the ticket that lets the last block write
            if (atomicAdd(&clock->ticket, 1u) == gridDim.x * gridDim.y - 1) {   // every block has read it
                __threadfence();
                clock->ticket = 0;
                clock->step = step + 1;
            }
        }
        __syncthreads();
        out += (size_t)step * 5 * n_rec * gridDim.y;
    }
    double g = 0.0;   // lane t: fluid m_x, m_y, p; solid s_xx, s_yy, s_xy, v_x, v_y
#pragma unroll
    for (int j = 0; j < REC_MAX_N; ++j)
        if (use && j < n) g = fma(phi[j], double(val[j]), g);
    auto of = [](double x, int lane) { return __shfl_sync(0xffffffffu, x, lane, REC_LANES); };
    // plain receivers: [p, m_x, m_y] or [v_x, v_y, s_xx, s_yy, s_xy]
    double o = of(g, kind == 0 ? (t == 0 ? 2 : t == 1 ? 0 : 1) : (t < 2 ? 6 + t : t < 5 ? 1 + t : 0));
    // interface: lanes 0..2 the fluxes tau_f p - m.n_f, tau_s v - s n_s
    const double u = of(g, t == 0 ? 2 : t == 1 ? 6 : 7), a = of(g, t == 0 ? 0 : t == 1 ? 3 : 5),
                 b = of(g, t == 0 ? 1 : t == 1 ? 5 : 4);
    double flux = 0.0;
    if (kind == 2) {
        const double* c = d + 2 * n;   // tau_f, tau_s, n_f, n_s
        flux = c[t == 0 ? 0 : 1] * u - (a * c[t == 0 ? 2 : 4] + b * c[t == 0 ? 3 : 5]);
    }
    const double w0 = of(flux, 0), w1 = of(flux, 1), w2 = of(flux, 2);
    if (kind == 2 && t < 3) {
        const double* Ai = d + 2 * n + 6 + 3 * t;
        o = Ai[0] * w0 + Ai[1] * w1 + Ai[2] * w2;
    }
    if (at < n_rec && t < 5) out[(size_t)blockIdx.y * 5 * n_rec + 5 * r + t] = TO(kind != 1 && t >= 3 ? 0.0 : o);
}

template <class T, class TO>
void launch_record(const hho_ops* ops, int n_shots, const T* state, TO* out, StageClock* clock, cudaStream_t st) {
    const int threads = (int64_t)ops->n_rec * n_shots <= 16 * GB300_SMS ? 32 : 128, per = threads / REC_LANES;
    launch_dependent(record_kernel<T, TO>, dim3((ops->n_rec + per - 1) / per, n_shots), threads, 0, st, ops->dev,
                     ops->n_rec, ops->d_rec_int, ops->d_rec_dbl, state, ops->n_state, out, clock);
}

template <class T, int MODE>
void launch_k(int k, const StageArgsT<T>& a, int n_shots, cudaStream_t s) {
    if (k == 1) hho_stage::launch_stage<T, 1, MODE>(a, n_shots, s);
    else if (k == 2) hho_stage::launch_stage<T, 2, MODE>(a, n_shots, s);
    else hho_stage::launch_stage<T, 3, MODE>(a, n_shots, s);
}

// A stage launch of erk_run: the tensor-core stage when the batched call
// asked for HHO_BF16X3, else the stage kernel of the arithmetic.
template <class T, int MODE>
void launch_stage(const hho_ops* ops, const StageArgsT<T>& a, int n_shots, cudaStream_t s) {
    if constexpr (std::is_same<T, float>::value) {
        if (ops->tc_on) {
            if (ops->k == 1) hho_stage::launch_tc<1, MODE>(ops, a, n_shots, s);
            else if (ops->k == 2) hho_stage::launch_tc<2, MODE>(ops, a, n_shots, s);
            else hho_stage::launch_tc<3, MODE>(ops, a, n_shots, s);
            return;
        }
    }
    launch_k<T, MODE>(ops->k, a, n_shots, s);
}

}  // namespace

int build_plan(const hho_tableau* tab, std::vector<StagePlan>& plan, int* n_buf) {
    const int s = tab->s;
    if (s < 1 || s > 6) return HHO_EINVAL;
    auto coef = [&](int i, int j) { return i == s ? tab->b[j] : tab->a[i][j]; };
    std::vector<int> buf(s + 1, -1);      // row -> buffer index
    std::vector<bool> touched(s + 1, false);
    int nb = 0;
    plan.assign(s, StagePlan{});
    for (int j = 0; j < s; ++j) {
        StagePlan& P = plan[j];
        P.n_tgt = 0;
        const int r0 = j + 1;
        TargetPlan t0;
        t0.src = touched[r0] ? buf[r0] : SRC_STATE;
        t0.dst = (r0 == s) ? SRC_STATE : SRC_X;
        t0.a = coef(r0, j);
        P.t[P.n_tgt++] = t0;
        for (int i = j + 2; i <= s; ++i) {
            const double a = coef(i, j);
            if (a == 0.0) continue;
            if (P.n_tgt >= MAX_PLAN_TARGETS) return HHO_EINVAL;
            if (buf[i] < 0) buf[i] = nb++;
            TargetPlan t;
            t.src = touched[i] ? buf[i] : SRC_STATE;
            t.dst = buf[i];
            t.a = a;
            touched[i] = true;
            P.t[P.n_tgt++] = t;
        }
    }
    *n_buf = nb;
    return HHO_OK;
}

namespace {

int64_t n_energy_blocks(const hho_ops* ops) { return ((int64_t)ops->dev.Nf + ops->dev.Ns + 255) / 256 + 1; }

double ricker(double t, double f0, double t0, double amp) {
    const double a = M_PI * f0 * (t - t0);
    const double a2 = a * a;
    return amp * (1.0 - 2.0 * a2) * std::exp(-a2);
}

int check_launch(const char* what) {
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) {
        hho_set_error("%s: %s", what, cudaGetErrorString(e));
        return HHO_ECUDA;
    }
    return HHO_OK;
}

template <class T>
const T* src_g_of(const hho_ops* ops);
template <>
const double* src_g_of<double>(const hho_ops* ops) { return ops->d_src_g; }
template <>
const float* src_g_of<float>(const hho_ops* ops) { return ops->d_src_g32; }
template <>
const f2x* src_g_of<f2x>(const hho_ops* ops) { return ops->d_src_gx; }
template <class T>
const T* shot_g_of(const hho_ops* ops);
template <>
const double* shot_g_of<double>(const hho_ops* ops) { return ops->d_shot_src_g; }
template <>
const float* shot_g_of<float>(const hho_ops* ops) { return ops->d_shot_src_g32; }
template <>
const f2x* shot_g_of<f2x>(const hho_ops* ops) { return ops->d_shot_src_gx; }

// Value of point source s for the stage of step time tn, stage j (time
// tn + cdt): its Ricker wavelet, or, for a sampled time function, the sample
// of step round((tn - t_start) / dt) and stage j (zero outside the sampled
// steps and for j < 0, a call with no stage index).
double source_value(const hho_ops* ops, int s, double tn, int j, double cdt) {
    if (!ops->src_sampled) return ricker(tn + cdt, ops->src_f0[s], ops->src_t0[s], ops->src_amp[s]);
    if (j < 0 || j >= ops->samp_s) return 0.0;
    const int64_t n = std::llround((tn - ops->samp_t0) / ops->samp_dt);
    if (n < 0 || n >= ops->samp_n) return 0.0;
    return ops->src_samples[((size_t)s * ops->samp_n + n) * ops->samp_s + j];
}

template <class T>
void fill_sources(const hho_ops* ops, StageArgsT<T>& a, double tn, int j, double cdt, int n_shots) {
    a.n_src = ops->n_src;
    a.src_g = src_g_of<T>(ops);
    for (int s = 0; s < ops->n_src; ++s) {
        a.src_dom[s] = ops->src_dom[s];
        a.src_q[s] = ops->src_q[s];
        a.src_w[s] = T(source_value(ops, s, tn, j, cdt));
    }
    if (ops->n_shot_src > 0 && n_shots <= ops->n_shot_src) {
        a.shot_src_dom = ops->d_shot_src_dom;
        a.shot_src_q = ops->d_shot_src_q;
        a.shot_src_g = shot_g_of<T>(ops);
        a.shot_src_w = T(ricker(tn + cdt, ops->shot_f0, ops->shot_t0, ops->shot_amp));
    } else {
        a.shot_src_dom = nullptr;
        a.shot_src_q = nullptr;
        a.shot_src_g = nullptr;
        a.shot_src_w = T(0);
    }
}

}  // namespace

extern "C" int hho_ricker_samples(const hho_tableau* tab, double t_start, double dt, int64_t nsteps, double f0,
                                  double t0, double amp, double* h_out) {
    if (!tab || tab->s < 1 || tab->s > 6 || nsteps < 0 || !(dt > 0.0) || !std::isfinite(dt) ||
        !std::isfinite(t_start) || !(f0 > 0.0) || (nsteps > 0 && !h_out)) {
        hho_set_error("hho_ricker_samples: bad arguments");
        return HHO_EINVAL;
    }
    // the same rounded stage times as the ERK loops: (t_start + n dt) + c_j dt
    for (int64_t n = 0; n < nsteps; ++n) {
        const double tn = t_start + (double)n * dt;
        for (int j = 0; j < tab->s; ++j) h_out[n * tab->s + j] = ricker(tn + tab->c[j] * dt, f0, t0, amp);
    }
    return HHO_OK;
}

extern "C" int hho_work_size(const hho_ops* ops, const hho_tableau* tab, int64_t* out) {
    if (!ops || !tab || !out) {
        hho_set_error("hho_work_size: null pointer");
        return HHO_EINVAL;
    }
    std::vector<StagePlan> plan;
    int nb = 0;
    if (build_plan(tab, plan, &nb) != HHO_OK) {
        hho_set_error("hho_work_size: unsupported tableau");
        return HHO_EINVAL;
    }
    *out = ops->n_state * (2 + nb) + 2 * ops->trace_doubles + n_energy_blocks(ops) + 8;
    return HHO_OK;
}

namespace {
__global__ void clock_set_kernel(StageClock* c, double t0) {
    c->t0 = t0;
    c->step = 0;
    c->ticket = 0;
}
__global__ void clock_advance_kernel(StageClock* c) { c->step += 1; }

// Sources for a stage evaluated from the device clock (graph replay).
template <class T>
void fill_sources_clock(const hho_ops* ops, StageArgsT<T>& a, double c_stage, double dt, int n_shots) {
    fill_sources<T>(ops, a, 0.0, -1, 0.0, n_shots);   // cells, vectors and pointers
    for (int s = 0; s < MAX_SOURCES; ++s) a.src_w[s] = T(0);
    a.shot_src_w = T(0);
    a.clock = ops->d_clock;
    a.dt = dt;
    a.c_stage = c_stage;
    for (int s = 0; s < ops->n_src; ++s) {
        a.src_f0[s] = ops->src_f0[s];
        a.src_t0[s] = ops->src_t0[s];
        a.src_amp[s] = ops->src_amp[s];
    }
    if (a.shot_src_q) {
        a.shot_f0 = ops->shot_f0;
        a.shot_t0 = ops->shot_t0;
        a.shot_amp = ops->shot_amp;
    }
}

template <class V>
void append_bytes(std::vector<unsigned char>& key, const V& v) {
    const unsigned char* p = reinterpret_cast<const unsigned char*>(&v);
    key.insert(key.end(), p, p + sizeof(V));
}
}  // namespace

// Time stepping for n_shots states of element type T.  Work layout (elements
// of T): [X: S n_state][partial sums: nb S n_state][traces: 2 x S trace].
template <class T>
struct SeisOf {   // element type of recorded traces: the state's, FP64 for double-float
    using type = T;
};
template <>
struct SeisOf<f2x> {
    using type = double;
};

// What a host-buffer call in pieces (HostPieces) keeps with the operator: its copy
// stream and the events of the pieces.
struct HostPipe {
    cudaStream_t copy = nullptr;
    cudaEvent_t start = nullptr, in[HostPieces::MAX] = {}, out[HostPieces::MAX] = {};
};

// Whether erk_run replays the step as a graph.  AUTO does not: consecutive stages
// of a stream are dependent launches that overlap across steps too, while a graph
// ends with its step, and the host launches a stage in less time than the
// smallest one runs (512 triangles, k = 1, four stages and a record: 28.3 us a
// step launched, 36.9 replayed).
static bool uses_graph(const hho_ops* ops) {
    return !ops->prof_on && ops->d_clock && !ops->src_sampled && ops->launch_mode == HHO_LAUNCH_GRAPH;
}

// A call that takes its state and hands it back in pieces (HostPieces): arrive(c)
// enqueues host piece c into the state, leave(c) out of it.
struct PieceHooks {
    std::function<int(int)> arrive, leave;
};

// The first stage (its pieces follow their arrivals and the traces they need),
// the last one (its pieces are followed by the host pieces they complete), or a
// stage that is both.
template <class T>
static int stage_pieces(const hho_ops* ops, const StageArgsT<T>& traces, const StageArgsT<T>& stage,
                        const PieceHooks& hooks, bool first, bool last, cudaStream_t st) {
    const HostPieces& p = ops->host_pieces;
    auto part = [&](StageArgsT<T> a, int d) {
        a.warp0 = p.warps[d];
        a.n_warps = p.warps[d + 1] - p.warps[d];
        return a;
    };
    int rc = HHO_OK;
    for (int c = 0, i = 0; c < p.n && !rc; ++c) {
        if (first) {
            rc = hooks.arrive(c);
            for (int d = 0; d < p.n && !rc; ++d)
                if (p.own[d] == c) launch_stage<T, MODE_TRACES>(ops, part(traces, d), 1, st);
        }
        for (; i < p.n && !rc && (!first || p.need[p.order[i]] <= c); ++i) {
            launch_stage<T, MODE_STAGE>(ops, part(stage, p.order[i]), 1, st);
            for (int h = 0; h < p.n && last && !rc; ++h)
                if (p.last[h] == i) rc = hooks.leave(h);
        }
    }
    return rc;
}

template <class T>
static int erk_run(hho_ops* ops, const hho_tableau* tab, double t0, double dt, int64_t nsteps, int n_shots,
                   T* d_state, T* d_work, void* d_seis_v, void* stream, const char* who,
                   const PieceHooks* pieces = nullptr) {
    using TS = typename SeisOf<T>::type;
    TS* d_seis = (TS*)d_seis_v;
    if (!ops || !tab || !d_state || !d_work || nsteps < 0 || n_shots < 1 || n_shots > 65535 || !std::isfinite(dt) ||
        !std::isfinite(t0)) {
        hho_set_error("%s: bad arguments", who);
        return HHO_EINVAL;
    }
    std::vector<StagePlan> plan;
    int nb = 0;
    if (build_plan(tab, plan, &nb) != HHO_OK) {
        hho_set_error("%s: unsupported tableau (s <= 6, at most %d partial sums per stage)", who, MAX_PLAN_TARGETS);
        return HHO_EINVAL;
    }
    if (nsteps == 0) return HHO_OK;
    cudaStream_t st = (cudaStream_t)stream;
    const int64_t S = ops->n_state * n_shots;
    const int64_t TRS = ops->trace_doubles * n_shots;
    T* X = d_work;
    T* bufs = d_work + S;
    T* tr[2] = {d_work + S * (1 + nb), d_work + S * (1 + nb) + TRS};
    const dim3 grid((ops->dev.Nf + ops->dev.Ns + 127) / 128, n_shots);
    if (grid.x == 0) return HHO_OK;
    auto resolve = [&](int code) -> T* {
        if (code == SRC_STATE) return d_state;
        if (code == SRC_X) return X;
        if (code == SRC_ZERO) return nullptr;
        return bufs + S * code;
    };
    StageArgsT<T> a;
    memset(&a, 0, sizeof(a));
    a.op = ops->dev;
    a.state_stride = ops->n_state;
    a.trace_stride = ops->trace_doubles;
    a.inp = d_state;
    a.tr_out = tr[0];
    a.n_tgt = 0;
    const bool use_graph = uses_graph(ops);
    const StageArgsT<T> traces = a;
    int rc = HHO_OK;
    if (!pieces) {
        launch_stage<T, MODE_TRACES>(ops, traces, n_shots, st);
        rc = check_launch(who);
        if (rc) return rc;
    }
    int cur = 0;
    if (use_graph) {
        // One step = its stage kernels, the receiver record and the clock
        // increment, captured once per distinct set of arguments (two sets
        // when an odd stage count alternates the trace buffers) and replayed.
        clock_set_kernel<<<1, 1, 0, st>>>(ops->d_clock, t0);
        rc = check_launch(who);
        if (rc) return rc;
        const bool rec = d_seis && ops->n_rec > 0;
        cudaGraphExec_t execs[2] = {nullptr, nullptr};
        for (int par = 0; par < ((tab->s & 1) ? 2 : 1); ++par) {
            std::vector<StageArgsT<T>> args(tab->s);
            int c2 = par;
            std::vector<unsigned char> key;
            append_bytes(key, (int)sizeof(T));
            append_bytes(key, ops->tc_on);
            append_bytes(key, grid);
            for (int j = 0; j < tab->s; ++j) {
                StageArgsT<T>& b = args[j];
                b = a;
                const StagePlan& P = plan[j];
                b.inp = (j == 0) ? d_state : X;
                b.tr_in = tr[c2];
                b.tr_out = tr[c2 ^ 1];
                b.n_tgt = P.n_tgt;
                for (int t = 0; t < P.n_tgt; ++t) {
                    b.tgt[t].src = resolve(P.t[t].src);
                    b.tgt[t].dst = resolve(P.t[t].dst);
                    b.tgt[t].coef = T(P.t[t].a * dt);
                }
                fill_sources_clock<T>(ops, b, tab->c[j], dt, n_shots);
                append_bytes(key, b);
                c2 ^= 1;
            }
            append_bytes(key, rec ? (const void*)d_seis : nullptr);
            append_bytes(key, ops->d_rec_int);
            append_bytes(key, ops->d_rec_dbl);
            append_bytes(key, ops->n_rec);
            cudaGraphExec_t found = nullptr;
            for (auto& g : ops->graphs)
                if (g.key == key) found = (cudaGraphExec_t)g.exec;
            if (!found) {
                if (!ops->cap_stream) {
                    cudaStream_t cs;
                    if (cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking) != cudaSuccess) {
                        hho_set_error("%s: capture stream creation failed", who);
                        return HHO_ECUDA;
                    }
                    ops->cap_stream = (void*)cs;
                }
                cudaStream_t cs = (cudaStream_t)ops->cap_stream;
                cudaGraph_t graph = nullptr;
                if (cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal) != cudaSuccess) {
                    hho_set_error("%s: stream capture failed to start", who);
                    return HHO_ECUDA;
                }
                for (int j = 0; j < tab->s; ++j) launch_stage<T, MODE_STAGE>(ops, args[j], n_shots, cs);
                if (rec)   // advances the clock too
                    launch_record<T, TS>(ops, n_shots, d_state, d_seis, ops->d_clock, cs);
                else
                    clock_advance_kernel<<<1, 1, 0, cs>>>(ops->d_clock);
                const cudaError_t ce = cudaStreamEndCapture(cs, &graph);
                if (ce != cudaSuccess || !graph || cudaGraphInstantiate(&found, graph, 0) != cudaSuccess) {
                    if (graph) cudaGraphDestroy(graph);
                    cudaGetLastError();
                    hho_set_error("%s: step graph capture or instantiation failed", who);
                    return HHO_ECUDA;
                }
                cudaGraphDestroy(graph);
                if (ops->graphs.size() >= 8) {
                    cudaGraphExecDestroy((cudaGraphExec_t)ops->graphs.front().exec);
                    ops->graphs.erase(ops->graphs.begin());
                }
                ops->graphs.push_back({key, (void*)found});
            }
            execs[par] = found;
        }
        for (int64_t step = 0; step < nsteps; ++step) {
            if (cudaGraphLaunch(execs[(tab->s & 1) ? (int)(step & 1) : 0], st) != cudaSuccess) {
                hho_set_error("%s: graph launch failed", who);
                return HHO_ECUDA;
            }
        }
        return check_launch(who);
    }
    for (int64_t step = 0; step < nsteps; ++step) {
        const double tn = t0 + (double)step * dt;
        for (int j = 0; j < tab->s; ++j) {
            const StagePlan& P = plan[j];
            a.inp = (j == 0) ? d_state : X;
            a.tr_in = tr[cur];
            a.tr_out = tr[cur ^ 1];
            a.n_tgt = P.n_tgt;
            for (int t = 0; t < P.n_tgt; ++t) {
                a.tgt[t].src = resolve(P.t[t].src);
                a.tgt[t].dst = resolve(P.t[t].dst);
                a.tgt[t].coef = T(P.t[t].a * dt);
            }
            fill_sources<T>(ops, a, tn, j, tab->c[j] * dt, n_shots);
            const bool prof = ops->prof_on && 2 * ops->prof_n + 1 < (int)ops->prof_events.size();
            if (prof) cudaEventRecord((cudaEvent_t)ops->prof_events[2 * ops->prof_n], st);
            const bool first = pieces && step == 0 && j == 0, last = pieces && step == nsteps - 1 && j == tab->s - 1;
            if (first || last) rc = stage_pieces<T>(ops, traces, a, *pieces, first, last, st);
            else launch_stage<T, MODE_STAGE>(ops, a, n_shots, st);
            if (prof) cudaEventRecord((cudaEvent_t)ops->prof_events[2 * ops->prof_n++ + 1], st);
            if (!rc) rc = check_launch(who);
            if (rc) return rc;
            cur ^= 1;
        }
        if (d_seis && ops->n_rec > 0) {
            launch_record<T, TS>(ops, n_shots, d_state, d_seis + (size_t)step * 5 * ops->n_rec * n_shots, nullptr, st);
            rc = check_launch(who);
            if (rc) return rc;
        }
    }
    return HHO_OK;
}

// Doubles of the FP64 work layout [X][partial sums][2 traces][energy scratch];
// hho_work_size adds one state of double-float pairs after it.
static int64_t work_f64_part(const hho_ops* ops, int nb) {
    return ops->n_state * (1 + nb) + 2 * ops->trace_doubles + n_energy_blocks(ops) + 8;
}

namespace {
__global__ void to_pairs_kernel(const double* __restrict__ x, f2x* __restrict__ y, int64_t n) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        y[i] = f64_to_pair(x[i]);
}
__global__ void from_pairs_kernel(const f2x* __restrict__ x, double* __restrict__ y, int64_t n) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        y[i] = pair_to_f64(x[i]);
}
int pairs_grid(int64_t n) { return (int)std::min<int64_t>((n + 255) / 256, GB300_SMS * 16); }
}  // namespace

// Single-shot stepping: FP64, or double-float on a pair copy of the state
// kept at the end of the work buffer (converted in and out once per call).
static int erk_single(hho_ops* ops, const hho_tableau* tab, double t0, double dt, int64_t nsteps, double* d_state,
                      double* d_work, double* d_seis, void* stream, const char* who) {
    if (!ops || ops->arith != HHO_F32X2)
        return erk_run<double>(ops, tab, t0, dt, nsteps, 1, d_state, d_work, d_seis, stream, who);
    std::vector<StagePlan> plan;
    int nb = 0;
    if (!tab || !d_state || !d_work || build_plan(tab, plan, &nb) != HHO_OK) {
        hho_set_error("%s: bad arguments", who);
        return HHO_EINVAL;
    }
    if (nsteps <= 0 || ops->n_state == 0)
        return erk_run<f2x>(ops, tab, t0, dt, nsteps, 1, (f2x*)d_state, (f2x*)d_work, d_seis, stream, who);
    cudaStream_t st = (cudaStream_t)stream;
    f2x* ux = (f2x*)(d_work + work_f64_part(ops, nb));
    to_pairs_kernel<<<pairs_grid(ops->n_state), 256, 0, st>>>(d_state, ux, ops->n_state);
    int rc = check_launch(who);
    if (rc) return rc;
    rc = erk_run<f2x>(ops, tab, t0, dt, nsteps, 1, ux, (f2x*)d_work, d_seis, stream, who);
    if (rc) return rc;
    from_pairs_kernel<<<pairs_grid(ops->n_state), 256, 0, st>>>(ux, d_state, ops->n_state);
    return check_launch(who);
}

template <class T>
static int launch_host_pack(const hho_ops* ops, const double* canon, T* state, int block0, int blocks, cudaStream_t st) {
    const size_t smem = sizeof(double) * STAGED_CELLS * 5 * ops->n;
    pack_host_kernel<T><<<blocks, STAGED_CELLS, smem, st>>>(ops->d_cell_dom, ops->d_cell_pos, ops->d_canon_off,
                                                            (int)ops->nc, ops->n_canonical, ops->dev.Nf, ops->dev.Ns,
                                                            ops->n, canon, state, block0);
    return check_launch("hho_erk_run_host");
}
template <class T>
static int launch_host_unpack(const hho_ops* ops, const T* state, double* canon, int block0, int blocks, cudaStream_t st) {
    const size_t smem = sizeof(double) * STAGED_CELLS * 5 * ops->n;
    unpack_host_kernel<T><<<blocks, STAGED_CELLS, smem, st>>>(ops->d_cell_dom, ops->d_cell_pos, ops->d_canon_off,
                                                              (int)ops->nc, ops->n_canonical, ops->dev.Nf, ops->dev.Ns,
                                                              ops->n, state, canon, block0);
    return check_launch("hho_erk_run_host");
}

void free_host_pipe(HostPipe* p) {
    if (!p) return;
    for (int c = 0; c < HostPieces::MAX; ++c) {
        if (p->in[c]) cudaEventDestroy(p->in[c]);
        if (p->out[c]) cudaEventDestroy(p->out[c]);
    }
    if (p->start) cudaEventDestroy(p->start);
    if (p->copy) cudaStreamDestroy(p->copy);
    delete p;
}

static HostPipe* host_pipe(hho_ops* ops) {
    if (ops->host_pipe) return ops->host_pipe;
    std::unique_ptr<HostPipe, void (*)(HostPipe*)> p(new HostPipe, free_host_pipe);
    bool ok = cudaStreamCreateWithFlags(&p->copy, cudaStreamNonBlocking) == cudaSuccess &&
              cudaEventCreateWithFlags(&p->start, cudaEventDisableTiming) == cudaSuccess;
    for (int c = 0; c < ops->host_pieces.n; ++c)
        ok = ok && cudaEventCreateWithFlags(&p->in[c], cudaEventDisableTiming) == cudaSuccess &&
             cudaEventCreateWithFlags(&p->out[c], cudaEventDisableTiming) == cudaSuccess;
    return ok ? ops->host_pipe = p.release() : nullptr;
}

// hho_erk_run_host on a pinned host buffer: the state is packed into the
// arithmetic's device state (the double-float pair copy, or the FP64 state),
// stepped and unpacked.  Small meshes: the pack kernels read and write the
// mapped buffer themselves.  Large ones, but for buffers made in the call: in
// pieces (HostPieces) through the device's canonical buffer by the copy engine,
// which moves the same bytes a second (209 GB/s in, 191 out) without holding SM
// resources.
template <class T>
static int erk_run_pinned(hho_ops* ops, const hho_tableau* tab, double t0, double dt, int64_t nsteps,
                          double* h_canonical, double* m_canonical, T* dst, bool made, cudaStream_t st) {
    const char* who = "hho_erk_run_host";
    const int nc = (int)ops->nc;
    if (nc == 0) return HHO_OK;
    const int blocks = (nc + STAGED_CELLS - 1) / STAGED_CELLS, np = host_pieces(ops, nsteps, uses_graph(ops), made);
    if (np == 1) {
        int rc = launch_host_pack<T>(ops, m_canonical, dst, 0, blocks, st);
        if (!rc) rc = erk_run<T>(ops, tab, t0, dt, nsteps, 1, dst, (T*)ops->d_host_work, nullptr, st, who);
        if (!rc) rc = launch_host_unpack<T>(ops, dst, m_canonical, 0, blocks, st);
        if (!rc && ops->host_pieces.n == 0) cut_host_pieces(ops);   // while the GPU works
        return rc;
    }
    const HostPieces& cut = ops->host_pieces;
    HostPipe* p = host_pipe(ops);
    if (!p) {
        cudaGetLastError();
        hho_set_error("%s: stream or event creation failed", who);
        return HHO_ECUDA;
    }
    auto ok = [&](cudaError_t e) {
        if (e != cudaSuccess) hho_set_error("%s: %s", who, cudaGetErrorString(e));
        return e == cudaSuccess;
    };
    double* canon = ops->d_host_canon;
    auto bytes = [&](int c) { return sizeof(double) * (size_t)(cut.off[c + 1] - cut.off[c]); };
    PieceHooks hooks{[&](int c) -> int {   // host piece c arrives
                         if (!ok(cudaStreamWaitEvent(st, p->in[c], 0))) return HHO_ECUDA;
                         return launch_host_pack<T>(ops, canon, dst, cut.blocks[c], cut.blocks[c + 1] - cut.blocks[c], st);
                     },
                     [&](int c) -> int {   // and leaves
                         const int rc = launch_host_unpack<T>(ops, dst, canon, cut.blocks[c],
                                                              cut.blocks[c + 1] - cut.blocks[c], st);
                         if (rc) return rc;
                         if (!ok(cudaEventRecord(p->out[c], st)) || !ok(cudaStreamWaitEvent(p->copy, p->out[c], 0)) ||
                             !ok(cudaMemcpyAsync(h_canonical + cut.off[c], canon + cut.off[c], bytes(c),
                                                 cudaMemcpyDeviceToHost, p->copy)))
                             return HHO_ECUDA;
                         return HHO_OK;
                     }};
    int rc = HHO_OK;
    if (!ok(cudaEventRecord(p->start, st)) || !ok(cudaStreamWaitEvent(p->copy, p->start, 0))) rc = HHO_ECUDA;
    for (int c = 0; c < np && !rc; ++c)
        if (!ok(cudaMemcpyAsync(canon + cut.off[c], h_canonical + cut.off[c], bytes(c), cudaMemcpyHostToDevice, p->copy)) ||
            !ok(cudaEventRecord(p->in[c], p->copy)))
            rc = HHO_ECUDA;
    if (!rc) rc = erk_run<T>(ops, tab, t0, dt, nsteps, 1, dst, (T*)ops->d_host_work, nullptr, st, who, &hooks);
    if (!ok(cudaStreamSynchronize(p->copy)) && !rc) rc = HHO_ECUDA;   // the buffer is the caller's again
    return rc;
}

static int erk_run_mapped(hho_ops* ops, const hho_tableau* tab, double t0, double dt, int64_t nsteps,
                          double* h_canonical, double* m_canonical, bool made, cudaStream_t st) {
    std::vector<StagePlan> plan;
    int nb = 0;
    if (build_plan(tab, plan, &nb) != HHO_OK) {
        hho_set_error("hho_erk_run_host: unsupported tableau");
        return HHO_EINVAL;
    }
    if (ops->arith == HHO_F32X2)
        return erk_run_pinned<f2x>(ops, tab, t0, dt, nsteps, h_canonical, m_canonical,
                                   (f2x*)(ops->d_host_work + work_f64_part(ops, nb)), made, st);
    return erk_run_pinned<double>(ops, tab, t0, dt, nsteps, h_canonical, m_canonical, ops->d_host_state, made, st);
}

extern "C" int hho_set_launch_mode(hho_ops* ops, int32_t mode) {
    if (!ops || (mode != HHO_LAUNCH_STREAM && mode != HHO_LAUNCH_GRAPH && mode != HHO_LAUNCH_AUTO)) {
        hho_set_error("hho_set_launch_mode: mode must be HHO_LAUNCH_STREAM, HHO_LAUNCH_GRAPH or HHO_LAUNCH_AUTO");
        return HHO_EINVAL;
    }
    ops->launch_mode = mode;
    return HHO_OK;
}

extern "C" int hho_set_arithmetic(hho_ops* ops, int32_t arith) {
    if (!ops || (arith != HHO_F64 && arith != HHO_F32X2)) {
        hho_set_error("hho_set_arithmetic: arith must be HHO_F64 or HHO_F32X2");
        return HHO_EINVAL;
    }
    ops->arith = arith;
    return HHO_OK;
}

extern "C" int hho_erk_step(hho_ops* ops, const hho_tableau* tab, double t0, double dt, int64_t nsteps,
                            double* d_state, double* d_work, void* stream) {
    return erk_single(ops, tab, t0, dt, nsteps, d_state, d_work, nullptr, stream, "hho_erk_step");
}

extern "C" int hho_erk_step_record(hho_ops* ops, const hho_tableau* tab, double t0, double dt, int64_t nsteps,
                                   double* d_state, double* d_work, double* d_seismogram, void* stream) {
    if (ops && ops->n_rec > 0 && !d_seismogram) {
        hho_set_error("hho_erk_step_record: null seismogram buffer");
        return HHO_EINVAL;
    }
    return erk_single(ops, tab, t0, dt, nsteps, d_state, d_work, d_seismogram, stream, "hho_erk_step_record");
}

// ---- one stage at a time (drivers that exchange halos between stages) ---------------
// The same kernel arguments as erk_run's stream path, so a sequence
// hho_erk_traces, hho_erk_stage(n, j) for n < nsteps, j < s reproduces
// hho_erk_step in stream launch mode bit for bit.

namespace {
__global__ void halo_gather_kernel(const double* __restrict__ src, const int64_t* __restrict__ idx, int64_t n,
                                   double* __restrict__ dst) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        dst[i] = src[idx[i]];
}
__global__ void halo_scatter_kernel(const double* __restrict__ src, const int64_t* __restrict__ idx, int64_t n,
                                    double* __restrict__ dst) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        dst[idx[i]] = src[i];
}
}  // namespace

static int stage_api_check(const hho_ops* ops, const hho_tableau* tab, const void* d_state, const void* d_work,
                           std::vector<StagePlan>& plan, int* nb, const char* who) {
    if (!ops || !tab || !d_state || !d_work) {
        hho_set_error("%s: null pointer", who);
        return HHO_EINVAL;
    }
    if (ops->arith != HHO_F64) {
        hho_set_error("%s: the stage-at-a-time entry points run the FP64 arithmetic only", who);
        return HHO_EINVAL;
    }
    if (build_plan(tab, plan, nb) != HHO_OK) {
        hho_set_error("%s: unsupported tableau", who);
        return HHO_EINVAL;
    }
    return HHO_OK;
}

extern "C" int hho_trace_buffer_offset(const hho_ops* ops, const hho_tableau* tab, int32_t which, int64_t* offset) {
    std::vector<StagePlan> plan;
    int nb = 0;
    if (!ops || !tab || !offset || (which != 0 && which != 1) || build_plan(tab, plan, &nb) != HHO_OK) {
        hho_set_error("hho_trace_buffer_offset: bad arguments");
        return HHO_EINVAL;
    }
    *offset = ops->n_state * (1 + nb) + (int64_t)which * ops->trace_doubles;
    return HHO_OK;
}

extern "C" int hho_erk_traces(hho_ops* ops, const hho_tableau* tab, const double* d_state, double* d_work,
                              void* stream) {
    std::vector<StagePlan> plan;
    int nb = 0;
    int rc = stage_api_check(ops, tab, d_state, d_work, plan, &nb, "hho_erk_traces");
    if (rc) return rc;
    const dim3 grid((ops->dev.Nf + ops->dev.Ns + 127) / 128, 1);
    if (grid.x == 0) return HHO_OK;
    StageArgsT<double> a;
    memset(&a, 0, sizeof(a));
    a.op = ops->dev;
    a.state_stride = ops->n_state;
    a.trace_stride = ops->trace_doubles;
    a.inp = d_state;
    a.tr_out = d_work + ops->n_state * (1 + nb);
    launch_k<double, MODE_TRACES>(ops->k, a, 1, (cudaStream_t)stream);
    return check_launch("hho_erk_traces");
}

extern "C" int hho_erk_stage(hho_ops* ops, const hho_tableau* tab, int64_t n, int32_t j, double tn, double dt,
                             double* d_state, double* d_work, void* stream) {
    std::vector<StagePlan> plan;
    int nb = 0;
    int rc = stage_api_check(ops, tab, d_state, d_work, plan, &nb, "hho_erk_stage");
    if (rc) return rc;
    if (n < 0 || j < 0 || j >= tab->s || !std::isfinite(tn) || !std::isfinite(dt)) {
        hho_set_error("hho_erk_stage: bad step or stage index");
        return HHO_EINVAL;
    }
    const dim3 grid((ops->dev.Nf + ops->dev.Ns + 127) / 128, 1);
    if (grid.x == 0) return HHO_OK;
    const int64_t S = ops->n_state;
    double* X = d_work;
    double* bufs = d_work + S;
    double* tr[2] = {d_work + S * (1 + nb), d_work + S * (1 + nb) + ops->trace_doubles};
    const int cur = (int)((n * tab->s + j) & 1);
    auto resolve = [&](int code) -> double* {
        if (code == SRC_STATE) return d_state;
        if (code == SRC_X) return X;
        if (code == SRC_ZERO) return nullptr;
        return bufs + S * code;
    };
    StageArgsT<double> a;
    memset(&a, 0, sizeof(a));
    a.op = ops->dev;
    a.state_stride = ops->n_state;
    a.trace_stride = ops->trace_doubles;
    const StagePlan& P = plan[j];
    a.inp = (j == 0) ? d_state : X;
    a.tr_in = tr[cur];
    a.tr_out = tr[cur ^ 1];
    a.n_tgt = P.n_tgt;
    for (int t = 0; t < P.n_tgt; ++t) {
        a.tgt[t].src = resolve(P.t[t].src);
        a.tgt[t].dst = resolve(P.t[t].dst);
        a.tgt[t].coef = P.t[t].a * dt;
    }
    fill_sources<double>(ops, a, tn, j, tab->c[j] * dt, 1);
    launch_k<double, MODE_STAGE>(ops->k, a, 1, (cudaStream_t)stream);
    return check_launch("hho_erk_stage");
}

extern "C" int hho_trace_offsets(const hho_ops* ops, int64_t n, const int64_t* h_cells, const int32_t* h_faces,
                                 int64_t* h_out) {
    if (!ops || n < 0 || (n > 0 && (!h_cells || !h_faces || !h_out))) {
        hho_set_error("hho_trace_offsets: bad arguments");
        return HHO_EINVAL;
    }
    const int f = ops->f;
    for (int64_t i = 0; i < n; ++i) {
        const int64_t c = h_cells[i];
        if (c < 0 || c >= ops->nc) {
            hho_set_error("hho_trace_offsets: cell %lld out of range", (long long)c);
            return HHO_EINVAL;
        }
        const int32_t* ci = &ops->h_cls_int[ops->cell_class_of[c] * CI_STRIDE];
        const int j = h_faces[i];
        if (j < 0 || j >= ci[CI_NF]) {
            hho_set_error("hho_trace_offsets: cell %lld has no local face %d", (long long)c, j);
            return HHO_EINVAL;
        }
        const int64_t slot = ci[CI_SLOT] + (int64_t)j * ci[CI_NPAD] + (ops->cell_pos[c] - ci[CI_START]);
        int64_t* o = h_out + i * 2 * f;
        if (ops->cell_dom[c] == 0) {
            for (int l = 0; l < f; ++l) o[l] = (int64_t)l * ops->dev.SF + slot;
            for (int l = f; l < 2 * f; ++l) o[l] = -1;
        } else {
            const int64_t base = (int64_t)2 * f * ops->dev.SF;
            for (int l = 0; l < 2 * f; ++l) o[l] = base + (int64_t)l * ops->dev.SS + slot;
        }
    }
    return HHO_OK;
}

extern "C" int hho_halo_gather(const double* d_src, const int64_t* d_idx, int64_t n, double* d_dst, void* stream) {
    if (n < 0 || (n > 0 && (!d_src || !d_idx || !d_dst))) {
        hho_set_error("hho_halo_gather: bad arguments");
        return HHO_EINVAL;
    }
    if (n == 0) return HHO_OK;
    const int64_t blocks = std::min<int64_t>((n + 255) / 256, 4096);
    halo_gather_kernel<<<(unsigned)blocks, 256, 0, (cudaStream_t)stream>>>(d_src, d_idx, n, d_dst);
    return check_launch("hho_halo_gather");
}

extern "C" int hho_halo_scatter(const double* d_src, const int64_t* d_idx, int64_t n, double* d_dst, void* stream) {
    if (n < 0 || (n > 0 && (!d_src || !d_idx || !d_dst))) {
        hho_set_error("hho_halo_scatter: bad arguments");
        return HHO_EINVAL;
    }
    if (n == 0) return HHO_OK;
    const int64_t blocks = std::min<int64_t>((n + 255) / 256, 4096);
    halo_scatter_kernel<<<(unsigned)blocks, 256, 0, (cudaStream_t)stream>>>(d_src, d_idx, n, d_dst);
    return check_launch("hho_halo_scatter");
}

// ---- batched shots -----------------------------------------------------------------

static bool batch_args_ok(const hho_ops* ops, int32_t n_shots, int32_t precision, const char* who) {
    if (!ops || n_shots < 1 || n_shots > 65535 ||
        (precision != HHO_F64 && precision != HHO_F32 && precision != HHO_F32X2 && precision != HHO_BF16X3)) {
        hho_set_error("%s: bad arguments (1 <= n_shots <= 65535, precision HHO_F64, HHO_F32, HHO_F32X2 or HHO_BF16X3)",
                      who);
        return false;
    }
    return true;
}

extern "C" int hho_batch_sizes(const hho_ops* ops, const hho_tableau* tab, int32_t n_shots, int32_t precision,
                               int64_t* state_elems, int64_t* work_elems) {
    if (!batch_args_ok(ops, n_shots, precision, "hho_batch_sizes") || !tab) {
        if (!tab) hho_set_error("hho_batch_sizes: null tableau");
        return HHO_EINVAL;
    }
    std::vector<StagePlan> plan;
    int nb = 0;
    if (build_plan(tab, plan, &nb) != HHO_OK) {
        hho_set_error("hho_batch_sizes: unsupported tableau");
        return HHO_EINVAL;
    }
    if (state_elems) *state_elems = ops->n_state * n_shots;
    if (work_elems) *work_elems = (ops->n_state * (1 + nb) + 2 * ops->trace_doubles) * n_shots;
    return HHO_OK;
}

extern "C" int hho_batch_pack(const hho_ops* ops, int32_t n_shots, int32_t precision, const double* d_canonical,
                              void* d_state, void* stream) {
    if (!batch_args_ok(ops, n_shots, precision, "hho_batch_pack") || !d_canonical || !d_state) {
        if (ops) hho_set_error("hho_batch_pack: bad arguments");
        return HHO_EINVAL;
    }
    if (ops->dev.Nf + ops->dev.Ns == 0) return HHO_OK;
    cudaStream_t st = (cudaStream_t)stream;
    if (precision == HHO_F64) launch_pack<double>(ops, n_shots, d_canonical, d_state, st);
    else if (precision == HHO_F32X2) launch_pack<f2x>(ops, n_shots, d_canonical, d_state, st);
    else launch_pack<float>(ops, n_shots, d_canonical, d_state, st);
    return check_launch("hho_batch_pack");
}

extern "C" int hho_batch_unpack(const hho_ops* ops, int32_t n_shots, int32_t precision, const void* d_state,
                                double* d_canonical, void* stream) {
    if (!batch_args_ok(ops, n_shots, precision, "hho_batch_unpack") || !d_canonical || !d_state) {
        if (ops) hho_set_error("hho_batch_unpack: bad arguments");
        return HHO_EINVAL;
    }
    if (ops->dev.Nf + ops->dev.Ns == 0) return HHO_OK;
    cudaStream_t st = (cudaStream_t)stream;
    if (precision == HHO_F64) launch_unpack<double>(ops, n_shots, d_state, d_canonical, st);
    else if (precision == HHO_F32X2) launch_unpack<f2x>(ops, n_shots, d_state, d_canonical, st);
    else launch_unpack<float>(ops, n_shots, d_state, d_canonical, st);
    return check_launch("hho_batch_unpack");
}

extern "C" int hho_batch_erk_step(hho_ops* ops, const hho_tableau* tab, int32_t n_shots, int32_t precision, double t0,
                                  double dt, int64_t nsteps, void* d_state, void* d_work, void* d_seismogram,
                                  void* stream) {
    if (!batch_args_ok(ops, n_shots, precision, "hho_batch_erk_step")) return HHO_EINVAL;
    if (ops->n_shot_src > 0 && ops->n_shot_src < n_shots) {
        hho_set_error("hho_batch_erk_step: %d shot sources set for %d shots", ops->n_shot_src, n_shots);
        return HHO_EINVAL;
    }
    if (precision == HHO_F64)
        return erk_run<double>(ops, tab, t0, dt, nsteps, n_shots, (double*)d_state, (double*)d_work, d_seismogram,
                               stream, "hho_batch_erk_step");
    if (precision == HHO_F32X2)
        return erk_run<f2x>(ops, tab, t0, dt, nsteps, n_shots, (f2x*)d_state, (f2x*)d_work, d_seismogram, stream,
                            "hho_batch_erk_step");
    ops->tc_on = precision == HHO_BF16X3;
    const int rc = erk_run<float>(ops, tab, t0, dt, nsteps, n_shots, (float*)d_state, (float*)d_work, d_seismogram,
                                  stream, "hho_batch_erk_step");
    ops->tc_on = false;
    return rc;
}

extern "C" int hho_tc_error(hho_ops* ops, int32_t* h_flag) {
    if (!ops || !h_flag) {
        hho_set_error("hho_tc_error: null pointer");
        return HHO_EINVAL;
    }
    int32_t v = 0;
    if (cudaMemcpy(&v, ops->d_tc_err, sizeof(v), cudaMemcpyDeviceToHost) != cudaSuccess ||
        cudaMemset(ops->d_tc_err, 0, sizeof(v)) != cudaSuccess) {
        hho_set_error("hho_tc_error: copy failed");
        return HHO_ECUDA;
    }
    *h_flag = v;
    return HHO_OK;
}

extern "C" int hho_profile_enable(hho_ops* ops, int32_t on) {
    if (!ops) {
        hho_set_error("hho_profile_enable: null ops");
        return HHO_EINVAL;
    }
    if (on && ops->prof_events.empty()) {
        for (int i = 0; i < 8192; ++i) {
            cudaEvent_t e;
            if (cudaEventCreate(&e) != cudaSuccess) {
                hho_set_error("hho_profile_enable: cudaEventCreate failed");
                return HHO_ECUDA;
            }
            ops->prof_events.push_back((void*)e);
        }
    }
    ops->prof_on = on != 0;
    ops->prof_n = 0;
    return HHO_OK;
}

extern "C" int hho_profile_read(hho_ops* ops, double* ms, int64_t* n) {
    if (!ops || !ms || !n) {
        hho_set_error("hho_profile_read: null pointer");
        return HHO_EINVAL;
    }
    double tot = 0.0;
    for (int i = 0; i < ops->prof_n; ++i) {
        float t = 0.0f;
        if (cudaEventSynchronize((cudaEvent_t)ops->prof_events[2 * i + 1]) != cudaSuccess ||
            cudaEventElapsedTime(&t, (cudaEvent_t)ops->prof_events[2 * i], (cudaEvent_t)ops->prof_events[2 * i + 1]) !=
                cudaSuccess) {
            hho_set_error("hho_profile_read: event query failed");
            return HHO_ECUDA;
        }
        tot += t;
    }
    *ms = tot;
    *n = ops->prof_n;
    ops->prof_n = 0;
    return HHO_OK;
}

// FP64 lane-ops of one stage thread, mirroring fluid_cell / solid_cell.
extern "C" int hho_stage_cost(const hho_ops* ops, const hho_tableau* tab, int64_t* fp64_ops, int64_t* bytes_min,
                              int64_t* bytes_kernel) {
    if (!ops || !tab) {
        hho_set_error("hho_stage_cost: null pointer");
        return HHO_EINVAL;
    }
    std::vector<StagePlan> plan;
    int nbuf = 0;
    if (build_plan(tab, plan, &nbuf) != HHO_OK) {
        hho_set_error("hho_stage_cost: unsupported tableau");
        return HHO_EINVAL;
    }
    const int K = ops->k, n = ops->n, f = ops->f;
    const int64_t dsm = (int64_t)K * (K - 1) / 2, dvalid = (int64_t)K * (K + 1) / 2;
    // entries of the rectangle parity patterns (the same count on every face),
    // of an axis-aligned face's trace, and of a general face; a square's trace
    // takes K(K+1)/2 multiply-adds (trace_square)
    int64_t rect_tr = 0, rect_lift = 0, square_lift = 0, axis_tr = 0;
    const int64_t square_tr = (int64_t)K * (K + 1) / 2, full = (int64_t)f * n;
    for (int i = 0; i < n; ++i) {
        const int e = ea(i);
        for (int l = 0; l < f; ++l) {
            rect_tr += (e == l);
            rect_lift += (((e + l) % 2) == 0);
            square_lift += (((e + l) % 2) == 0) && e - l != 2;
            axis_tr += e >= l;
        }
    }
    int64_t ops_total = 0, bytes_k = 0, dofs = 0;
    for (int cl = 0; cl < ops->n_classes; ++cl) {
        const int32_t* ci = &ops->h_cls_int[cl * CI_STRIDE];
        const int dom = ci[CI_DOMAIN], nF = ci[CI_NF], count = ci[CI_COUNT];
        const int npad = ci[CI_NPAD], sbase = ci[CI_SLOT];
        const bool rect = ci[CI_KIND] != KIND_GENERIC;
        const int nv = (dom ? 5 : 3) * n, pc = dom ? 2 : 1;   // state values, primal components
        const int64_t nnzT = ci[CI_KIND] == KIND_SQUARE ? square_tr : rect_tr;
        const int64_t nnzL = ci[CI_KIND] == KIND_SQUARE ? square_lift : rect_lift;
        const uint32_t axis = (uint32_t)(ci[CI_HOR] | ci[CI_VER]);
        dofs += (int64_t)count * nv;
        for (int r = 0; r < count; ++r) {
            int64_t rate = dom ? 5 * dsm + 3 * dvalid + 2 * n : 3 * dsm + dvalid;   // derivatives (+ stress mix)
            if (rect) rate += pc * n;                                               // tau, once per cell
            int64_t traces = 0, bytes_faces = 0;
            for (int j = 0; j < nF; ++j) {
                const int32_t nb = (dom ? ops->h_nb_s : ops->h_nb_f)[sbase + j * npad + r];
                const bool bnd = nb == NB_BOUNDARY, ifc = nb < NB_BOUNDARY;
                const bool ax = j < 32 && ((axis >> j) & 1);
                rate += bnd ? 0 : (ifc && !dom ? 3 * f : pc * f);                  // jump
                // lift and the normal / tau combinations; rectangles lift each mirror pair of
                // faces at once (lift_pair: 2f + 2 nnz(L) per pair and component)
                rate += rect ? pc * (nnzL + f) : pc * full + (dom ? (ax ? 4 * n : 6 * n) : (ax ? 2 * n : 3 * n));
                traces += rect ? 2 * pc * nnzT : ax ? 2 * pc * axis_tr : dom ? 5 * full + 4 * f : 3 * full + 2 * f;
                traces += dom ? 2 * f + (ifc ? 4 * f : 2 * f) : 2 * f;
                bytes_faces += 8 * (int64_t)pc * f * (1 + (bnd ? 0 : 1) + 2) + 4 + 8;
            }
            for (int j = 0; j < tab->s; ++j) {
                const StagePlan& P = plan[j];
                ops_total += rate + (int64_t)P.n_tgt * (nv + 3) + traces;
                int64_t passes = 1;   // stage input
                for (int t = 0; t < P.n_tgt; ++t) passes += 1 + (P.t[t].src != SRC_ZERO ? 1 : 0);
                bytes_k += 8 * passes * nv + bytes_faces + 8 * (dom ? SCS : SCF);
            }
        }
    }
    int64_t passes_min = 0;
    for (int j = 0; j < tab->s; ++j) {
        const StagePlan& P = plan[j];
        std::vector<int> reads, writes;
        reads.push_back(j == 0 ? SRC_STATE : SRC_X);
        for (int t = 0; t < P.n_tgt; ++t) {
            if (P.t[t].src != SRC_ZERO) reads.push_back(P.t[t].src);
            writes.push_back(P.t[t].dst);
        }
        std::sort(reads.begin(), reads.end());
        reads.erase(std::unique(reads.begin(), reads.end()), reads.end());
        passes_min += (int64_t)reads.size() + (int64_t)writes.size();
    }
    if (fp64_ops) *fp64_ops = ops_total;
    if (bytes_min) *bytes_min = 8 * passes_min * dofs;
    if (bytes_kernel) *bytes_kernel = bytes_k;
    return HHO_OK;
}

template <class T>
static int apply_t(hho_ops* ops, double t, const T* d_state, T* d_rate, T* d_traces, cudaStream_t st) {
    const dim3 grid((ops->dev.Nf + ops->dev.Ns + 127) / 128, 1);
    if (grid.x == 0) return HHO_OK;
    StageArgsT<T> a;
    memset(&a, 0, sizeof(a));
    a.op = ops->dev;
    a.state_stride = ops->n_state;
    a.trace_stride = ops->trace_doubles;
    a.inp = d_state;
    a.tr_out = d_traces;
    launch_k<T, MODE_TRACES>(ops->k, a, 1, st);
    int rc = check_launch("hho_apply (trace kernel)");
    if (rc) return rc;
    a.tr_in = d_traces;
    a.tr_out = nullptr;
    a.n_tgt = 1;
    a.tgt[0].src = nullptr;
    a.tgt[0].dst = d_rate;
    a.tgt[0].coef = T(1.0);
    fill_sources<T>(ops, a, t, -1, 0.0, 1);
    launch_k<T, MODE_APPLY>(ops->k, a, 1, st);
    return check_launch("hho_apply (stage kernel)");
}

extern "C" int hho_apply(hho_ops* ops, double t, const double* d_state, double* d_rate, double* d_work,
                         void* stream) {
    if (!ops || !d_state || !d_rate || !d_work) {
        hho_set_error("hho_apply: null pointer");
        return HHO_EINVAL;
    }
    if (ops->src_sampled) {
        hho_set_error("hho_apply: sampled source time functions are indexed by ERK stages, not by time");
        return HHO_EINVAL;
    }
    cudaStream_t st = (cudaStream_t)stream;
    if (ops->arith != HHO_F32X2) return apply_t<double>(ops, t, d_state, d_rate, d_work, st);
    // double-float: [traces][state pairs][rate pairs] inside the work buffer
    if (ops->n_state == 0) return HHO_OK;
    f2x* tr = (f2x*)d_work;
    f2x* ux = (f2x*)(d_work + ops->trace_doubles);
    f2x* rx = ux + ops->n_state;
    to_pairs_kernel<<<pairs_grid(ops->n_state), 256, 0, st>>>(d_state, ux, ops->n_state);
    int rc = check_launch("hho_apply");
    if (rc) return rc;
    rc = apply_t<f2x>(ops, t, ux, rx, tr, st);
    if (rc) return rc;
    from_pairs_kernel<<<pairs_grid(ops->n_state), 256, 0, st>>>(rx, d_rate, ops->n_state);
    return check_launch("hho_apply");
}

extern "C" int hho_state_pack(const hho_ops* ops, const double* d_canonical, double* d_state, void* stream) {
    if (!ops || !d_canonical || !d_state) {
        hho_set_error("hho_state_pack: null pointer");
        return HHO_EINVAL;
    }
    return hho_batch_pack(ops, 1, HHO_F64, d_canonical, d_state, stream);
}

extern "C" int hho_state_unpack(const hho_ops* ops, const double* d_state, double* d_canonical, void* stream) {
    if (!ops || !d_canonical || !d_state) {
        hho_set_error("hho_state_unpack: null pointer");
        return HHO_EINVAL;
    }
    return hho_batch_unpack(ops, 1, HHO_F64, d_state, d_canonical, stream);
}

extern "C" int hho_energy(hho_ops* ops, const double* d_state, double* d_work, double* h_energy, void* stream) {
    if (!ops || !d_state || !d_work || !h_energy) {
        hho_set_error("hho_energy: null pointer");
        return HHO_EINVAL;
    }
    cudaStream_t st = (cudaStream_t)stream;
    const int tot = ops->dev.Nf + ops->dev.Ns;
    const int nblk = (tot + 255) / 256;
    double* partial = d_work;
    double* result = d_work + nblk;
    if (nblk > 0) {
        if (ops->k == 1) energy_kernel<1><<<nblk, 256, 0, st>>>(ops->dev, d_state, ops->d_mass_f, ops->d_mass_s, partial);
        else if (ops->k == 2) energy_kernel<2><<<nblk, 256, 0, st>>>(ops->dev, d_state, ops->d_mass_f, ops->d_mass_s, partial);
        else energy_kernel<3><<<nblk, 256, 0, st>>>(ops->dev, d_state, ops->d_mass_f, ops->d_mass_s, partial);
    }
    sum_kernel<<<1, 256, 0, st>>>(partial, nblk, result);
    int rc = check_launch("hho_energy");
    if (rc) return rc;
    double e = 0.0;
    if (cudaMemcpyAsync(&e, result, sizeof(double), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess) {
        hho_set_error("hho_energy: copy failed");
        return HHO_ECUDA;
    }
    *h_energy = e;
    if (!std::isfinite(e)) {
        hho_set_error("hho_energy: non-finite energy");
        return HHO_EUNSTABLE;
    }
    return HHO_OK;
}

extern "C" int hho_record(hho_ops* ops, const double* d_state, double* d_out, void* stream) {
    if (!ops || !d_state || (ops->n_rec > 0 && !d_out)) {
        hho_set_error("hho_record: null pointer");
        return HHO_EINVAL;
    }
    if (ops->n_rec == 0) return HHO_OK;
    launch_record<double, double>(ops, 1, d_state, d_out, nullptr, (cudaStream_t)stream);
    return check_launch("hho_record");
}

// The call on buffers that are ready; returns with work queued on st where it fails.
static int erk_run_host(hho_ops* ops, const hho_tableau* tab, double t0, double dt, int64_t nsteps, double* h_canonical,
                        bool made, void* stream) {
    cudaStream_t st = (cudaStream_t)stream;
    // A pinned host buffer mapped into the device's address space is read
    // and written by the pack kernels directly (over NVLink-C2C on GB300) or,
    // on large meshes, copied in overlapping pieces; any other host memory goes
    // through one staging copy.
    cudaPointerAttributes pa;
    if (cudaPointerGetAttributes(&pa, h_canonical) == cudaSuccess && pa.type == cudaMemoryTypeHost &&
        pa.devicePointer) {
        const int rc = erk_run_mapped(ops, tab, t0, dt, nsteps, h_canonical, (double*)pa.devicePointer, made, st);
        if (rc) return rc;
        if (cudaStreamSynchronize(st) != cudaSuccess) {
            hho_set_error("hho_erk_run_host: %s", cudaGetErrorString(cudaGetLastError()));
            return HHO_ECUDA;
        }
        return HHO_OK;
    }
    cudaGetLastError();   // an unregistered pointer leaves an error on some drivers
    if (cudaMemcpyAsync(ops->d_host_canon, h_canonical, sizeof(double) * ops->n_canonical, cudaMemcpyHostToDevice,
                        st) != cudaSuccess) {
        hho_set_error("hho_erk_run_host: host-to-device copy failed");
        return HHO_ECUDA;
    }
    int rc = hho_state_pack(ops, ops->d_host_canon, ops->d_host_state, stream);
    if (rc) return rc;
    rc = hho_erk_step(ops, tab, t0, dt, nsteps, ops->d_host_state, ops->d_host_work, stream);
    if (rc) return rc;
    rc = hho_state_unpack(ops, ops->d_host_state, ops->d_host_canon, stream);
    if (rc) return rc;
    if (cudaMemcpyAsync(h_canonical, ops->d_host_canon, sizeof(double) * ops->n_canonical, cudaMemcpyDeviceToHost,
                        st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess) {
        hho_set_error("hho_erk_run_host: device-to-host copy failed");
        return HHO_ECUDA;
    }
    return HHO_OK;
}

extern "C" int hho_erk_run_host(hho_ops* ops, const hho_tableau* tab, double t0, double dt, int64_t nsteps,
                                double* h_canonical, void* stream) {
    if (!ops || !tab || !h_canonical) {
        hho_set_error("hho_erk_run_host: null pointer");
        return HHO_EINVAL;
    }
    int64_t wsz = 0;
    int rc = hho_work_size(ops, tab, &wsz);
    if (rc) return rc;
    cudaStream_t st = (cudaStream_t)stream;
    bool made = false;
    rc = grow_host_buffers(
        ops, wsz,
        [](size_t n) {
            double* p = nullptr;
            if (cudaMalloc((void**)&p, sizeof(double) * std::max<size_t>(n, 1)) == cudaSuccess) return p;
            cudaGetLastError();   // reported here; not for the next launch to find
            return (double*)nullptr;
        },
        [](double* p) { cudaFree(p); },
        [&](double* p, size_t n) { return cudaMemsetAsync(p, 0, sizeof(double) * n, st) == cudaSuccess; }, &made);
    if (rc == HHO_ENOMEM) hho_set_error("hho_erk_run_host: device allocation failed");
    if (rc == HHO_ECUDA) hho_set_error("hho_erk_run_host: device memset failed");
    if (rc) return rc;
    rc = erk_run_host(ops, tab, t0, dt, nsteps, h_canonical, made, stream);
    if (rc) cudaStreamSynchronize(st);   // the next call may come on another stream; the buffers are free for it
    return rc;
}

extern "C" int hho_cfl_bracket(hho_ops* ops, const hho_tableau* tab, const double* d_state0, double T_f,
                               int64_t N0, double eps, double delta, int64_t max_trials, double* d_state,
                               double* d_work, int64_t* n_stable, int64_t* n_unstable, void* stream) {
    if (!ops || !tab || !d_state0 || !d_state || !d_work || !n_stable || !n_unstable || !(T_f > 0.0) || N0 < 1 ||
        !(eps > 0.0) || !(delta > 0.0) || max_trials < 1) {
        hho_set_error("hho_cfl_bracket: bad arguments");
        return HHO_EINVAL;
    }
    cudaStream_t st = (cudaStream_t)stream;
    const int saved_src = ops->n_src, saved_shot = ops->n_shot_src;
    ops->n_src = 0;        // Algorithm 1 runs without sources
    ops->n_shot_src = 0;
    int rc = HHO_OK;
    int64_t N = N0, last = -1, first_unstable = -1;
    for (int64_t trial = 0; trial < max_trials && N >= 1 && rc == HHO_OK; ++trial) {
        const double dt = T_f / (double)N;
        if (cudaMemcpyAsync(d_state, d_state0, sizeof(double) * ops->n_state, cudaMemcpyDeviceToDevice, st) !=
            cudaSuccess) {
            hho_set_error("hho_cfl_bracket: copy failed");
            rc = HHO_ECUDA;
            break;
        }
        double E0 = 0.0;
        rc = hho_energy(ops, d_state, d_work, &E0, stream);
        if (rc) break;
        if (!(E0 > 0.0) || !std::isfinite(E0)) {   // the relative increases below divide by E0
            hho_set_error("hho_cfl_bracket: the initial energy must be positive and finite (got %g)", E0);
            rc = HHO_EINVAL;
            break;
        }
        double Eprev = E0;
        bool stable = true;
        for (int64_t n = 0; n < N; ++n) {
            rc = hho_erk_step(ops, tab, (double)n * dt, dt, 1, d_state, d_work, stream);
            if (rc) break;
            double E = 0.0;
            rc = hho_energy(ops, d_state, d_work, &E, stream);
            if (rc == HHO_EUNSTABLE) {   // non-finite energy: the trial is unstable
                rc = HHO_OK;
                stable = false;
                break;
            }
            if (rc) break;
            if ((E - E0) / E0 > eps || (E - Eprev) / Eprev > eps) {
                stable = false;
                break;
            }
            Eprev = E;
        }
        if (rc) break;
        if (!stable) {
            first_unstable = N;
            break;
        }
        last = N;
        int64_t dec = (int64_t)std::floor(delta * (double)N);
        N -= dec < 1 ? 1 : dec;
    }
    ops->n_src = saved_src;
    ops->n_shot_src = saved_shot;
    *n_stable = last;
    *n_unstable = first_unstable;
    return rc;
}

// ---- energy without allocation ------------------------------------------------------
// Block partial sums of hho_energy_static live in this fixed array instead of
// a caller buffer.  Host code must not take its address directly (the host
// symbol is only a stand-in for the device variable); the device address is
// looked up with cudaGetSymbolAddress, with the device current, on every
// call.  The lookup allocates nothing and is cheap, and an address kept from
// an earlier call would go stale after a device reset.
namespace {
constexpr int kEnergyStaticMaxBlocks = (int)(HHO_ENERGY_STATIC_MAX_CELLS / 256);
static __device__ __align__(256) double g_energy_partials[kEnergyStaticMaxBlocks];

// Device address of g_energy_partials on the current device.
int energy_scratch(double** out) {
    void* p = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&p, g_energy_partials);
    if (e != cudaSuccess || !p) {
        hho_set_error("hho_energy_static: cudaGetSymbolAddress failed: %s", cudaGetErrorString(e));
        return HHO_ECUDA;
    }
    *out = (double*)p;
    return HHO_OK;
}
}  // namespace

extern "C" int hho_energy_static(hho_ops* ops, const double* d_state, double* d_energy, void* stream) {
    if (!ops || !d_state || !d_energy) {
        hho_set_error("hho_energy_static: null pointer");
        return HHO_EINVAL;
    }
    const int64_t tot = (int64_t)ops->dev.Nf + ops->dev.Ns;
    if (tot > HHO_ENERGY_STATIC_MAX_CELLS) {
        hho_set_error("hho_energy_static: %lld padded cell slots exceed the fixed scratch limit of %lld; use hho_energy",
                      (long long)tot, (long long)HHO_ENERGY_STATIC_MAX_CELLS);
        return HHO_EINVAL;
    }
    double* partial = nullptr;
    int rc = energy_scratch(&partial);
    if (rc) return rc;
    cudaStream_t st = (cudaStream_t)stream;
    const int nblk = (int)((tot + 255) / 256);
    // energy_kernel writes every partial[0..nblk) before sum_kernel reads it,
    // so the array's previous contents never matter.
    if (nblk > 0) {
        if (ops->k == 1) energy_kernel<1><<<nblk, 256, 0, st>>>(ops->dev, d_state, ops->d_mass_f, ops->d_mass_s, partial);
        else if (ops->k == 2) energy_kernel<2><<<nblk, 256, 0, st>>>(ops->dev, d_state, ops->d_mass_f, ops->d_mass_s, partial);
        else energy_kernel<3><<<nblk, 256, 0, st>>>(ops->dev, d_state, ops->d_mass_f, ops->d_mass_s, partial);
    }
    sum_kernel<<<1, 256, 0, st>>>(partial, nblk, d_energy);
    return check_launch("hho_energy_static");
}

// ---- launchers for the adjoint driver (adjoint.cu) -----------------------------------
void launch_stage_f64(const hho_ops* ops, int mode, StageArgsT<double>& a, int n_shots, double tn, int j, double cdt,
                      bool sources, void* stream) {
    const dim3 grid((ops->dev.Nf + ops->dev.Ns + 127) / 128, n_shots);
    if (grid.x == 0) return;
    a.state_stride = ops->n_state;
    a.trace_stride = ops->trace_doubles;
    if (sources) {
        fill_sources<double>(ops, a, tn, j, cdt, n_shots);
    } else {
        a.n_src = 0;
        a.shot_src_q = nullptr;
        a.shot_src_dom = nullptr;
        a.shot_src_g = nullptr;
    }
    cudaStream_t st = (cudaStream_t)stream;
    switch (mode) {
        case MODE_TRACES: launch_k<double, MODE_TRACES>(ops->k, a, n_shots, st); break;
        case MODE_STAGE: launch_k<double, MODE_STAGE>(ops->k, a, n_shots, st); break;
        case MODE_APPLY: launch_k<double, MODE_APPLY>(ops->k, a, n_shots, st); break;
        default: break;
    }
}

void launch_stage_f32(const hho_ops* ops, int mode, StageArgsT<float>& a, int n_shots, double tn, int j, double cdt,
                      bool sources, void* stream) {
    const dim3 grid((ops->dev.Nf + ops->dev.Ns + 127) / 128, n_shots);
    if (grid.x == 0) return;
    a.state_stride = ops->n_state;
    a.trace_stride = ops->trace_doubles;
    if (sources) {
        fill_sources<float>(ops, a, tn, j, cdt, n_shots);
    } else {
        a.n_src = 0;
        a.shot_src_q = nullptr;
        a.shot_src_dom = nullptr;
        a.shot_src_g = nullptr;
    }
    cudaStream_t st = (cudaStream_t)stream;
    switch (mode) {
        case MODE_TRACES: launch_k<float, MODE_TRACES>(ops->k, a, n_shots, st); break;
        case MODE_STAGE: launch_k<float, MODE_STAGE>(ops->k, a, n_shots, st); break;
        case MODE_APPLY: launch_k<float, MODE_APPLY>(ops->k, a, n_shots, st); break;
        default: break;
    }
}

template <class T>
static void launch_grad_t(const hho_ops* ops, StageArgsT<T>& a, const GradArgsT<T>& g, double tn, int j, double cdt,
                          void* stream) {
    const unsigned grid = (unsigned)((ops->dev.Nf + ops->dev.Ns + 127) / 128);
    if (grid == 0) return;
    a.state_stride = ops->n_state;
    a.trace_stride = ops->trace_doubles;
    fill_sources<T>(ops, a, tn, j, cdt, 1);
    cudaStream_t st = (cudaStream_t)stream;
    if (ops->k == 1) hho_stage::launch_grad<T, 1>(a, g, st);
    else if (ops->k == 2) hho_stage::launch_grad<T, 2>(a, g, st);
    else hho_stage::launch_grad<T, 3>(a, g, st);
}
void launch_grad_f64(const hho_ops* ops, StageArgsT<double>& a, const GradArgsT<double>& g, double tn, int j, double cdt,
                     void* stream) {
    launch_grad_t<double>(ops, a, g, tn, j, cdt, stream);
}
void launch_grad_f32(const hho_ops* ops, StageArgsT<float>& a, const GradArgsT<float>& g, double tn, int j, double cdt,
                     void* stream) {
    launch_grad_t<float>(ops, a, g, tn, j, cdt, stream);
}

int erk_steps_f32(hho_ops* ops, const hho_tableau* tab, double t0, double dt, int64_t nsteps, float* d_state,
                  float* d_work, void* stream) {
    return erk_run<float>(ops, tab, t0, dt, nsteps, 1, d_state, d_work, nullptr, stream, "hho_adjoint_vjp_f32");
}

void launch_record_f64(const hho_ops* ops, const double* state, double* out, void* stream) {
    if (ops->n_rec == 0) return;
    launch_record<double, double>(ops, 1, state, out, nullptr, (cudaStream_t)stream);
}

int check_cuda(const char* what) { return check_launch(what); }
