// The block-Jacobi product of the SDIRK solver's GMRES, y = s P^-1 x, with the
// face traces of y published in the same pass (the first half of the operator
// that GMRES applies next).
//
// A block of 8 warps takes 32 cells of one class: x in shared memory (column =
// lane), two rows of the inverse blocks per warp at a time.  Bound by the FP64
// pipe (24 multiply-adds a value at k = 2: 37 us for 786,432 values at 19
// cycles an instruction) and not far from memory (157 MB of blocks, 24 us); two
// rows share each entry of x, which the pipe takes in 16 cycles.  One thread a
// value read each x entry 30 times from L2 and took 60 us, and the traces
// another 10.7 us in a launch of their own.
#include "stage_kernels.cuh"

namespace {

constexpr int BJ_W = 8;

template <int K, bool SOLID>
__device__ __forceinline__ void bj_cells(const DevOps& op, const double* __restrict__ bj, const double* __restrict__ x,
                                         double s, double* y, int accumulate, double* tr, int gw, double* smem) {
    constexpr int n = Dims<K>::n, FS = Dims<K>::FS, NV = SOLID ? 5 * n : 3 * n;
    const int lane = threadIdx.x & 31;
    const int w = ((threadIdx.x >> 5) + blockIdx.x * 3) % BJ_W;   // as the team form: even over the sub-partitions
    const int N = SOLID ? op.Ns : op.Nf;
    const int q = (gw - (SOLID ? op.n_warps_f : 0)) * 32 + lane;
    const size_t off = SOLID ? (size_t)3 * n * op.Nf : 0;
    double* X = smem + lane;
    double* Y = X + 32 * 5 * n;
    double* cd = smem + 2 * 32 * 5 * n;
    const double* xq = x + off + q;
    for (int i = w; i < NV; i += BJ_W) X[32 * i] = s * xq[(size_t)i * N];
    const int* ci = op.cls_int + __ldg(op.warp_class + gw) * CI_STRIDE;
    const int nF = __ldg(ci + CI_NF);
    if (tr) {
        const float4* src = reinterpret_cast<const float4*>(op.cls_dbl + __ldg(ci + CI_DOFF) + Dims<K>::M0P);
        float4* dst = reinterpret_cast<float4*>(cd);
        for (int e = threadIdx.x; e < nF * FS / 2; e += 32 * BJ_W) dst[e] = __ldg(src + e);
    }
    __syncthreads();
    double* yq = y + off + q;
    if (!bj) {   // no preconditioner: y = s x
        for (int i = w; i < NV; i += BJ_W) {
            const double v = X[32 * i];
            yq[(size_t)i * N] = v;
            Y[32 * i] = v;
        }
    } else {
        const double* b = bj + (SOLID ? (size_t)9 * n * n * op.Nf : 0) + q;
        for (int p = w; p < (NV + 1) / 2; p += BJ_W) {
            const int r0 = 2 * p, r1 = min(2 * p + 1, NV - 1);
            const double* b0 = b + (size_t)r0 * NV * N;
            const double* b1 = b + (size_t)r1 * NV * N;
            double s0 = 0.0, s1 = 0.0;
#pragma unroll(NV % 10 == 0 ? 10 : 9)
            for (int c = 0; c < NV; ++c) {
                const double xv = X[32 * c];
                s0 = fma(b0[(size_t)c * N], xv, s0);
                s1 = fma(b1[(size_t)c * N], xv, s1);
            }
            Y[32 * r0] = s0;
            Y[32 * r1] = s1;
            yq[(size_t)r0 * N] = accumulate ? yq[(size_t)r0 * N] + s0 : s0;
            if (r1 != r0) yq[(size_t)r1 * N] = accumulate ? yq[(size_t)r1 * N] + s1 : s1;
        }
    }
    if (!tr) return;
    __syncthreads();
    TeamFaces<double> F;
    F.nF = nF;
    F.npad = __ldg(ci + CI_NPAD);
    F.sbase = __ldg(ci + CI_SLOT);
    F.kind = __ldg(ci + CI_KIND);
    F.lq = q - __ldg(ci + CI_START);
    F.hor = (uint32_t)__ldg(ci + CI_HOR);
    F.other = (nF >= 32 ? 0xffffffffu : (1u << nF) - 1u) & ~(F.hor | (uint32_t)__ldg(ci + CI_VER));
    F.cd = cd;
    F.tau = __ldg((SOLID ? op.scal_s : op.scal_f) + (size_t)(SOLID ? SS_TAU : SF_TAU) * N + q);
    F.real = F.lq < __ldg(ci + CI_COUNT);
    team_traces<double, K, BJ_W, SOLID>(op, F, Y, tr, w);
}

template <int K>
__global__ void __launch_bounds__(32 * BJ_W, 4)
    bj_kernel(const DevOps op, const double* __restrict__ bj, const double* __restrict__ x,
              const double* __restrict__ scale, double* y, int accumulate, double* tr) {
    extern __shared__ __align__(16) unsigned char bj_smem[];
    double* smem = reinterpret_cast<double*>(bj_smem);
    const double s = scale ? *scale : 1.0;
    const int gw = gridDim.x - 1 - blockIdx.x;   // solid cells, the longer ones, first
    if (gw < op.n_warps_f) bj_cells<K, false>(op, bj, x, s, y, accumulate, tr, gw, smem);
    else bj_cells<K, true>(op, bj, x, s, y, accumulate, tr, gw, smem);
}

template <int K>
struct BjTag {};

template <int K>
void launch(const DevOps& op, const double* bj, const double* x, const double* scale, double* y, int accumulate,
            double* tr, cudaStream_t st) {
    const size_t smem = sizeof(double) * ((size_t)2 * 32 * 5 * Dims<K>::n + (tr ? op.max_nf * Dims<K>::FS : 0));
    stage_smem_attributes<BjTag<K>>(bj_kernel<K>, smem, true);
    bj_kernel<K><<<op.n_warps_f + op.n_warps_s, 32 * BJ_W, smem, st>>>(op, bj, x, scale, y, accumulate, tr);
}

}  // namespace

void launch_bj(const hho_ops* ops, const double* bj, const double* x, const double* scale, double* y, bool accumulate,
               double* tr, void* stream) {
    if (ops->dev.n_warps_f + ops->dev.n_warps_s == 0) return;
    cudaStream_t st = (cudaStream_t)stream;
    if (ops->k == 1) launch<1>(ops->dev, bj, x, scale, y, accumulate, tr, st);
    else if (ops->k == 2) launch<2>(ops->dev, bj, x, scale, y, accumulate, tr, st);
    else launch<3>(ops->dev, bj, x, scale, y, accumulate, tr, st);
}
