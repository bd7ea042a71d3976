// Discrete adjoint of the ERK time stepping (vector-Jacobian product of the
// receiver traces with respect to the materials and the source wavelet).
//
// Forward: k_i = A Y_i + w(t_i) g (A = -M^-1 K_cond, Eq. ex_solve), Y_i the
// stage values of Eq. ERK_compact, U^n = U^{n-1} + dt sum_i b_i k_i, and the
// traces d^n = R U^n (hho_record after every step).
// Backward, for a cotangent G^n = dL/dd^n: lambda^n += R^T G^n, then for the
// stages in reverse order
//     mu_i = dt (b_i lambda^n + sum_{l>i} a_li nu_l),   nu_i = A^T mu_i,
//     lambda^{n-1} = lambda^n + sum_i nu_i,
//     dL/dtheta += mu_i^T dk_i/dtheta,   dL/dw(t_i) += mu_i^T g.
// A^T is applied without a transposed kernel: the block structure of the
// paper's system (Sec. 3.3) gives A^T = S M A' M^-1 S, where S flips the
// signs of the dual fields (m, s) and A' is the same operator with the sign
// of the interface coupling block reversed.  The sweep runs on
// lambda^ = S M^-1 lambda, for which the mass matrices cancel:
//     x_i = S M^-1 mu_i = dt (b_i lambda^ + sum_{l>i} a_li A' x_l),
//     lambda^ += sum_i A' x_i,   at a time node lambda^ += S M^-1 R^T G.
// With x_i = dt sigma_i z_i, sigma_i = b_i, that is an explicit step
//     z_i = lambda^ + dt sum_{l>i} (b_l a_li / b_i) A' z_l,
//     lambda^ += dt sum_i b_i A' z_i
// (the adjoint Runge-Kutta scheme), so every backward stage is ONE stage
// kernel launch of the forward path, targets and published traces included;
// weights b_i that vanish or are small take sigma_i = 1 (adjoint_plan).
// Measured on 256 x 256 squares, k = 2: the mass kernels on both sides, the
// separate traces and the application took 161 us a stage, the stage kernel
// takes 33.
//
// Parameters.  (1) The per-cell factors of the inverse mass, theta =
// (1/(rho h), kappa/h) in fluid cells and ((lambda+2mu)/h, lambda/(lambda+2mu),
// mu/h, 1/(rho h)) in solid cells; dk/dtheta is the raw rate (MODE_GRAD).
// (2) The stabilisation weights tau (Sec. 3.3: tau^f = eta_f/(rho c_P),
// tau^s = eta_s rho c^s).  The full stiffness is affine in tau: dK/dtau_c is
// cell c's least-squares stabilisation (Eq. stab) without its weight, so
//     d(eta^T K_cond Y)/dtau_c = sum_{F of c} (eta_c - eta_F, Y_c - Y_F)_F
// on the primal unknowns, with Y_F the face values of the stage value Y and
// eta_F = -K_F^-T K_TF^T eta the adjoint face values of eta = M^-1 mu.  By the
// same block structure eta_F are the face values of the coupling-reversed
// operator A' applied to x = S eta, which the backward stage computes anyway:
// tau_grad (stage_kernels.cuh) takes the products of both jumps from the two trace
// buffers.  The interface receivers read face values, which depend on tau
// too (rec_tau).  The host maps dL/dtheta and dL/dtau to
// dL/d(rho, kappa, lambda, mu); with tau given explicitly
// (hho_operators_build_tau) tau is a constant and only (1) remains.
//
// Checkpointing: U is stored every `checkpoint_every` steps in the forward
// pass; each segment is recomputed, keeping its stage values and their face
// traces, before its backward sweep.
//
// Arithmetic: the driver and its kernels are templates on the state type,
// FP64 (hho_adjoint_vjp) or FP32 (hho_adjoint_vjp_f32: the FP32 stage
// kernels, states, traces and adjoint vectors in FP32).  A cell's products of one
// backward stage are FP64 sums, or in FP32 scaled double-float ones
// (stage_kernels.cuh, Range); the sums over stages and steps are FP64 in both.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "hho_internal.h"

namespace {

// out = a x + b y over n values (x or y may be null: treated as zero; out may
// alias x or y, each element is read before it is written by the same thread).
template <class T>
__global__ void axpby_kernel(int64_t n, double a, const T* x, double b, const T* y, T* out) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        T v = T(0);
        if (x) v = T(a) * x[i];
        if (y) v = fma(T(b), y[i], v);
        out[i] = v;
    }
}

// d(G^T d)/dtau of an interface receiver at one time node.  Such a
// receiver records [p_F, v_F] = Ai w at its point, w = (tau_f p - m.n_f,
// tau_s v - s n_s) from the two cells' values there and A = [tau_f, n^T;
// -n, tau_s I]; so dd/dtau_f = Ai e_0 (p - p_F) and dd/dtau_s = Ai [0; v - v_F].
// grec[2r] (the fluid cell's tau) and grec[2r + 1] (the solid cell's) sum
// these over the time nodes; other receivers do not depend on tau.  One block a
// receiver, the eight field values by eight threads (as record_kernel).
template <class T>
__device__ __forceinline__ void rec_tau(const DevOps& op, int r, const int32_t* __restrict__ ri,
                                        const double* __restrict__ rd, const T* __restrict__ state,
                                        const T* __restrict__ G, double* __restrict__ grec) {
    __shared__ double val[8][10], g[8], w[3], o[3], hg[3];
    if (ri[4 * r] != 2) return;
    const int n = op.n, t = threadIdx.x;
    const double* d = rd + (size_t)r * (2 * n + 15);
    const int qf = ri[4 * r + 1], qs = ri[4 * r + 2];
    const T* ss = state + (size_t)3 * n * op.Nf;
    for (int e = t; e < 8 * n; e += blockDim.x) {   // m_x, m_y, p; s_xx, s_yy, s_xy, v_x, v_y
        const int fld = e / n, i = e - fld * n;
        val[fld][i] = fld < 3 ? (double)state[(size_t)(fld * n + i) * op.Nf + qf]
                              : (double)ss[(size_t)((fld - 3) * n + i) * op.Ns + qs];
    }
    __syncthreads();
    const double* Ai = d + 2 * n + 6;
    if (t < 8) {
        const double* phi = t < 3 ? d : d + n;
        double v = 0.0;
        for (int i = 0; i < n; ++i) v = fma(phi[i], val[t][i], v);
        g[t] = v;
    } else if (t < 11) {   // Ai^T g
        const int j = t - 8;
        hg[j] = Ai[j] * (double)G[5 * r] + Ai[3 + j] * (double)G[5 * r + 1] + Ai[6 + j] * (double)G[5 * r + 2];
    }
    __syncthreads();
    if (t < 3) {
        const double tf = d[2 * n], ts = d[2 * n + 1];
        const double nfx = d[2 * n + 2], nfy = d[2 * n + 3], nsx = d[2 * n + 4], nsy = d[2 * n + 5];
        w[t] = t == 0   ? tf * g[2] - (g[0] * nfx + g[1] * nfy)
               : t == 1 ? ts * g[6] - (g[3] * nsx + g[5] * nsy)
                        : ts * g[7] - (g[5] * nsx + g[4] * nsy);
    }
    __syncthreads();
    if (t < 3) o[t] = Ai[3 * t] * w[0] + Ai[3 * t + 1] * w[1] + Ai[3 * t + 2] * w[2];
    __syncthreads();
    if (t == 0) grec[2 * r] += hg[0] * (g[2] - o[0]);
    if (t == 1) grec[2 * r + 1] += hg[1] * (g[6] - o[1]) + hg[2] * (g[7] - o[2]);
}
// One time node's receiver part: lambda^ += S M^-1 R^T G (the transpose of
// record_kernel, lambda^ = S M^-1 lambda) and d(G^T d)/dtau of the interface
// receivers.  Blocks 0 .. n_inj - 1 own one cell that receivers read: thread
// (field, i) adds up the contributions of that cell's receivers in increasing
// receiver order, then the block applies the cell's inverse mass in shared
// memory.  The blocks after them take the interface receivers' tau terms, so
// that the two run side by side (one receiver a thread: 14.7 us a launch
// for 128 receivers, now 7.6).  blockDim >= 5 n.
template <class T>
__global__ void node_kernel(DevOps op, int n_inj, const int32_t* __restrict__ inj,
                            const int32_t* __restrict__ ri, const double* __restrict__ rd, const T* __restrict__ G,
                            const double* __restrict__ mass_f, const double* __restrict__ mass_s,
                            const double* __restrict__ cls_minv, const T* __restrict__ state, T* lam,
                            double* __restrict__ grec) {
    __shared__ double sh[2][50];
    const int n = op.n;
    const int stride = 2 * n + 15;
    if ((int)blockIdx.x >= n_inj) {
        rec_tau(op, (int)blockIdx.x - n_inj, ri, rd, state, G, grec);
        return;
    }
    const int t = blockIdx.x;
    const int fld = threadIdx.x / n, i = threadIdx.x - fld * n;
    const int dom = inj[n_inj + 1 + 2 * t], q = inj[n_inj + 1 + 2 * t + 1];
    const int nfld = dom == 0 ? 3 : 5;
    const int32_t* recs = inj + 3 * n_inj + 1;
    const int N = dom == 0 ? op.Nf : op.Ns;
    double acc = 0.0;
    if (fld < nfld)
        for (int e = inj[t]; e < inj[t + 1]; ++e) {
            const int r = recs[e];
            const double* d = rd + (size_t)r * stride;
            const int kind = ri[4 * r];
            double g[5];
            for (int j = 0; j < 5; ++j) g[j] = (double)G[5 * r + j];
            double v;
            const double* phi = d;
            if (kind == 0) {          // [p, m_x, m_y]
                v = fld == 2 ? g[0] : (fld == 0 ? g[1] : g[2]);
            } else if (kind == 1) {   // [v_x, v_y, s_xx, s_yy, s_xy]
                v = fld == 3 ? g[0] : fld == 4 ? g[1] : fld == 0 ? g[2] : fld == 1 ? g[3] : g[4];
            } else {                  // interface: [p_F, v_F] = Ai [w_f, w_sx, w_sy]
                const double tf = d[2 * n], ts = d[2 * n + 1];
                const double nfx = d[2 * n + 2], nfy = d[2 * n + 3], nsx = d[2 * n + 4], nsy = d[2 * n + 5];
                const double* Ai = d + 2 * n + 6;
                if (dom == 0) {
                    const double hf = Ai[0] * g[0] + Ai[3] * g[1] + Ai[6] * g[2];
                    v = fld == 2 ? tf * hf : (fld == 0 ? -nfx * hf : -nfy * hf);
                } else {
                    const double hx = Ai[1] * g[0] + Ai[4] * g[1] + Ai[7] * g[2];
                    const double hy = Ai[2] * g[0] + Ai[5] * g[1] + Ai[8] * g[2];
                    phi = d + n;
                    v = fld == 3 ? ts * hx
                        : fld == 4 ? ts * hy
                        : fld == 0 ? -nsx * hx
                        : fld == 2 ? -(nsy * hx + nsx * hy)
                                   : -nsy * hy;
                }
            }
            if (v != 0.0) acc += v * phi[i];
        }
    if (fld < nfld) sh[0][threadIdx.x] = acc;
    __syncthreads();
    const double* Mi = cls_minv + (size_t)op.warp_class[(dom == 0 ? 0 : op.n_warps_f) + (q >> 5)] * n * n;
    if (fld < nfld) {   // M0^-1 per field
        double v = 0.0;
        for (int j = 0; j < n; ++j) v = fma(Mi[i * n + j], sh[0][fld * n + j], v);
        sh[1][threadIdx.x] = v;
    }
    __syncthreads();
    if (fld >= nfld) return;
    const double y = sh[1][threadIdx.x];
    double v;
    if (dom == 0) {
        v = fld < 2 ? -y / mass_f[q] : y / mass_f[N + q];
    } else if (fld < 2) {   // (h^2 D)^-1 on (s_xx, s_yy), D = [[d0, d1], [d1, d0]]
        const double d0 = mass_s[q], d1 = mass_s[N + q], det = d0 * d0 - d1 * d1;
        v = -(d0 * y - d1 * sh[1][(1 - fld) * n + i]) / det;
    } else {
        v = fld == 2 ? -y / mass_s[2 * (size_t)N + q] : y / mass_s[3 * (size_t)N + q];
    }
    T* base = (dom == 0 ? lam : lam + (size_t)3 * n * op.Nf) + (size_t)(fld * n + i) * N + q;
    *base = T((double)*base + v);
}

template <class E>
struct AdjBuffers {
    int64_t S, T;           // state and trace sizes
    E *ckpt, *stages, *stage_tr, *erk_work, *lam, *X, *bufs, *tr[2];
    double *grad_f, *grad_s, *wgrad;
    double *gstab, *grec;   // tau parts: per device cell slot; per receiver (fluid, solid)
};

// Work layout in elements of E; the FP64 gradient sums take 8 / sizeof(E)
// elements per value (every piece starts on a 128-byte boundary).
template <class E>
int64_t adjoint_layout(const hho_ops* ops, const hho_tableau* tab, int64_t nsteps, int64_t C, AdjBuffers<E>* b,
                       E* base) {
    const int s = tab->s;
    const int64_t S = ops->n_state, T = ops->trace_doubles;
    const int64_t n_ckpt = (nsteps + C - 1) / C + 1;
    int64_t erk = 0;
    hho_work_size(ops, tab, &erk);
    int64_t off = 0;
    auto take = [&](int64_t n) {
        E* p = base ? base + off : nullptr;
        off += (n + 31) / 32 * 32;
        return p;
    };
    constexpr int64_t DW = (int64_t)(sizeof(double) / sizeof(E));
    auto take_d = [&](int64_t n) { return reinterpret_cast<double*>(take(n * DW)); };
    AdjBuffers<E> B;
    B.S = S;
    B.T = T;
    B.ckpt = take(n_ckpt * S);
    B.stages = take((C * s + 1) * S);     // stage inputs of a segment, then its end state
    B.stage_tr = take((C * s + 1) * T);   // their face traces
    B.erk_work = take(erk);
    B.lam = take(S);
    B.bufs = take(s * S);   // partial sums of the backward stages, at most one per row
    // the backward stages' values and traces: erk_run's layout of its work
    // buffer, which is idle between a segment's recompute and the next
    B.X = B.erk_work;
    std::vector<StagePlan> plan;
    int nb = 0;
    build_plan(tab, plan, &nb);
    for (int e = 0; e < 2; ++e) B.tr[e] = base ? B.erk_work + S * (1 + nb) + e * T : nullptr;
    B.grad_f = take_d(2 * (int64_t)ops->dev.Nf);
    B.grad_s = take_d(4 * (int64_t)ops->dev.Ns);
    B.wgrad = take_d(nsteps * s * MAX_SOURCES);
    B.gstab = take_d((int64_t)ops->dev.Nf + ops->dev.Ns);
    B.grec = take_d(2 * (int64_t)std::max(ops->n_rec, 1));
    if (b) *b = B;
    return off;
}

int64_t grid1(int64_t n) {
    int64_t g = (n + 255) / 256;
    return g > 4096 ? 4096 : (g < 1 ? 1 : g);
}

// the stage launcher and the operator data of the arithmetic
template <class E>
void launch_stage_t(const hho_ops* ops, int mode, StageArgsT<E>& a, double tn, int j, double cdt, bool sources,
                    void* stream);
template <>
void launch_stage_t<double>(const hho_ops* ops, int mode, StageArgsT<double>& a, double tn, int j, double cdt,
                            bool sources, void* stream) {
    launch_stage_f64(ops, mode, a, 1, tn, j, cdt, sources, stream);
}
template <>
void launch_stage_t<float>(const hho_ops* ops, int mode, StageArgsT<float>& a, double tn, int j, double cdt,
                           bool sources, void* stream) {
    launch_stage_f32(ops, mode, a, 1, tn, j, cdt, sources, stream);
}
int forward_steps(hho_ops* ops, const hho_tableau* tab, double t0, double dt, int64_t n, double* x, double* w,
                  void* stream) {
    return hho_erk_step(ops, tab, t0, dt, n, x, w, stream);
}
int forward_steps(hho_ops* ops, const hho_tableau* tab, double t0, double dt, int64_t n, float* x, float* w,
                  void* stream) {
    return erk_steps_f32(ops, tab, t0, dt, n, x, w, stream);
}
void launch_grad_t(const hho_ops* ops, StageArgsT<double>& a, const GradArgsT<double>& g, double tn, int j, double cdt,
                   void* stream) {
    launch_grad_f64(ops, a, g, tn, j, cdt, stream);
}
void launch_grad_t(const hho_ops* ops, StageArgsT<float>& a, const GradArgsT<float>& g, double tn, int j, double cdt,
                   void* stream) {
    launch_grad_f32(ops, a, g, tn, j, cdt, stream);
}

// The backward step as an explicit tableau on A' (file header): stage i of
// the plan is tableau stage j = s - 1 - i, row i < s holds z_j and row s the
// new lambda^.  sigma[j] = b_j where b_j is not small against the largest
// weight, else 1 (then row j starts from b_j lambda^ in its own buffer, or
// from zero).
struct AdjointPlan {
    std::vector<StagePlan> plan;
    double sigma[6];
    double init[6];   // of unscaled rows: b_j
    bool scaled[6];
    int buf[7];       // buffer of row i, -1: none
};
AdjointPlan adjoint_plan(const hho_tableau* tab) {
    const int s = tab->s;
    AdjointPlan P;
    double bmax = 0.0;
    for (int j = 0; j < s; ++j) bmax = std::max(bmax, std::fabs(tab->b[j]));
    for (int j = 0; j < s; ++j) {
        P.scaled[j] = std::fabs(tab->b[j]) > 1e-3 * bmax;
        P.sigma[j] = P.scaled[j] ? tab->b[j] : 1.0;
        P.init[j] = P.scaled[j] ? 0.0 : tab->b[j];
    }
    int nb = 0;
    bool touched[7] = {};
    for (int i = 0; i <= s; ++i) P.buf[i] = -1;
    for (int i = 1; i < s; ++i) {   // row 0 starts in X, see the driver
        if (P.init[s - 1 - i] == 0.0) continue;
        P.buf[i] = nb++;
        touched[i] = true;
    }
    P.plan.assign(s, StagePlan{});
    for (int l = 0; l < s; ++l) {
        const int tl = s - 1 - l;   // tableau stage
        for (int r = l + 1; r <= s; ++r) {
            const int tj = s - 1 - r;
            const double a = r == s ? P.sigma[tl] : P.sigma[tl] * tab->a[tl][tj] / P.sigma[tj];
            if (a == 0.0 && r > l + 1) continue;
            const bool last = r == l + 1;   // row complete after this stage
            TargetPlan t;
            t.src = touched[r] ? P.buf[r] : (r == s || P.scaled[tj]) ? SRC_STATE : SRC_ZERO;
            if (last) {
                t.dst = r == s ? SRC_STATE : SRC_X;
            } else {
                if (P.buf[r] < 0) P.buf[r] = nb++;
                t.dst = P.buf[r];
                touched[r] = true;
            }
            t.a = a;
            P.plan[l].t[P.plan[l].n_tgt++] = t;   // r = l + 1 comes first: target 0
        }
    }
    return P;
}

template <class E>
int adjoint_vjp_t(hho_ops* ops, const hho_tableau* tab, double t0, double dt, int64_t nsteps, int64_t checkpoint_every,
                  const E* d_state0, const E* d_cotangent, E* d_work, int64_t work_elems, double* h_grad_cell,
                  double* h_grad_wavelet, double* h_grad_tau, void* stream, const char* who);

}  // namespace

extern "C" int hho_adjoint_work_size(const hho_ops* ops, const hho_tableau* tab, int64_t nsteps,
                                     int64_t checkpoint_every, int64_t* n_doubles) {
    if (!ops || !tab || !n_doubles || nsteps < 1 || checkpoint_every < 1) {
        hho_set_error("hho_adjoint_work_size: bad arguments");
        return HHO_EINVAL;
    }
    *n_doubles = adjoint_layout<double>(ops, tab, nsteps, checkpoint_every, nullptr, nullptr);
    return HHO_OK;
}

extern "C" int hho_adjoint_work_size_f32(const hho_ops* ops, const hho_tableau* tab, int64_t nsteps,
                                         int64_t checkpoint_every, int64_t* n_floats) {
    if (!ops || !tab || !n_floats || nsteps < 1 || checkpoint_every < 1) {
        hho_set_error("hho_adjoint_work_size_f32: bad arguments");
        return HHO_EINVAL;
    }
    *n_floats = adjoint_layout<float>(ops, tab, nsteps, checkpoint_every, nullptr, nullptr);
    return HHO_OK;
}

extern "C" int hho_adjoint_vjp(hho_ops* ops, const hho_tableau* tab, double t0, double dt, int64_t nsteps,
                               int64_t checkpoint_every, const double* d_state0, const double* d_cotangent,
                               double* d_work, int64_t work_doubles, double* h_grad_cell, double* h_grad_wavelet,
                               double* h_grad_tau, void* stream) {
    return adjoint_vjp_t<double>(ops, tab, t0, dt, nsteps, checkpoint_every, d_state0, d_cotangent, d_work,
                                 work_doubles, h_grad_cell, h_grad_wavelet, h_grad_tau, stream, "hho_adjoint_vjp");
}

extern "C" int hho_adjoint_vjp_f32(hho_ops* ops, const hho_tableau* tab, double t0, double dt, int64_t nsteps,
                                   int64_t checkpoint_every, const float* d_state0, const float* d_cotangent,
                                   float* d_work, int64_t work_floats, double* h_grad_cell, double* h_grad_wavelet,
                                   double* h_grad_tau, void* stream) {
    return adjoint_vjp_t<float>(ops, tab, t0, dt, nsteps, checkpoint_every, d_state0, d_cotangent, d_work,
                                work_floats, h_grad_cell, h_grad_wavelet, h_grad_tau, stream, "hho_adjoint_vjp_f32");
}

namespace {
template <class E>
int adjoint_vjp_t(hho_ops* ops, const hho_tableau* tab, double t0, double dt, int64_t nsteps, int64_t checkpoint_every,
                  const E* d_state0, const E* d_cotangent, E* d_work, int64_t work_doubles, double* h_grad_cell,
                  double* h_grad_wavelet, double* h_grad_tau, void* stream, const char* who) {
    if (!ops || !tab || !d_state0 || !d_cotangent || !d_work || !h_grad_cell || nsteps < 1 || checkpoint_every < 1 ||
        !std::isfinite(dt)) {
        hho_set_error("%s: bad arguments", who);
        return HHO_EINVAL;
    }
    std::vector<StagePlan> plan;
    int nb = 0;
    if (build_plan(tab, plan, &nb) != HHO_OK) {
        hho_set_error("%s: unsupported tableau", who);
        return HHO_EINVAL;
    }
    const int64_t C = checkpoint_every;
    const int s = tab->s;
    AdjBuffers<E> B;
    const int64_t need = adjoint_layout<E>(ops, tab, nsteps, C, &B, d_work);
    if (work_doubles < need) {
        hho_set_error("%s: work buffer has %lld elements, needs %lld", who, (long long)work_doubles, (long long)need);
        return HHO_EINVAL;
    }
    cudaStream_t st = (cudaStream_t)stream;
    const int64_t S = B.S;
    const int nthr = ops->dev.Nf + ops->dev.Ns;
    const AdjointPlan back = adjoint_plan(tab);
    int rc = HHO_OK;
    auto copy = [&](E* dst, const E* src, int64_t n) {
        return cudaMemcpyAsync(dst, src, sizeof(E) * n, cudaMemcpyDeviceToDevice, st) == cudaSuccess;
    };
    // the ERK partial-sum buffers of the segment recompute, laid out as in
    // erk_run ([X][partial sums][2 traces]; X and the traces live in the
    // segment store here)
    E* bufs = B.erk_work + S;
    auto partial = [&](int code) -> E* { return code == SRC_ZERO ? nullptr : bufs + S * code; };
    DevOps adj = ops->dev;
    adj.if_coef = ops->d_if_coef_adj;
    adj.if_coef_f32 = ops->d_if_coef_adj_f32;

    // ---- forward pass: checkpoints ------------------------------------------------
    if (!copy(B.ckpt, d_state0, S)) {
        hho_set_error("%s: copy failed", who);
        return HHO_ECUDA;
    }
    const int64_t n_segments = (nsteps + C - 1) / C;
    for (int64_t c = 1; c < n_segments; ++c) {   // the last segment's end state is not a checkpoint
        if (!copy(B.ckpt + c * S, B.ckpt + (c - 1) * S, S)) return HHO_ECUDA;
        rc = forward_steps(ops, tab, t0 + (double)((c - 1) * C) * dt, dt, C, B.ckpt + c * S, B.erk_work, stream);
        if (rc) return rc;
    }

    // ---- backward sweep ---------------------------------------------------------------
    auto zero = [&](void* p, size_t bytes) { return bytes == 0 || cudaMemsetAsync(p, 0, bytes, st) == cudaSuccess; };
    // all zero bits are +0.0; padding slots of X and the partial sums are never read
    if (!zero(B.lam, sizeof(E) * S) ||
        !zero(B.grad_f, sizeof(double) * 2 * ops->dev.Nf) || !zero(B.grad_s, sizeof(double) * 4 * ops->dev.Ns) ||
        !zero(B.gstab, sizeof(double) * nthr) || !zero(B.grec, sizeof(double) * 2 * std::max(ops->n_rec, 1))) {
        hho_set_error("%s: work initialisation failed", who);
        return HHO_ECUDA;
    }
    for (int64_t seg = n_segments - 1; seg >= 0; --seg) {
        const int64_t n0 = seg * C;                                   // segment starts at U^{n0}
        const int64_t nst = (n0 + C <= nsteps) ? C : nsteps - n0;
        // Recompute the segment.  Stage j of step m reads its input Y_{m,j}
        // and that input's face traces from slot m s + j of the segment store
        // and writes the next stage input (slot m s + j + 1, or the next
        // step's state in slot (m + 1) s) with its traces straight into the
        // store: no copies, and the backward sweep needs no trace launch for
        // the forward stage values.
        auto Y = [&](int64_t m, int j) { return B.stages + (m * s + j) * S; };
        auto TY = [&](int64_t m, int j) { return B.stage_tr + (m * s + j) * B.T; };
        if (!copy(Y(0, 0), B.ckpt + seg * S, S)) return HHO_ECUDA;
        StageArgsT<E> a;
        memset(&a, 0, sizeof(a));
        a.op = ops->dev;
        a.inp = Y(0, 0);
        a.tr_out = TY(0, 0);
        launch_stage_t<E>(ops, MODE_TRACES, a, 0.0, -1, 0.0, false, stream);
        for (int64_t m = 0; m < nst; ++m) {
            const double tn = t0 + (double)(n0 + m) * dt;
            for (int j = 0; j < s; ++j) {
                const StagePlan& P = plan[j];
                const bool last = j + 1 == s;
                a.inp = Y(m, j);
                a.tr_in = TY(m, j);
                a.tr_out = last ? TY(m + 1, 0) : TY(m, j + 1);
                a.n_tgt = P.n_tgt;
                for (int t = 0; t < P.n_tgt; ++t) {
                    const int sc = P.t[t].src, dc = P.t[t].dst;
                    a.tgt[t].src = sc == SRC_STATE ? Y(m, 0) : partial(sc);
                    a.tgt[t].dst = dc == SRC_STATE ? Y(m + 1, 0) : dc == SRC_X ? Y(m, j + 1) : partial(dc);
                    a.tgt[t].coef = E(P.t[t].a * dt);
                }
                launch_stage_t<E>(ops, MODE_STAGE, a, tn, j, tab->c[j] * dt, true, stream);
            }
        }
        rc = check_cuda(who);
        if (rc) return rc;
        // backward through the segment
        for (int64_t m = nst - 1; m >= 0; --m) {
            const int64_t n = n0 + m + 1;                            // step n: U^{n-1} -> U^n
            const double tn = t0 + (double)(n - 1) * dt;
            if (ops->n_rec > 0) {   // U^n is the next step's first stage value in the store
                const int thr = (5 * ops->n + 31) / 32 * 32;
                node_kernel<E><<<ops->n_inj + ops->n_rec, thr, 0, st>>>(
                    ops->dev, ops->n_inj, ops->d_inj, ops->d_rec_int, ops->d_rec_dbl,
                    d_cotangent + (size_t)(n - 1) * 5 * ops->n_rec, ops->d_mass_f, ops->d_mass_s, ops->d_cls_minv,
                    Y(m + 1, 0), B.lam, B.grec);
            }
            // rows of unscaled stages start from b_j lambda^ (row 0, the first stage's input, in X)
            const E* z = back.scaled[s - 1] ? B.lam : B.X;
            if (!back.scaled[s - 1])
                axpby_kernel<E><<<grid1(S), 256, 0, st>>>(S, back.init[s - 1], B.lam, 0.0, nullptr, B.X);
            for (int i = 1; i < s; ++i)
                if (back.init[s - 1 - i] != 0.0)
                    axpby_kernel<E><<<grid1(S), 256, 0, st>>>(S, back.init[s - 1 - i], B.lam, 0.0, nullptr,
                                                              B.bufs + back.buf[i] * S);
            StageArgsT<E> b;
            memset(&b, 0, sizeof(b));
            b.op = adj;
            b.inp = z;
            b.tr_out = B.tr[0];
            launch_stage_t<E>(ops, MODE_TRACES, b, 0.0, -1, 0.0, false, stream);
            int cur = 0;
            for (int i = 0; i < s; ++i) {
                const int j = s - 1 - i;
                // gradients of stage j: the rate of Y_{m,j} (its traces are stored) against mu_j = dt sigma_j S M z_j
                StageArgsT<E> r;
                memset(&r, 0, sizeof(r));
                r.op = ops->dev;
                r.inp = Y(m, j);
                r.tr_in = TY(m, j);
                GradArgsT<E> g;
                g.z = z;
                g.tr_z = B.tr[cur];
                g.if_coef_z = ops->d_if_coef_adj;
                g.w = dt * back.sigma[j];
                g.mass_f = ops->d_mass_f;
                g.mass_s = ops->d_mass_s;
                g.grad_f = B.grad_f;
                g.grad_s = B.grad_s;
                g.gstab = B.gstab;
                g.wgrad = h_grad_wavelet ? B.wgrad + ((n - 1) * s + j) * MAX_SOURCES : nullptr;
                launch_grad_t(ops, r, g, tn, j, tab->c[j] * dt, stream);
                // the next row and the partial sums: nu^_j = dt sigma_j A' z_j
                const StagePlan& P = back.plan[i];
                auto at = [&](int code) -> E* {
                    return code == SRC_STATE ? B.lam : code == SRC_X ? B.X : code == SRC_ZERO ? nullptr : B.bufs + S * code;
                };
                b.inp = z;
                b.tr_in = B.tr[cur];
                b.tr_out = B.tr[cur ^ 1];
                b.n_tgt = P.n_tgt;
                for (int t = 0; t < P.n_tgt; ++t) {
                    b.tgt[t].src = at(P.t[t].src);
                    b.tgt[t].dst = at(P.t[t].dst);
                    b.tgt[t].coef = E(P.t[t].a * dt);
                }
                launch_stage_t<E>(ops, MODE_STAGE, b, 0.0, -1, 0.0, false, stream);
                z = B.X;
                cur ^= 1;
                rc = check_cuda(who);
                if (rc) return rc;
            }
        }
    }
    // ---- gradients to the host, mapped to the materials ----------------------------------------
    // What the mapping needs besides the sums is prepared while the GPU works:
    // o[0..3] = dL/d(rho, kappa, lambda, mu) are linear in the cell's sums.
    const int Nf = ops->dev.Nf, Ns = ops->dev.Ns;
    const int64_t nc = ops->nc;
    std::vector<double> gf(2 * (size_t)Nf), gs(4 * (size_t)Ns);
    std::vector<double> gstab((size_t)nthr), grec(2 * (size_t)std::max(ops->n_rec, 1));
    std::vector<double> gtau((size_t)nc, 0.0);
    std::vector<int32_t> orig((size_t)nthr, -1);
    struct Map {
        double m[4];   // fluid: d(A_m)/d rho, 1/h; solid: d(A_v)/d rho, 1/h, dr/d lambda, dr/d mu
        double t[3];   // dtau/d rho, and / d kappa or d lambda, and / d mu
    };
    std::vector<Map> map((size_t)nc);
    for (int64_t c = 0; c < nc; ++c) {
        Map& M = map[c];
        const double h = ops->diam[c], rho = ops->rho[c], t = ops->tau[c];
        orig[(ops->cell_dom[c] == 0 ? 0 : Nf) + ops->cell_pos[c]] = (int32_t)c;
        M.m[0] = -1.0 / (rho * rho * h);   // A_m = 1/(rho h), A_v = 1/(rho h)
        M.m[1] = 1.0 / h;                  // A_p = kappa/h, c1 = (lambda + 2 mu)/h, c3 = mu/h
        // tau^f = eta_f (rho kappa)^-1/2; tau^s = eta_s (rho (lambda + 2 mu))^1/2 or eta_s (rho mu)^1/2
        // (an optional 1/k factor cancels in these logarithmic derivatives)
        if (ops->cell_dom[c] == 0) {
            M.t[0] = -0.5 * t / rho;
            M.t[1] = -0.5 * t / ops->kappa[c];
            M.t[2] = 0.0;
        } else {
            const double lam = ops->lam[c], mu = ops->mu[c], l2m = lam + 2.0 * mu;
            M.m[2] = 2.0 * mu / (l2m * l2m);    // r = lambda/(lambda + 2 mu)
            M.m[3] = -2.0 * lam / (l2m * l2m);
            M.t[0] = 0.5 * t / rho;
            M.t[1] = ops->stab_speed == 0 ? 0.5 * t / l2m : 0.0;
            M.t[2] = ops->stab_speed == 0 ? t / l2m : 0.5 * t / mu;
        }
    }
    std::vector<int32_t> ri(4 * (size_t)std::max(ops->n_rec, 1));
    std::vector<double> wg(ops->n_src > 0 && h_grad_wavelet ? (size_t)nsteps * s * MAX_SOURCES : 0);
    auto fetch = [&](void* dst, const void* src, size_t bytes) {
        return bytes == 0 || cudaMemcpyAsync(dst, src, bytes, cudaMemcpyDeviceToHost, st) == cudaSuccess;
    };
    if (!fetch(gf.data(), B.grad_f, sizeof(double) * gf.size()) || !fetch(gs.data(), B.grad_s, sizeof(double) * gs.size()) ||
        !fetch(gstab.data(), B.gstab, sizeof(double) * gstab.size()) ||
        !fetch(grec.data(), B.grec, sizeof(double) * grec.size()) ||
        !fetch(wg.data(), B.wgrad, sizeof(double) * wg.size()) ||
        !fetch(ri.data(), ops->d_rec_int, sizeof(int32_t) * 4 * ops->n_rec) || cudaStreamSynchronize(st) != cudaSuccess) {
        hho_set_error("%s: gradient copy failed", who);
        return HHO_ECUDA;
    }
    for (int64_t e = 0; e < (int64_t)(wg.size() / MAX_SOURCES); ++e)
        for (int k2 = 0; k2 < ops->n_src; ++k2) h_grad_wavelet[e * ops->n_src + k2] = wg[e * MAX_SOURCES + k2];
    // dL/dtau per cell: the stage part (face integrals scale with h) and the
    // interface receivers' part, mapped from device positions to cell ids
    for (int g = 0; g < nthr; ++g)
        if (orig[g] >= 0) gtau[orig[g]] = -ops->diam[orig[g]] * gstab[g];
    for (int r = 0; r < ops->n_rec; ++r)
        if (ri[4 * r] == 2) {
            gtau[orig[ri[4 * r + 1]]] += grec[2 * r];
            gtau[orig[Nf + ri[4 * r + 2]]] += grec[2 * r + 1];
        }
    if (h_grad_tau) std::copy(gtau.begin(), gtau.end(), h_grad_tau);
    for (int64_t c = 0; c < nc; ++c) {
        double* o = h_grad_cell + 4 * c;
        const Map& M = map[c];
        const int q = ops->cell_pos[c];
        o[0] = o[1] = o[2] = o[3] = 0.0;
        if (ops->cell_dom[c] == 0) {
            o[0] = gf[q] * M.m[0];
            o[1] = gf[Nf + q] * M.m[1];
        } else {
            const double gc1 = gs[q], gr = gs[Ns + q], gc3 = gs[2 * Ns + q], gav = gs[3 * Ns + q];
            o[0] = gav * M.m[0];
            o[2] = gc1 * M.m[1] + gr * M.m[2];
            o[3] = gc1 * 2.0 * M.m[1] + gr * M.m[3] + gc3 * M.m[1];
        }
        if (ops->tau_explicit) continue;
        const double gt = gtau[c];
        o[0] += gt * M.t[0];
        if (ops->cell_dom[c] == 0) {
            o[1] += gt * M.t[1];
        } else {
            if (ops->stab_speed == 0) o[2] += gt * M.t[1];
            o[3] += gt * M.t[2];
        }
    }
    return HHO_OK;
}
}  // namespace
