// Internal declarations shared by the host C++ sources and the CUDA sources.
#pragma once

#include <cstdint>
#include <string>
#include <vector>

#include "hho.h"

void hho_set_error(const char* fmt, ...);

#if defined(__CUDACC__)
#define HHO_HD __host__ __device__
#else
#define HHO_HD
#endif

// A double-float value hi + lo: two FP32 numbers with hi = RN(hi + lo),
// about 48 significant bits (arithmetic in f2x.cuh).  8 bytes: arrays of it
// have the layout of FP64 arrays.
struct alignas(8) f2x {
    float hi, lo;
    f2x() = default;
    HHO_HD constexpr f2x(float h, float l) : hi(h), lo(l) {}
    HHO_HD constexpr explicit f2x(int v) : hi((float)v), lo(0.0f) {}
    // split of an FP64 value: hi = RN(v), lo = RN(v - hi) (v - hi is exact)
    HHO_HD explicit f2x(double v) : hi((float)v), lo((float)(v - (double)(float)v)) {}
    HHO_HD explicit operator double() const { return (double)hi + (double)lo; }
};

// Face types (Sec. 3.1 face sets).
enum { FT_FLUID = 0, FT_SOLID = 1, FT_IFACE = 2, FT_BND_FLUID = 3, FT_BND_SOLID = 4 };

struct hho_mesh {
    int64_t nv = 0, nc = 0, nf = 0;
    std::vector<double> xy;            // 2 nv
    std::vector<int64_t> cell_ptr;     // nc + 1
    std::vector<int64_t> cell_vtx;
    std::vector<uint8_t> domain;       // nc
    std::vector<int64_t> rep;          // nv
    std::vector<int64_t> face_cells;   // 2 nf
    std::vector<int32_t> face_local;   // 2 nf: local edge index in cell 0 / cell 1
    std::vector<int64_t> cell_faces;   // indexed by cell_ptr
    std::vector<int32_t> face_type, face_colour, cell_class;
    std::vector<double> centroid;      // 2 nc
    std::vector<double> diam, area;    // nc
    int32_t n_classes = 0, n_colours = 0, max_nf = 0;
    std::vector<int64_t> class_first;  // first cell of each class
    // per class: vertex coordinates relative to the reference cell's centroid
    // over its diameter, [x_0, y_0, x_1, ...] from class_ref_off[cl]; the
    // class matrices are built from these.  A sub-mesh inherits them from its
    // parent mesh, so its operators use the same class matrices bit for bit.
    std::vector<double> class_ref;
    std::vector<int64_t> class_ref_off;
};

// Per-class integer record on the device (stride CI_STRIDE ints).
// CI_HOR, CI_VER: bit j set where local face j (a cell has at most 32,
// hho_mesh_create) is horizontal (n_x = 0) or vertical (n_y = 0).
enum { CI_DOMAIN = 0, CI_NF, CI_START, CI_COUNT, CI_NPAD, CI_SLOT, CI_DOFF, CI_KIND, CI_HOR, CI_VER, CI_STRIDE };

// Class kinds: generic polygon (dense class matrices) or axis-aligned
// rectangle with faces ordered bottom, right, top, left, whose trace and
// lifting matrices have a sparsity pattern fixed by monomial parity; a
// square rectangle's traces are known in closed form (operators.cpp).
enum { KIND_GENERIC = 0, KIND_RECT = 1, KIND_SQUARE = 2 };

// Scale of the face basis psi_l = (FACE_RHO xi)^l, xi in [-1, 1] along a
// face: 1/(2 sqrt 2), the half side over the diameter of a square, so that a
// square cell's scaled coordinates are +-FACE_RHO on its faces.
#define FACE_RHO 0.35355339059327376220

// Device-side description of one stage launch and the static operator data.
struct DevOps {
    int32_t k, n, f;
    int32_t Nf, Ns;          // padded cell slots per domain (multiples of 32)
    int32_t SF, SS;          // face-side slots per domain
    int32_t n_warps_f, n_warps_s;
    int32_t max_nf;              // most faces of any class
    int32_t n_warps_rect;        // warps whose class is a rectangle
    const int32_t* warp_class;   // [n_warps_f + n_warps_s]
    const int32_t* cls_int;      // [n_classes][CI_STRIDE]
    const double* cls_dbl;       // class matrices, see operators.cpp
    const double* scal_f;        // fluid per-cell scalars [SCF][Nf]
    const double* scal_s;        // solid per-cell scalars [SCS][Ns]
    const int32_t* nb_f;         // face-side neighbour slot, fluid [SF]
    const int32_t* nb_s;         // solid [SS]
    const double* beta_f;        // face-side coefficient, fluid [SF]
    const double* beta_s;        // solid [SS]
    const int32_t* if_nb;        // interface records: neighbour slot in the other domain
    const double* if_coef;       // interface records: 6 coefficients each
    // FP32 copies of the same data, for the FP32 batched path
    const float* cls_f32;
    const float* scal_f_f32;
    const float* scal_s_f32;
    const float* beta_f_f32;
    const float* beta_s_f32;
    const float* if_coef_f32;
    // double-float copies, for the double-float path
    const f2x* cls_x;
    const f2x* scal_f_x;
    const f2x* scal_s_x;
    const f2x* beta_f_x;
    const f2x* beta_s_x;
    const f2x* if_coef_x;
};

// Fluid scalars: A_m = 1/(rho h), A_p = kappa/h, tau.  Solid: c1 = (lambda+2mu)/h,
// r = lambda/(lambda+2mu), c3 = mu/h, A_v = 1/(rho h), tau.
enum { SF_AM = 0, SF_AP, SF_TAU, SCF };
enum { SS_C1 = 0, SS_R, SS_C3, SS_AV, SS_TAU, SCS };

// Face-side neighbour encoding: >= 0 same-domain neighbour slot, -1 boundary,
// <= -2 interface record (-2 - r).
constexpr int32_t NB_BOUNDARY = -1;

constexpr int GB300_SMS = 152;

constexpr int MAX_TARGETS = 6;        // of a stage launch: the adjoint of an accepted tableau may need six
constexpr int MAX_PLAN_TARGETS = 4;   // of a forward tableau's stage (build_plan)
constexpr int MAX_SOURCES = 8;

// Simulation clock read by graph-replayed stage kernels: the time of stage
// j of step n of a call is (t0 + n dt) + c_j dt.
struct StageClock {
    double t0;
    int64_t step;
    uint32_t ticket;   // blocks of the receiver kernel that have read the step
    uint32_t pad;
};

template <class T>
struct TargetT {
    const T* src;   // nullptr: zero
    T* dst;
    T coef;
};

// One stage launch.  Shots are blockIdx.y; every state, trace and target
// pointer is the base of shot 0 and advances by state_stride / trace_stride
// elements per shot.
template <class T>
struct StageArgsT {
    DevOps op;
    const T* inp;            // device-layout state read by the stage
    const T* tr_in;          // traces of inp: fluid [2f][SF] then solid [4f][SS]
    T* tr_out;               // traces of the target-0 result (same layout)
    TargetT<T> tgt[MAX_TARGETS];
    int32_t n_tgt;
    int32_t warp0, n_warps;  // the launch's warps of cells (of both domains' concatenation); n_warps 0: all
    int32_t pad0;
    int64_t state_stride, trace_stride;
    // point sources applied to every shot
    int32_t n_src;
    int32_t src_dom[MAX_SOURCES];
    int32_t src_q[MAX_SOURCES];
    T src_w[MAX_SOURCES];            // wavelet value at the stage time
    const T* src_g;                  // [n_src][2][n] lifted load vectors
    // one point source per shot (batched shots); shot_src_q == nullptr: none
    const int32_t* shot_src_dom;
    const int32_t* shot_src_q;
    const T* shot_src_g;             // [shots][2][n]
    T shot_src_w;
    // graph replay: with clock set the stage time comes from the device clock
    // and the wavelets are evaluated in the kernel from these parameters
    const StageClock* clock;
    double dt, c_stage;
    double src_f0[MAX_SOURCES], src_t0[MAX_SOURCES], src_amp[MAX_SOURCES];
    double shot_f0, shot_t0, shot_amp;
};

// MODE_GRAD forms the rate before the per-cell material factors (and, in
// solids, before the stress mixing), which is the derivative of the rate with
// respect to those factors, and accumulates one backward stage's share of the
// adjoint gradients from it (GradArgsT).
enum { MODE_TRACES = 0, MODE_STAGE = 1, MODE_APPLY = 2, MODE_GRAD = 3 };

// The adjoint side of a MODE_GRAD launch: the adjoint stage value z with its
// traces under the coupling-reversed operator, and the gradient sums.  The
// stage's adjoint is mu = w S M z (adjoint.cu).
template <class T>
struct GradArgsT {
    const T* z;
    const T* tr_z;
    const double* if_coef_z;   // interface coefficients of the coupling-reversed operator
    double w;
    const double* mass_f;      // [2][Nf]: rho h^2, h^2/kappa
    const double* mass_s;      // [4][Ns]: h^2 compliance (3), rho h^2
    double* grad_f;            // [2][Nf]: d/d(1/(rho h)), d/d(kappa/h)
    double* grad_s;            // [4][Ns]: d/d(c1, r, c3, 1/(rho h))
    double* gstab;             // [Nf + Ns]: sum of face integrals of the jump products
    double* wgrad;             // [n_src]: mu^T g (may be null)
};

// ERK plan (stage.cu): row i of the extended tableau (a_{s+1,:} = b) is the
// partial sum P_i = U^{n-1} + dt sum_j a_ij k_j.
enum { SRC_ZERO = -3, SRC_STATE = -2, SRC_X = -1 };   // >= 0: row buffer index
struct TargetPlan {
    int src, dst;
    double a;
};
struct StagePlan {
    int n_tgt;
    TargetPlan t[MAX_TARGETS];
};
void free_host_pipe(struct HostPipe* p);
int build_plan(const hho_tableau* tab, std::vector<StagePlan>& plan, int* n_buf);

// Launches one stage-kernel pass (FP64) over n_shots shots; and the receiver
// kernel.  Defined in stage.cu, used by the adjoint driver.
struct hho_ops;
// Stage launch for the adjoint and SDIRK drivers.  Sources (when `sources`)
// are evaluated for step time tn, stage j (time tn + cdt); j < 0 for calls
// that have no stage index (sampled source time functions are then zero).
void launch_stage_f64(const hho_ops* ops, int mode, StageArgsT<double>& a, int n_shots, double tn, int j, double cdt,
                      bool sources, void* stream);
void launch_stage_f32(const hho_ops* ops, int mode, StageArgsT<float>& a, int n_shots, double tn, int j, double cdt,
                      bool sources, void* stream);
void launch_grad_f64(const hho_ops* ops, StageArgsT<double>& a, const GradArgsT<double>& g, double tn, int j, double cdt,
                     void* stream);
void launch_grad_f32(const hho_ops* ops, StageArgsT<float>& a, const GradArgsT<float>& g, double tn, int j, double cdt,
                     void* stream);
void launch_record_f64(const hho_ops* ops, const double* state, double* out, void* stream);
// nsteps ERK steps of one FP32 state (the batched FP32 path with one shot)
int erk_steps_f32(hho_ops* ops, const hho_tableau* tab, double t0, double dt, int64_t nsteps, float* d_state,
                  float* d_work, void* stream);
int check_cuda(const char* what);
// y = *scale P^-1 x (scale null: 1; bj null: P = I; accumulate: y += ..., not with
// traces), P^-1 the inverse cell blocks of hho_ops::d_bj; with tr, the FP64
// face traces of y too.
void launch_bj(const hho_ops* ops, const double* bj, const double* x, const double* scale, double* y, bool accumulate,
               double* tr, void* stream);

// The pieces of a host-buffer call on a large mesh: host pieces are runs of
// canonical cells, compute pieces runs of warps in the device order.  The copy
// engine brings host piece c while earlier pieces are packed, traced and taken
// through the first stage; after the last stage each piece returns as soon as its
// cells are done.  A compute piece's traces need its own cells, its first stage
// the traces of its face neighbours too.  The order only decides what overlaps:
// a mesh whose device order is unrelated to its cell order runs one after the other.
//
// Two, four or eight pieces of 2000 warps of cells and more (smaller ones leave the
// SMs idle between them for longer than the copies they hide; three cut a piece at
// the domains' border), from BYTES on each way, and one where not even the traces
// of a piece can start before the last one has arrived: the second pass over memory
// and the smaller grids then cost more than overlaps.  One step of ERK4, us, by
// pieces 1 | 2 | 4 | 8, FP64 and double-float:
//   1024 x 512, k = 2, 100 MB         2032 | 1916 | 1847 | 1745    1829 | 1745 | 1711 | 1661
//   1024 x 512, k = 1, 50 MB          1066 | 1014 | 1006 |  981     972 |  933 |  922 |  954
//   724 x 362, k = 2, 50 MB           1106 | 1057 | 1032 | 1050    1049 |  996 | 1023 |  969
//   512 x 272, k = 3, 45 MB            991 |  942 |  962 | 1075     924 |  883 |  901 |  992
//   512 x 272, k = 2, 27 MB            610 |  599 |  610 |  717     551 |  576 |  569 |  635
//   724 x 362, k = 1, 25 MB            602 |  588 |  600 |  658     520 |  503 |  556 |  574
//   512 x 512 triangles, k = 2, 100 MB 2796 | 2598 | 2663 | 2597   1940 | 1843 | 1845 | 1804
// and where two pieces both wait for the last arrival, and with four every stage does:
//   400 x 400 hybrid, k = 3, 63 MB    1556 | 1654 | 1590 | 1630    1291 | 1380 | 1258 | 1281
//   300 x 300 triangles, k = 3, 58 MB 1782 | 1923 | 1935 | 1895    1239 | 1324 | 1281 | 1291
//   400 x 400 hanging, k = 3, 52 MB   1201 | 1326 | 1342 | 1320    1112 | 1183 | 1093 | 1123
//   680 x 340 hybrid, k = 3, 91 MB    2173 | 2262 | 2190 | 2193    1773 | 1901 | 1734 | 1692
//   800 x 600 hanging, k = 2, 91 MB   2066 | 2173 | 2078 | 1974    1759 | 1856 | 1862 | 1718
//   1000 x 700 hybrid, k = 2, 175 MB  3835 | 3959 | 3596 | 3404    3046 | 3173 | 2931 | 2776
constexpr int STAGED_CELLS = 64;   // cells of a block of the host pack kernels
struct HostPieces {
    static constexpr int MAX = 8, WARPS = 2000;
    static constexpr int64_t BYTES = 40000000;
    int n = 0;   // 0: not cut yet (cut_host_pieces, under the GPU's work of the first pinned call)
    int blocks[MAX + 1], warps[MAX + 1];   // host pieces in blocks of STAGED_CELLS cells, compute pieces in warps
    int64_t off[MAX + 1];                  // host pieces in values
    int own[MAX], need[MAX];               // the last host piece that compute piece d's traces / first stage wait for
    int order[MAX];                        // compute pieces by need
    int last[MAX];                         // host piece c is complete after order[last[c]]
};
struct HostPipe;
struct hho_ops {
    int32_t k = 0, n = 0, f = 0;
    int64_t nc = 0;
    int32_t n_classes = 0;
    DevOps dev{};
    // device allocations owned by ops
    std::vector<void*> allocations;
    // host copies needed later
    std::vector<int32_t> cell_dom, cell_pos;   // per original cell: domain, device position
    std::vector<int64_t> canon_off;            // per original cell: offset in canonical vector
    int64_t n_canonical = 0;
    int32_t* d_dev2orig = nullptr;             // [Nf + Ns]: original cell id or -1 (padding)
    int64_t* d_canon_off = nullptr;            // [nc]
    int32_t* d_cell_dom = nullptr;             // [nc]: 0 fluid, 1 solid
    int32_t* d_cell_pos = nullptr;             // [nc]: device position within the cell's domain
    double c_max = 0.0, h_min = 0.0;
    // host-side per-cell data kept for sources/receivers
    std::vector<double> centroid, diam, rho, tau;
    bool tau_explicit = false;   // tau given by the caller (hho_operators_build_tau): not a function of the materials
    int32_t stab_speed = 0;      // c^s in tau^s: 0 = c_P, 1 = c_S
    std::vector<int32_t> cell_class_of;
    std::vector<std::vector<double>> class_M0inv;     // per class, n x n
    std::vector<std::vector<double>> class_normals;   // per class, 2 per face
    std::vector<double> kappa, lam, mu;
    std::vector<double> poly_xy;                      // copy of vertex coordinates for location
    std::vector<int64_t> poly_ptr, poly_vtx;
    std::vector<uint8_t> poly_dom;
    std::vector<int64_t> face_cells, cell_faces;
    std::vector<int32_t> face_type, face_local;
    std::vector<int64_t> iface_faces;                 // the fluid-solid interface faces
    // point location: uniform bucket grid over the cells' bounding boxes,
    // each bucket listing its cells in increasing order
    int32_t loc_gx = 0, loc_gy = 0;
    double loc_x0 = 0.0, loc_y0 = 0.0, loc_dx = 1.0, loc_dy = 1.0;
    std::vector<int64_t> loc_ptr, loc_ids;
    // per-shot sources of the batched path
    int32_t n_shot_src = 0;
    int32_t* d_shot_src_dom = nullptr;
    int32_t* d_shot_src_q = nullptr;
    double* d_shot_src_g = nullptr;
    float* d_shot_src_g32 = nullptr;
    double shot_f0 = 0.0, shot_t0 = 0.0, shot_amp = 0.0;
    float* d_src_g32 = nullptr;
    f2x* d_src_gx = nullptr;
    f2x* d_shot_src_gx = nullptr;
    // arithmetic of the single-shot stepping entry points (HHO_F64 or HHO_F32X2)
    int32_t arith = HHO_F64;
    // launch mode of the ERK loops and the captured steps (stage.cu)
    int32_t launch_mode = HHO_LAUNCH_AUTO;
    StageClock* d_clock = nullptr;
    void* cap_stream = nullptr;                      // cudaStream_t used for capture
    struct StepGraph {
        std::vector<unsigned char> key;              // byte image of the step's kernel arguments
        void* exec = nullptr;                        // cudaGraphExec_t
    };
    std::vector<StepGraph> graphs;
    // sampled source time functions (hho_sources_set_samples): the value of
    // source s at step n, stage j is src_samples[(s samp_n + n) samp_s + j]
    bool src_sampled = false;
    std::vector<double> src_samples;
    double samp_t0 = 0.0, samp_dt = 0.0;
    int64_t samp_n = 0;
    int32_t samp_s = 0;
    // sources
    int32_t n_src = 0;
    int32_t src_dom[MAX_SOURCES], src_q[MAX_SOURCES];
    double src_f0[MAX_SOURCES], src_t0[MAX_SOURCES], src_amp[MAX_SOURCES];
    double* d_src_g = nullptr;
    // receivers
    int32_t n_rec = 0;
    int32_t* d_rec_int = nullptr;
    double* d_rec_dbl = nullptr;
    // transpose of recording (adjoint): the cells the receivers read, each with
    // its receivers in increasing order.  One int block:
    // [ptr: n_inj + 1][cell: 2 n_inj (domain, position)][receiver ids]
    int32_t n_inj = 0;
    int32_t* d_inj = nullptr;
    // energy
    double* d_mass_f = nullptr;   // per fluid cell: rho h^2, h^2/kappa
    double* d_mass_s = nullptr;   // per solid cell: h^2 * compliance (3), rho h^2
    // host-buffer entry point scratch
    double* d_host_state = nullptr;
    double* d_host_canon = nullptr;
    double* d_host_work = nullptr;
    int64_t host_work_size = 0;
    HostPieces host_pieces;
    HostPipe* host_pipe = nullptr;   // the copy stream and events of a call in pieces (stage.cu)
    int64_t n_state = 0;
    int64_t trace_doubles = 0;    // one trace buffer (fluid + solid parts)
    // tensor-core batched stage (HHO_BF16X3): per class the split-BF16
    // operand tiles of its two GEMMs (all faces' lifts, all faces' traces),
    // see tc_tiles in operators.cpp; meta [n_classes][6] = K1, N1, K2, N2,
    // offset of the class's tiles (16-byte units), tile bytes
    void* d_tc_b = nullptr;
    int32_t* d_tc_meta = nullptr;
    int32_t tc_kmax = 0;          // widest A tile (K) over the classes
    int64_t tc_bmax = 0;          // largest tile bytes of one class
    uint32_t tc_cols = 32;        // tensor-memory columns a block allocates
    int32_t* d_tc_err = nullptr;  // set by a tensor-core block whose MMA wait gave up
    bool tc_on = false;           // the current batched call runs the tensor-core stage
    // adjoint support: interface coefficients of the operator with the
    // coupling sign reversed, and per-class M0^-1 (n x n each)
    double* d_if_coef_adj = nullptr;
    float* d_if_coef_adj_f32 = nullptr;   // its FP32 copy (the FP32 adjoint)
    double* d_cls_minv = nullptr;
    // host copies for the cost model and the SDIRK preconditioner's colouring
    std::vector<double> h_cls_dbl;
    std::vector<int32_t> h_cls_int, h_nb_f, h_nb_s, h_if_nb;
    // SDIRK block-Jacobi preconditioner: (I - a* dt J_TT)^-1 of every cell,
    // entry (r, c) of a fluid cell q at d_bj[(r 3n + c) Nf + q], of a solid
    // cell at d_bj[9n^2 Nf + (r 5n + c) Ns + q], built for a* dt = bj_adt
    int32_t sdirk_precond = 1;
    double* d_bj = nullptr;
    double bj_adt = 0.0;
    int32_t* d_bj_colour = nullptr;   // cell colouring, fluid then solid slots
    int32_t bj_colours = 0;
    double* h_krylov = nullptr;       // pinned: a Krylov vector's sums and the combination's coefficients
    void* krylov_event = nullptr;     // cudaEvent_t: those sums have arrived
    // stage-kernel timing (hho_profile_*)
    bool prof_on = false;
    int32_t prof_n = 0;
    std::vector<void*> prof_events;   // cudaEvent_t pairs
};
