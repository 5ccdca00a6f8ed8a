// Internal declarations of the GB300 reservoir library (not part of the ABI).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>
#include <string>
#include <vector>

#include "../../include/sim.h"
#include "per_device.h"

#include <nvtx3/nvToolsExt.h>

// NVTX range over a host scope (a phase of a step); no cost unless a tool such
// as a profiler attaches to NVTX
struct NvtxRange {
    explicit NvtxRange(const char *name) { nvtxRangePushA(name); }
    ~NvtxRange() { nvtxRangePop(); }
    NvtxRange(const NvtxRange &) = delete;
    NvtxRange &operator=(const NvtxRange &) = delete;
};

#define SIM_GRAV 9.80665
#define SIM_DARCY (86400.0 * 9.869233e-16 * 1e5 / 1e-3)
#define SIM_MAX_PVT 64
#define SIM_MAX_M 32
#define SIM_MAX_ELL 512      // widest coarse AMG row: a wider Galerkin row stops coarsening
#define SIM_RED_BLOCKS 456   // 3 x 152 SMs: grid of the state's reductions (CNV, masses, finiteness)
#define SIM_THREADS 256
#define SIM_SETUP_SCALARS 16 // ints the set-up reads back: counts and flags, then 64-bit entry counts of the levels
#define SIM_SETUP_LEVELS 80  // a level has at most three quarters of the rows above it: 68 levels at 2^28 cells

// Reductions of the Krylov solvers over n entries: threads of a block that stream
// and the blocks of the grid.  One block per SM: the kernels are bound by the FP64
// pipe, which 8 warps keep busy, and every further block adds its own reduction and
// 8 bytes a value for the last block to fold (600k entries, 16 vectors: dots 27 us,
// update-and-dots 42 us; with two blocks per SM 31 and 46, with three 34 and 52).
// From 2M entries the loads in flight count more than that (12M entries, 16 vectors:
// dots 376 us, norm 347 us with two blocks per SM, 433 and 445 with one).
constexpr int kRedThreads = 256;
inline int sim_red_blocks(long n) {
    const long want = (n + kRedThreads - 1) / kRedThreads, most = n >= (1L << 21) ? 304 : 152;
    return (int)(want < 1 ? 1 : want < most ? want : most);
}
// blocks of SIM_THREADS of an elementwise pass over n entries: up to one full wave
inline int sim_stream_blocks(long n) {
    const long want = (n + SIM_THREADS - 1) / SIM_THREADS;
    return (int)(want < 1 ? 1 : want < 1216 ? want : 1216);
}

// fluid and rock constants, passed by value as a kernel parameter, so handles never
// share state; the PVT table is the handle's device array of npvt - 1 interval rows
// (p, then value and slope of Bo, Rs, mu_o, Bg, mu_g), its slopes divided once on
// the host
constexpr int SIM_PVT_ROW = 11;
struct FluidConst {
    int model, b, npvt;
    double rho_w_ref, rho_o_ref, c_w, c_o;
    double rho_ws, rho_os, rho_gs, bw_c, bw_pref, bo_c_us, muo_c_us;
    double swc, sor, sgc, sorg, nw, now, ng, nog;
    double c_rock, p_ref;
    // reciprocals: 1 / mu_w, 1 / mu_o, 1 / (1 - swc - sor), 1 / (1 - swc - sorg - sgc), 1 / (1 - swc - sorg)
    double i_muw, i_muo, i_mob, i_mobg, i_mobog;
    const double *pvt;
    double cnv_rho[3];
};

struct GridDesc {
    int nx, ny, nz, N;
    double dx, dy, dz, top;
    int H;              // cells of one colour in the colour-split arrays: ceil(nx / 2) ny nz
};

// device control block of one FGMRES solve (Givens, Hessenberg, flags)
struct KrylovCtl {
    int done;           // 1 once the Arnoldi residual estimate met the tolerance
    int k;              // inner iterations completed in the current cycle
    int active;         // batched solves: 1 while this member's solve goes on
    int iters;          // batched solves: inner iterations of this member's solve
    double tol, beta, rnorm2;
    double h[SIM_MAX_M + 1], h2[SIM_MAX_M + 1];
    double g[SIM_MAX_M + 1], cs[SIM_MAX_M + 1], sn[SIM_MAX_M + 1], y[SIM_MAX_M + 1];
    double H[(SIM_MAX_M + 1) * (SIM_MAX_M + 1)];
    unsigned int counter;   // last-block reduction ticket
    unsigned int pad2;
};

// One member of a batched FGMRES solve (an ensemble of independent systems):
// its operands, read by the batched kernels from a device table
struct KMember {
    GridDesc g;
    long n;                  // b N
    double theta;            // relative tolerance of this member's solve
    const double *J;
    double *V, *w, *r, *x;   // Krylov basis, work vector, residual, solution
    const double *rhs;       // right-hand side; null: the member does not solve in this round
    void *Z;                 // preconditioned directions (FP64 or FP32)
    KrylovCtl *ctl;
    double *red;             // the member's reduction partials and ticket
    unsigned int *ticket;
    int nred;                // virtual blocks of its reductions (sim_red_blocks(n))
};

// BiCGSTAB scalars (device); flag: 1 recursive residual met the tolerance,
// 2 breakdown, 3 iteration limit (each also sets done)
struct BicgCtl {
    int done, flag, it, half_j;
    int fresh, max_it;
    double tol, rho, rho_old, alpha, omega, rnorm;
};

struct AmgLevel {
    int n = 0, width = 0;        // level 0: width 7, structured
    double entries = 0.0;        // sum of the row lengths (level 0: 7 n)
    int *len = nullptr;          // entries of each row (levels >= 1)
    int *col = nullptr;          // ELL columns [width][n], -1 padding (behind len in its allocation)
    int *colA = nullptr;         // the same with padding on the row's own column (apply)
    double *val = nullptr;       // ELL values, FP64 (setup precision)
    void *valT = nullptr;        // ELL values in apply precision (float copy for mixed)
    void *dinvT = nullptr;       // 1 / l1 row sums, apply precision
    int *agg = nullptr;          // fine -> next level
    int *moff = nullptr, *mem = nullptr;   // members of each next-level aggregate, ascending (CSR)
    void *f = nullptr, *e = nullptr, *e2 = nullptr;   // V-cycle vectors (apply precision)
    void *coarse_inv = nullptr;  // coarsest: dense inverse, row-major n*n (FP64 in both forms)
    void *work = nullptr;        // the allocation dinvT, f, e, e2, colA and an FP32 valT lie in
};

struct sim {
    cudaStream_t stream = nullptr;
    bool own_stream = false;
    sim_status err = SIM_OK;
    std::string msg;
    FluidConst fc;
    GridDesc gd;
    sim_options opt;
    int N = 0, b = 0;
    int64_t launches = 0, newton_total = 0, linear_total = 0;
    size_t bytes = 0;
    // run totals for the run report: time steps (completed / failed), accepted
    // substeps, cuts, linear solves that hit their limit, simulated days, and the
    // per-phase device time and algorithmic bytes summed over every Newton call
    int64_t run_steps = 0, run_failed_steps = 0, run_substeps = 0, run_cuts = 0, run_lin_failures = 0;
    double run_days = 0.0, run_max_mb = 0.0;
    sim_phase_info run_phase = {};
    double m_start[3] = {0.0, 0.0, 0.0};   // component masses of the current step's start
    double last_mb = 0.0;                   // mass-balance error of the last accepted substep
    std::vector<void *> allocs;

    // geometry
    double *T = nullptr;         // [3][N] transmissibility to the + neighbour
    double *poro = nullptr;      // [N] porosity at p_ref
    int nperf = 0;
    int *perf_cell = nullptr, *perf_type = nullptr;
    double *perf_wi = nullptr, *perf_zh = nullptr;
    // wells (Eq. 16): perforations are grouped by well, woff[w]..woff[w+1]
    int nwells = 0, nrate = 0;
    int *perf_well = nullptr, *woff = nullptr, *wctrl = nullptr;
    double *wrate = nullptr;                 // [nwells] target of rate controls
    double *wbhp_c = nullptr;                // [nwells] BHP of BHP controls
    double *wp = nullptr, *wp_old = nullptr; // [nwells] bottom-hole pressures (unknowns under rate control)
    double *apw = nullptr, *awp = nullptr;   // [3][nperf] border blocks dR_cell/dp_h, dR_w/dx_cell
    double *aww = nullptr, *rw = nullptr;    // [nwells] dR_w/dp_h, well equation residual
    double *qwell = nullptr;                 // [3][nwells] component rates per well
    double *qperf = nullptr;                 // [4][nperf] component rates and the controlled rate per perforation
    double *wcnv = nullptr;                  // device scalar: largest |R_w| / max(|target|, 1)
    int *cell_perf = nullptr;                // [N] perforation of a rate-controlled well, or -1 (rate wells only)
    std::vector<int> h_wctrl;

    // state
    double *x = nullptr, *x_old = nullptr;   // [b][N]
    int8_t *ph = nullptr, *ph_old = nullptr;
    double *mold = nullptr;                  // [b][N]
    double *R = nullptr, *J = nullptr;       // [b][N], [7][b][b][N]
    double *props = nullptr;                 // [10 (b = 2) or 21][N] densities and mobilities (assemble.cu);
                                             // between assemblies the AMG set-up's integer scratch
    double *qtot = nullptr;                  // [3] well rates of the last assembly
    double cum_well[3] = {0, 0, 0};

    // reductions
    double *red = nullptr;       // partial sums [SIM_MAX_M+2][blocks of the reduction]
    double *scal = nullptr;      // small device scalars
    unsigned int *ticket = nullptr;
    double *h_pinned = nullptr;  // pinned host mirror for small reads
    cudaEvent_t pev[5] = {nullptr, nullptr, nullptr, nullptr, nullptr};   // phase marks of a Newton iteration

    // Krylov
    int m = 0;
    double *V = nullptr;         // [(m+1)][n]
    void *Z = nullptr;           // [m][n], FP64 or FP32
    double *w = nullptr, *r = nullptr, *xl = nullptr, *bl = nullptr, *dx = nullptr;
    KrylovCtl *ctl = nullptr;
    KrylovCtl *ctl_host = nullptr;
    cudaGraphExec_t cycle_exec = nullptr;   // captured restart cycle
    int64_t setup_gen = 0, cycle_gen = -1, graph_nodes = 0;
    int cycle_learned = -1;                  // learned-stage state the graph was captured with
    int tune_spmv = SIM_THREADS, tune_amg = 128, tune_stage = 64;   // block sizes picked by sim_autotune
    int last_cycle_k = 0;                    // inner iterations of the last restart cycle
    // BiCGSTAB: control block and the graph of one chunk of iterations
    BicgCtl *bctl = nullptr, *bctl_host = nullptr;
    cudaGraphExec_t bicg_exec = nullptr;
    int64_t bicg_gen = -1, bicg_nodes = 0;
    const double *bicg_x = nullptr;          // solution vector the chunk graph was captured with
    // inexact Newton: forcing term of the next solve, last linear residual b - J dx
    double theta = 0.0;
    double *rlin = nullptr;

    // CPR
    bool precond_ready = false;
    double *qiw = nullptr;       // [b][N]
    void *qiwT = nullptr;        // [b][N] apply precision (aliases qiw in FP64 mode)
    double *ap = nullptr;        // [7][N] pressure block, FP64
    void *apT = nullptr;         // [7][N] apply precision (aliases ap in FP64 mode)
    void *ahat = nullptr;        // [7][b][b][N] decoupled matrix, apply precision
    void *dinv = nullptr;        // [b][b][N] ILU / block-Jacobi inverse diagonal blocks
    double *dinv_d = nullptr;    // FP64 scratch of the same
    void *r2 = nullptr;          // [b][N] stage-2 work vector (apply precision)
    void *rpT = nullptr, *epacc = nullptr;   // [N] stage-P residual and accumulated correction
    // learned pressure stage (extra CPR stage after the V-cycles)
    sim_net_t *net = nullptr;
    int learned_on = 0;          // requested
    int learned_active = 0;      // used by the current solve (falls back to 0)
    int64_t learned_fallbacks = 0;
    float *lfeat = nullptr;      // [N][3] standardised log transmissibility features
    float *lx = nullptr, *ly = nullptr;   // [N][4] network input, [N] output
    void *lres = nullptr;        // [N] pressure residual after stage P (apply precision)
    void *lep = nullptr;         // [N] pressure correction after the learned stage
    double *lrms = nullptr;      // device scalar
    void *zr = nullptr;          // [b][N]
    double *lsc = nullptr;       // [b][b][N] per-cell left scaling L (quasi-IMPES or ABF)
    void *lscT = nullptr;        // [b][b][N] apply precision (aliases lsc in FP64 mode)
    void *rhT = nullptr, *x0 = nullptr;   // [b][N] CPR-FPF: L r - Ahat x0 and the first stage-F result
    std::vector<AmgLevel> lev;
    // AMG setup scratch (all but scan and iscal lie in props)
    int *partner = nullptr, *pick = nullptr, *pick2 = nullptr, *host = nullptr, *cnt = nullptr, *absorbed = nullptr;
    int *aggA = nullptr, *moffA = nullptr, *memA = nullptr, *aggB = nullptr, *moffB = nullptr, *memB = nullptr;
    int *scan = nullptr, *iscal = nullptr;
};

// ---- error helpers --------------------------------------------------------
sim_status sim_fail(sim_t *s, sim_status st, const std::string &m);
bool sim_cuda_ok(sim_t *s, cudaError_t e, const char *what);
#define SIM_CK(s, call) do { if (!sim_cuda_ok((s), (call), #call)) return (s)->err; } while (0)
#define SIM_LAUNCHED(s) do { (s)->launches++; if (!sim_cuda_ok((s), cudaGetLastError(), "kernel launch")) return (s)->err; } while (0)
void *sim_alloc(sim_t *s, size_t bytes);
void sim_free(sim_t *s, void *p);
inline int sim_blocks(long n, int t = SIM_THREADS) { long b = (n + t - 1) / t; return (int)(b < 1 ? 1 : b); }
bool sim_mixed(const sim_t *s);
// the current device, for PerDevice (outside its range when there is none)
inline int sim_device() { int d = -1; return cudaGetDevice(&d) == cudaSuccess ? d : -1; }

// ---- launches that overlap the drain of the one before --------------------------
// A CPR application is a chain of 4 to 45 launches of 2 to 60 us; between two plain
// launches of a stream the chip idles while the last blocks leave and the next grid is
// set up.  sim_launch() starts a kernel as soon as every block of the stream's previous
// kernel has passed sim_enter() and there is room for it; its own sim_enter() then waits
// until that kernel has completed and its writes are visible.  Every kernel launched
// this way calls sim_enter() before it touches anything another launch writes, and
// before any early return: a completed kernel then stands for all before it.
// An application at 400k two-phase cells 200 -> 161 us, at 1M three-phase cells (two
// V-cycles) 603 -> 522 us.
//   In a captured cycle, whose kernels follow each other sooner (about 1 us), the blocks
// that come early cost something too: they fill the SMs that drain first, and a grid of
// less than a wave is then spread unevenly.  With little work per SM (up to 65,536
// threads) latency decides and the overlap pays; beyond a wave (152 x 2,048 threads) the
// rest of the grid evens out; between the two the launch stays plain.  An FGMRES iteration
// in us, no launch overlapped / this rule / every one: two-phase 32k cells 88.6 / 86.3 /
// 86.3, 66k 141.3 / 135.8 / 136.0, 84k 157.7 / 147.7 / 145.6, 151k 207.8 / 199.3 / 210.0;
// three-phase 98k 211.6 / 201.3 / 201.7, 150k 252.9 / 245.0 / 266.0, 200k 275.2 / 271.7 /
// 287.3, 240k 308.8 / 305.9 / 313.9, 312k 362.0 / 357.0 / 361.2, 336k 379.5 / 375.2 / 375.9,
// 520k 515.9 / 505.4 / 502.9.
__device__ __forceinline__ void sim_enter() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
inline bool sim_overlaps(long threads, cudaStream_t st) {
    if (threads <= 65536 || threads > 152L * 2048) return true;
    cudaStreamCaptureStatus c;
    return cudaStreamIsCapturing(st, &c) == cudaSuccess && c == cudaStreamCaptureStatusNone;
}
// launch errors are left for cudaGetLastError, as by <<<>>>
template <typename... P, typename... A>
inline void sim_launch(void (*kernel)(P...), long blocks, int threads, cudaStream_t st, A... args) {
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.gridDim = dim3((unsigned)blocks); cfg.blockDim = dim3((unsigned)threads); cfg.stream = st;
    cfg.attrs = at; cfg.numAttrs = sim_overlaps(blocks * threads, st) ? 1 : 0;
    (void)cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

// ---- assemble.cu ----------------------------------------------------------
sim_status k_geometry(sim_t *s, const double *kx, const double *ky, const double *kz, const double *poro,
                      const int *wcell_host, const int *wtype_host, const int *pwell_host,
                      const double *wzh_host, const double *wrw_host, const double *wskin_host);
sim_status k_well_rhs(sim_t *s, double *b);                          // b += A_pw A_ww^-1 R_w
sim_status k_well_update(sim_t *s, const double *dx);                // p_h += dp_h (rate wells)
template <typename X> sim_status k_well_op(sim_t *s, const X *x, double *y, const int *done);   // y -= A_pw A_ww^-1 A_wp x
sim_status k_accumulation(sim_t *s, const double *x, const int8_t *ph, double *acc);   // acc [b][N]
sim_status k_assemble(sim_t *s, double dt);
sim_status k_cnv(sim_t *s, double dt, double *cnv_host, double *well_cnv_host = nullptr);
sim_status k_component_mass(sim_t *s, double *m3_host);
sim_status k_newton_update(sim_t *s, const double *dx);
sim_status k_finite(sim_t *s, const double *v, long n, int *ok_host);

// ---- sim_api.cu: the pieces of a Newton iteration (ensemble runtime) --------
sim_status nl_assemble_test(sim_t *s, double dt, int *state, sim_phase_info *ph);   // 0 solve, 1 converged, 2 non-finite
sim_status nl_prepare_solve(sim_t *s, sim_phase_info *ph);
sim_status nl_finish_solve(sim_t *s, const sim_linear_info &li, bool *finite_ok, sim_phase_info *ph);
sim_status nl_restore(sim_t *s);
sim_status accept_step(sim_t *s, double dt);
// a finished time step (sim_step or one member of a batch step) into the run totals
void run_record_step(sim_t *s, const sim_step_info &si, sim_status st);

// ---- krylov.cu ------------------------------------------------------------
sim_status k_spmv(sim_t *s, const double *x, double *y);                 // y = J x
sim_status k_spmv_f(sim_t *s, const float *x, double *y);
sim_status k_fgmres(sim_t *s, const double *b, double *x, sim_linear_info *info);
sim_status k_bicgstab(sim_t *s, const double *b, double *x, sim_linear_info *info);
sim_status k_linear_solve(sim_t *s, const double *b, double *x, sim_linear_info *info);
sim_status k_diff_norm2(sim_t *s, const double *a, const double *b, long n, double *out);
sim_status k_norm2(sim_t *s, const double *v, long n, double *out_host);
sim_status k_spmv_block(sim_t *s, const double *x, double *y, int block);
// FGMRES batched over ensemble members: every Krylov operation one launch for all
struct KrylovBatch;
KrylovBatch *k_batch_new();
void k_batch_free(KrylovBatch *kb);
int64_t k_batch_launches(const KrylovBatch *kb);
sim_status k_fgmres_batch(KrylovBatch *kb, sim_t *const *ms, int nm, cudaStream_t st, sim_linear_info *infos,
                          std::string *err);
sim_status k_orth_step(sim_t *s, int nv);              // measurement: one Arnoldi orthogonalisation step
double k_orth_step_bytes(const sim_t *s, int nv);      // its algorithmic bytes

// ---- cpr.cu ---------------------------------------------------------------
sim_status cpr_setup(sim_t *s);
sim_status cpr_apply(sim_t *s, const double *r, void *z, const int *done);   // z FP64 or FP32 (Z type)
void cpr_free(sim_t *s);
// batched CPR application over ensemble members (tables and work lists)
struct CprBatch;
bool cpr_batchable(sim_t *const *ms, int nm);
CprBatch *cpr_batch_new();
void cpr_batch_free(CprBatch *cb);
cudaError_t cpr_batch_build(CprBatch *cb, sim_t *const *ms, int nm, cudaStream_t st);   // after every member's setup
int cpr_batch_apply(const CprBatch *cb, cudaStream_t st, int j);                         // launches, or -1
sim_status cpr_copy_level_ell(sim_t *s, int level, int *col, double *val);
sim_status cpr_learned_pairs(sim_t *s, int k, float *x_dev, float *y_dev);
sim_status cpr_learned_features(sim_t *s);

// ---- learned.cu -----------------------------------------------------------
sim_status net_infer(sim_net_t *n, const float *x_dev, float *y_dev, cudaStream_t st, const int *done);
int64_t net_launches(sim_net_t *n);
// the convolutions' status word after the stream has drained: 0 fine, > 0 a
// bounded wait gave up, < 0 the read itself failed
int net_status_word(sim_net_t *n, cudaStream_t st);
int net_cells(sim_net_t *n);
