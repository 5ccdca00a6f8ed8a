// C ABI of the GB300 reservoir Newton step (declarations and contracts in
// include/sim.h).  Host orchestration only: every arithmetic step of the
// method runs in the kernels of assemble.cu, krylov.cu and cpr.cu.
#include <cmath>
#include <cstdio>
#include <cstring>
#include <set>

#include <algorithm>

#include "sim_internal.cuh"

static thread_local std::string g_create_error;

sim_status sim_fail(sim_t *s, sim_status st, const std::string &m) {
    if (!s) { g_create_error = m; return st; }
    if (s->err == SIM_OK) { s->err = st; s->msg = m; }
    return s->err;
}

bool sim_cuda_ok(sim_t *s, cudaError_t e, const char *what) {
    if (e == cudaSuccess) return true;
    std::string m = std::string(what) + ": " + cudaGetErrorString(e);
    sim_fail(s, e == cudaErrorMemoryAllocation ? SIM_ENOMEM : SIM_ECUDA, m);
    return false;
}

void *sim_alloc(sim_t *s, size_t bytes) {
    void *p = nullptr;
    cudaError_t e = cudaMalloc(&p, bytes ? bytes : 16);
    if (e != cudaSuccess) {
        sim_fail(s, SIM_ENOMEM, std::string("cudaMalloc of ") + std::to_string(bytes) + " bytes: " + cudaGetErrorString(e));
        return nullptr;
    }
    s->allocs.push_back(p);
    s->bytes += bytes;
    return p;
}

void sim_free(sim_t *s, void *p) {
    for (size_t k = 0; k < s->allocs.size(); k++)
        if (s->allocs[k] == p) { s->allocs.erase(s->allocs.begin() + k); break; }
    cudaFree(p);
}

namespace {
// NC independent FMA chains per thread, no memory traffic except one store
// per thread; each chain has its own multiplier so no two chains share all
// their operands
__device__ __forceinline__ unsigned long long global_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
// stamps (when not null): per block, SM clock cycles and global-timer
// nanoseconds between the first thread's start and end of the loop
template <typename T, int NC>
__global__ void fma_probe_kernel(T *out, int iters, long long *stamps = nullptr) {
    long long c0 = 0;
    unsigned long long n0 = 0;
    if (stamps && threadIdx.x == 0) { c0 = clock64(); n0 = global_ns(); }
    T a[NC], m[NC];
#pragma unroll
    for (int c = 0; c < NC; c++) { a[c] = threadIdx.x * (T)1e-3 + (T)c; m[c] = (T)0.9999999 - (T)c * (T)1e-9; }
    const T k = (T)1e-7;
    for (int i = 0; i < iters; i++) {
#pragma unroll
        for (int c = 0; c < NC; c++) a[c] = fma(a[c], m[c], k);
    }
    T t = 0;
#pragma unroll
    for (int c = 0; c < NC; c++) t += a[c];
    out[blockIdx.x * blockDim.x + threadIdx.x] = t;
    if (stamps && threadIdx.x == 0) {
        stamps[2 * blockIdx.x] = clock64() - c0;
        stamps[2 * blockIdx.x + 1] = (long long)(global_ns() - n0);
    }
}
// FMA rate of one launch shape: iters x NC FMAs per thread over the grid
template <typename T, int NC>
static double probe_rate(T *buf, int blocks, int threads, int iters, long long *stamps = nullptr) {
    cudaEvent_t e0, e1;
    cudaEventCreate(&e0); cudaEventCreate(&e1);
    fma_probe_kernel<T, NC><<<blocks, threads>>>(buf, 16);
    cudaEventRecord(e0);
    fma_probe_kernel<T, NC><<<blocks, threads>>>(buf, iters, stamps);
    cudaEventRecord(e1);
    cudaEventSynchronize(e1);
    float ms = 0.f;
    cudaEventElapsedTime(&ms, e0, e1);
    cudaEventDestroy(e0); cudaEventDestroy(e1);
    return ms > 0.f ? (double)blocks * threads * iters * NC / (ms * 1e-3) : 0.0;
}

__global__ void widen_kernel(const float *__restrict__ a, double *__restrict__ b, long n) {
    for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x) b[i] = (double)a[i];
}
__global__ void negate_kernel(const double *__restrict__ a, double *__restrict__ b, long n) {
    for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x) b[i] = -a[i];
}
}  // namespace

// time `reps` launches of f on the handle's stream (milliseconds per launch)
template <typename F>
static float time_launches(sim_t *s, int reps, F f) {
    cudaEvent_t e0, e1;
    cudaEventCreate(&e0); cudaEventCreate(&e1);
    f();
    cudaEventRecord(e0, s->stream);
    for (int r = 0; r < reps; r++) f();
    cudaEventRecord(e1, s->stream);
    cudaEventSynchronize(e1);
    float ms = 0.f;
    cudaEventElapsedTime(&ms, e0, e1);
    cudaEventDestroy(e0); cudaEventDestroy(e1);
    return ms / reps;
}

#define CHECK_HANDLE(s) do { if (!(s)) return SIM_EINVAL; if ((s)->err != SIM_OK) return (s)->err; } while (0)

extern "C" {

const char *sim_last_error(sim_t *s) { return s ? s->msg.c_str() : g_create_error.c_str(); }
void sim_clear_error(sim_t *s) { if (s) { s->err = SIM_OK; s->msg.clear(); } }
int32_t sim_block_size(sim_t *s) { return s ? s->b : 0; }

void sim_destroy(sim_t *s) {
    if (!s) return;
    if (s->stream) cudaStreamSynchronize(s->stream);
    cpr_free(s);
    if (s->stream) cudaStreamSynchronize(s->stream);
    if (s->cycle_exec) cudaGraphExecDestroy(s->cycle_exec);
    if (s->bicg_exec) cudaGraphExecDestroy(s->bicg_exec);
    for (void *p : s->allocs) cudaFree(p);
    if (s->h_pinned) cudaFreeHost(s->h_pinned);
    for (cudaEvent_t &e : s->pev) if (e) cudaEventDestroy(e);
    if (s->ctl_host) cudaFreeHost(s->ctl_host);
    if (s->bctl_host) cudaFreeHost(s->bctl_host);
    if (s->own_stream && s->stream) cudaStreamDestroy(s->stream);
    delete s;
}

sim_status sim_create(const sim_grid *g, const sim_rock *r, const sim_fluid *f, const sim_well *w, int32_t nwells,
                      const sim_options *o, void *cuda_stream, sim_t **out) {
    if (!out) return sim_fail(nullptr, SIM_EINVAL, "out is NULL");
    *out = nullptr;
    if (!g || !r || !f || !o || (nwells > 0 && !w)) return sim_fail(nullptr, SIM_EINVAL, "NULL argument");
    if (g->nx < 1 || g->ny < 1 || g->nz < 1 || (long)g->nx * g->ny * g->nz > 0x7fffffffL / 8)
        return sim_fail(nullptr, SIM_EINVAL, "grid dimensions out of range");
    if (!(g->dx > 0 && g->dy > 0 && g->dz > 0)) return sim_fail(nullptr, SIM_EINVAL, "cell sizes must be positive");
    if (f->model != 2 && f->model != 3) return sim_fail(nullptr, SIM_EINVAL, "fluid model must be 2 or 3");
    if (!r->kx || !r->ky || !r->kz || !r->poro) return sim_fail(nullptr, SIM_EINVAL, "rock arrays missing");
    if (o->gmres_m < 1 || o->gmres_m > SIM_MAX_M) return sim_fail(nullptr, SIM_EINVAL, "gmres_m must be in 1..32");
    if (o->precond < 0 || o->precond > 2 || o->stage2 < 0 || o->stage2 > 1 || o->precision < 0 || o->precision > 1)
        return sim_fail(nullptr, SIM_EINVAL, "bad preconditioner options");
    if (o->amg_coarse_max < 1 || o->amg_coarse_max > 1024 || o->amg_rounds < 1 || o->amg_max_levels < 1 ||
        o->amg_cycles < 1 || o->amg_cycles > 16)
        return sim_fail(nullptr, SIM_EINVAL, "bad AMG options");
    if (o->decouple < 0 || o->decouple > 1 || (o->cpr_stages != 2 && o->cpr_stages != 3))
        return sim_fail(nullptr, SIM_EINVAL, "bad CPR decoupling / stage options");
    if (o->krylov < 0 || o->krylov > 1 || o->lin_max_iter < 1 || o->forcing < 0 || o->forcing > 3 ||
        !(o->lin_tol > 0 && o->lin_tol < 1) || !(o->theta_max >= o->lin_tol && o->theta_max < 1) ||
        !(o->ew_gamma > 0 && o->ew_gamma <= 1) || !(o->ew_beta > 0))
        return sim_fail(nullptr, SIM_EINVAL, "bad Krylov / forcing-term options");
    if (o->orth < 0 || o->orth > 1) return sim_fail(nullptr, SIM_EINVAL, "orth must be 0 or 1");
    if (o->krylov == SIM_KRYLOV_BICGSTAB && o->gmres_m < 2)
        return sim_fail(nullptr, SIM_EINVAL, "BiCGSTAB needs gmres_m >= 2 (its two preconditioned vectors)");
    if (f->model == 3) {
        if (f->npvt < 2 || f->npvt > SIM_MAX_PVT) return sim_fail(nullptr, SIM_EINVAL, "npvt must be in 2..64");
        if (!f->pvt_p || !f->pvt_bo || !f->pvt_rs || !f->pvt_muo || !f->pvt_bg || !f->pvt_mug)
            return sim_fail(nullptr, SIM_EINVAL, "PVT table missing");
        for (int k = 0; k + 1 < f->npvt; k++)
            if (!(f->pvt_p[k + 1] > f->pvt_p[k])) return sim_fail(nullptr, SIM_EINVAL, "PVT pressures must increase");
    }
    const long N = (long)g->nx * g->ny * g->nz;
    for (long i = 0; i < N; i++)
        if (!(r->kx[i] > 0 && r->ky[i] > 0 && r->kz[i] > 0 && r->poro[i] > 0 && std::isfinite(r->kx[i]) &&
              std::isfinite(r->poro[i])))
            return sim_fail(nullptr, SIM_EINVAL, "permeability and porosity must be positive and finite");
    // perforations: distinct cells
    std::vector<int> pc, pt, pw, woff(1, 0), wctrl;
    std::vector<double> pz, prw, pskin, wrate, wbhp;
    std::set<int> seen;
    int nrate = 0;
    for (int k = 0; k < nwells; k++) {
        const sim_well &W = w[k];
        if (W.i < 0 || W.i >= g->nx || W.j < 0 || W.j >= g->ny || W.k_top < 0 || W.k_bot >= g->nz || W.k_top > W.k_bot)
            return sim_fail(nullptr, SIM_EINVAL, "well " + std::to_string(k) + " outside the grid");
        if (W.type != SIM_WELL_PRODUCER && W.type != SIM_WELL_WATER_INJECTOR)
            return sim_fail(nullptr, SIM_EINVAL, "unknown well type");
        if (!(W.r_w > 0)) return sim_fail(nullptr, SIM_EINVAL, "well radius must be positive");
        if (W.control < SIM_WELL_BHP || W.control > SIM_WELL_OIL_RATE ||
            (W.type == SIM_WELL_WATER_INJECTOR && W.control == SIM_WELL_OIL_RATE) || !std::isfinite(W.rate) ||
            !std::isfinite(W.bhp))
            return sim_fail(nullptr, SIM_EINVAL, "well " + std::to_string(k) + ": bad control");
        if (W.control != SIM_WELL_BHP) nrate++;
        const double zh = g->top_depth + (W.k_top + 0.5) * g->dz;
        for (int kk = W.k_top; kk <= W.k_bot; kk++) {
            const int c = W.i + g->nx * (W.j + g->ny * kk);
            if (!seen.insert(c).second) return sim_fail(nullptr, SIM_EINVAL, "two perforations share a cell");
            pc.push_back(c); pt.push_back(W.type); pw.push_back(k); pz.push_back(zh);
            prw.push_back(W.r_w); pskin.push_back(W.skin);
        }
        woff.push_back((int)pc.size());
        wctrl.push_back(W.control); wrate.push_back(W.rate); wbhp.push_back(W.bhp);
    }

    sim_t *s = new sim_t();
    s->opt = *o;
    s->N = (int)N;
    s->b = f->model == 3 ? 3 : 2;
    s->m = o->gmres_m;
    s->gd.nx = g->nx; s->gd.ny = g->ny; s->gd.nz = g->nz; s->gd.N = (int)N;
    s->gd.dx = g->dx; s->gd.dy = g->dy; s->gd.dz = g->dz; s->gd.top = g->top_depth;
    s->gd.H = ((g->nx + 1) / 2) * g->ny * g->nz;
    FluidConst &c = s->fc;
    memset(&c, 0, sizeof(c));
    c.model = f->model; c.b = s->b; c.npvt = f->model == 3 ? f->npvt : 0;
    c.rho_w_ref = f->rho_w_ref; c.rho_o_ref = f->rho_o_ref; c.c_w = f->c_w; c.c_o = f->c_o;
    c.rho_ws = f->rho_ws; c.rho_os = f->rho_os; c.rho_gs = f->rho_gs; c.bw_c = f->bw_c; c.bw_pref = f->bw_pref;
    c.bo_c_us = f->bo_c_us; c.muo_c_us = f->muo_c_us;
    c.swc = f->swc; c.sor = f->sor; c.sgc = f->sgc; c.sorg = f->sorg; c.nw = f->nw; c.now = f->now; c.ng = f->ng; c.nog = f->nog;
    c.c_rock = r->c_rock; c.p_ref = r->p_ref;
    c.i_muw = 1.0 / f->mu_w; c.i_muo = 1.0 / f->mu_o; c.i_mob = 1.0 / (1.0 - f->swc - f->sor);
    c.i_mobg = 1.0 / (1.0 - f->swc - f->sorg - f->sgc); c.i_mobog = 1.0 / (1.0 - f->swc - f->sorg);
    std::vector<double> pvt;                 // interval rows: p, then value and slope per column
    for (int k = 0; k + 1 < c.npvt; k++) {
        const double *col[5] = {f->pvt_bo, f->pvt_rs, f->pvt_muo, f->pvt_bg, f->pvt_mug};
        pvt.push_back(f->pvt_p[k]);
        for (const double *v : col) {
            pvt.push_back(v[k]);
            pvt.push_back((v[k + 1] - v[k]) / (f->pvt_p[k + 1] - f->pvt_p[k]));
        }
    }
    for (int k = 0; k < 3; k++) c.cnv_rho[k] = f->cnv_rho[k] > 0 ? f->cnv_rho[k] : 1.0;

    if (cuda_stream) s->stream = (cudaStream_t)cuda_stream;
    else {
        if (cudaStreamCreateWithFlags(&s->stream, cudaStreamNonBlocking) != cudaSuccess) {
            delete s;
            return sim_fail(nullptr, SIM_ECUDA, "cannot create a CUDA stream (no GPU?)");
        }
        s->own_stream = true;
    }
    const int b = s->b;
    const long n = N * b;
    const bool mixed = o->precision == SIM_PRECISION_MIXED;
    const size_t tsz = mixed ? sizeof(float) : sizeof(double);
    bool ok = true;
    auto A = [&](size_t bytes) -> void * { void *p = ok ? sim_alloc(s, bytes) : nullptr; if (!p) ok = false; return p; };
    s->T = (double *)A(sizeof(double) * 3 * N);
    s->poro = (double *)A(sizeof(double) * N);
    s->nperf = (int)pc.size();
    s->perf_cell = (int *)A(sizeof(int) * (pc.size() + 1));
    s->perf_type = (int *)A(sizeof(int) * (pc.size() + 1));
    s->perf_wi = (double *)A(sizeof(double) * (pc.size() + 1));
    s->perf_zh = (double *)A(sizeof(double) * (pc.size() + 1));
    s->nwells = nwells;
    s->nrate = nrate;
    s->h_wctrl = wctrl;
    s->perf_well = (int *)A(sizeof(int) * (pc.size() + 1));
    s->woff = (int *)A(sizeof(int) * (nwells + 1));
    s->wctrl = (int *)A(sizeof(int) * (nwells + 1));
    s->wrate = (double *)A(sizeof(double) * (nwells + 1));
    s->wbhp_c = (double *)A(sizeof(double) * (nwells + 1));
    s->wp = (double *)A(sizeof(double) * (nwells + 1));
    s->wp_old = (double *)A(sizeof(double) * (nwells + 1));
    s->aww = (double *)A(sizeof(double) * (nwells + 1));
    s->rw = (double *)A(sizeof(double) * (nwells + 1));
    s->qwell = (double *)A(sizeof(double) * 3 * (nwells + 1));
    s->apw = (double *)A(sizeof(double) * 3 * (pc.size() + 1));
    s->awp = (double *)A(sizeof(double) * 3 * (pc.size() + 1));
    s->qperf = (double *)A(sizeof(double) * 4 * (pc.size() + 1));
    s->wcnv = (double *)A(sizeof(double));
    if (nrate > 0) s->cell_perf = (int *)A(sizeof(int) * N);
    s->x = (double *)A(sizeof(double) * n);
    s->x_old = (double *)A(sizeof(double) * n);
    s->ph = (int8_t *)A(N);
    s->ph_old = (int8_t *)A(N);
    s->mold = (double *)A(sizeof(double) * n);
    s->R = (double *)A(sizeof(double) * n);
    s->J = (double *)A(sizeof(double) * 7 * b * b * N);
    // the properties live from an assembly's first pass to its second; the integer scratch
    // of the AMG set-up (68 bytes a cell) shares their memory
    struct { int **p; size_t n; } scratch[] = {
        {&s->partner, (size_t)N}, {&s->pick, (size_t)N}, {&s->pick2, (size_t)N}, {&s->absorbed, 6 * (size_t)N},
        {&s->host, (size_t)N}, {&s->cnt, (size_t)N}, {&s->aggA, (size_t)N}, {&s->aggB, (size_t)N},
        {&s->moffA, (size_t)N + 1}, {&s->memA, (size_t)N}, {&s->moffB, (size_t)N + 1}, {&s->memB, (size_t)N}};
    size_t scratch_bytes = 0;
    for (auto &a : scratch) scratch_bytes += (sizeof(int) * a.n + 255) & ~(size_t)255;
    s->props = (double *)A(std::max(sizeof(double) * (b == 2 ? 10 : 21) * N, scratch_bytes));
    size_t at = 0;
    for (auto &a : scratch) {
        *a.p = ok ? (int *)((char *)s->props + at) : nullptr;
        at += (sizeof(int) * a.n + 255) & ~(size_t)255;
    }
    double *pvt_dev = (double *)A(sizeof(double) * (pvt.size() + 1));
    c.pvt = pvt_dev;
    s->qtot = (double *)A(sizeof(double) * 4);
    s->red = (double *)A(sizeof(double) * (SIM_MAX_M + 2) * SIM_RED_BLOCKS);
    s->scal = (double *)A(sizeof(double) * 64);
    s->ticket = (unsigned int *)A(sizeof(unsigned int) * 4);
    s->V = (double *)A(sizeof(double) * (s->m + 1 > 5 ? s->m + 1 : 5) * n);   // BiCGSTAB keeps 5 vectors here
    s->Z = A(tsz * s->m * n);
    s->w = (double *)A(sizeof(double) * n);
    s->r = (double *)A(sizeof(double) * n);
    s->xl = (double *)A(sizeof(double) * n);
    s->bl = (double *)A(sizeof(double) * n);
    s->dx = (double *)A(sizeof(double) * n);
    s->ctl = (KrylovCtl *)A(sizeof(KrylovCtl));
    s->bctl = (BicgCtl *)A(sizeof(BicgCtl));
    s->rlin = (double *)A(sizeof(double) * n);
    s->theta = o->lin_tol;
    s->qiw = (double *)A(sizeof(double) * n);
    s->ap = (double *)A(sizeof(double) * 7 * N);
    s->qiwT = mixed ? A(sizeof(float) * n) : (void *)s->qiw;
    s->apT = mixed ? A(sizeof(float) * 7 * N) : (void *)s->ap;
    const size_t NS = 2 * (size_t)s->gd.H;     // colour-split positions (>= N)
    s->ahat = A(tsz * 7 * b * b * NS);
    s->dinv_d = (double *)A(sizeof(double) * b * b * NS);
    s->dinv = mixed ? A(sizeof(float) * b * b * NS) : (void *)s->dinv_d;
    s->r2 = A(tsz * n);
    s->rpT = A(tsz * N);
    s->epacc = A(tsz * N);
    s->zr = A(tsz * n);
    s->lsc = (double *)A(sizeof(double) * b * b * N);
    s->lscT = mixed ? A(sizeof(float) * b * b * N) : (void *)s->lsc;
    if (o->cpr_stages == 3) {
        s->rhT = A(tsz * n);
        s->x0 = A(tsz * n);
    }
    s->scan = (int *)A(sizeof(int) * 3 * (N / 256 + 2));
    s->iscal = (int *)A(sizeof(int) * (SIM_SETUP_SCALARS + 2 * SIM_SETUP_LEVELS));
    if (!ok) {
        std::string m = s->msg;
        sim_destroy(s);
        return sim_fail(nullptr, SIM_ENOMEM, m);
    }
    if (cudaMallocHost(&s->h_pinned, sizeof(double) * 128) != cudaSuccess ||
        cudaMallocHost(&s->ctl_host, sizeof(KrylovCtl)) != cudaSuccess ||
        cudaMallocHost(&s->bctl_host, sizeof(BicgCtl)) != cudaSuccess) {
        sim_destroy(s);
        return sim_fail(nullptr, SIM_ENOMEM, "pinned host allocation failed");
    }
    for (cudaEvent_t &e : s->pev) {
        if (cudaEventCreate(&e) != cudaSuccess) {
            e = nullptr;
            sim_destroy(s);
            return sim_fail(nullptr, SIM_ECUDA, "event creation failed");
        }
    }
    // a stream-ordered memory pool that keeps freed AMG buffers for reuse
    int dev = 0;
    cudaGetDevice(&dev);
    cudaMemPool_t pool;
    if (cudaDeviceGetDefaultMemPool(&pool, dev) == cudaSuccess) {
        uint64_t thr = ~0ULL;
        cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &thr);
    }
    cudaMemsetAsync(s->ticket, 0, sizeof(unsigned int) * 4, s->stream);
    cudaMemsetAsync(s->x, 0, sizeof(double) * n, s->stream);
    cudaMemsetAsync(s->ph, 1, N, s->stream);
    if (!pvt.empty() &&
        cudaMemcpy(pvt_dev, pvt.data(), sizeof(double) * pvt.size(), cudaMemcpyHostToDevice) != cudaSuccess) {
        sim_destroy(s);
        return sim_fail(nullptr, SIM_ECUDA, "PVT table upload failed");
    }
    if (ok && nwells > 0) {
        std::vector<int> cp;
        if (nrate > 0) {
            cp.assign(N, -1);
            for (size_t q = 0; q < pc.size(); q++)
                if (wctrl[pw[q]] != SIM_WELL_BHP) cp[pc[q]] = (int)q;
        }
        bool up = cudaMemcpy(s->woff, woff.data(), sizeof(int) * (nwells + 1), cudaMemcpyHostToDevice) == cudaSuccess &&
                  cudaMemcpy(s->wctrl, wctrl.data(), sizeof(int) * nwells, cudaMemcpyHostToDevice) == cudaSuccess &&
                  cudaMemcpy(s->wrate, wrate.data(), sizeof(double) * nwells, cudaMemcpyHostToDevice) == cudaSuccess &&
                  cudaMemcpy(s->wbhp_c, wbhp.data(), sizeof(double) * nwells, cudaMemcpyHostToDevice) == cudaSuccess &&
                  cudaMemcpy(s->wp, wbhp.data(), sizeof(double) * nwells, cudaMemcpyHostToDevice) == cudaSuccess &&
                  cudaMemcpy(s->wp_old, wbhp.data(), sizeof(double) * nwells, cudaMemcpyHostToDevice) == cudaSuccess &&
                  (nrate == 0 || cudaMemcpy(s->cell_perf, cp.data(), sizeof(int) * N, cudaMemcpyHostToDevice) == cudaSuccess);
        if (!up) {
            sim_destroy(s);
            return sim_fail(nullptr, SIM_ECUDA, "well upload failed");
        }
    }
    if (k_geometry(s, r->kx, r->ky, r->kz, r->poro, pc.data(), pt.data(), pw.data(), pz.data(), prw.data(),
                   pskin.data()) != SIM_OK) {
        std::string m = s->msg;
        sim_status st = s->err;
        sim_destroy(s);
        return sim_fail(nullptr, st, m);
    }
    *out = s;
    return SIM_OK;
}

// ---------------------------------------------------------------------------
// state
// ---------------------------------------------------------------------------
// the current state becomes the start of a step; m_known: its component
// masses when the caller has them, else they are computed here
static sim_status begin_step(sim_t *s, const double *m_known = nullptr) {
    const long n = (long)s->N * s->b;
    SIM_CK(s, cudaMemcpyAsync(s->x_old, s->x, sizeof(double) * n, cudaMemcpyDeviceToDevice, s->stream));
    SIM_CK(s, cudaMemcpyAsync(s->ph_old, s->ph, s->N, cudaMemcpyDeviceToDevice, s->stream));
    if (s->nwells) SIM_CK(s, cudaMemcpyAsync(s->wp_old, s->wp, sizeof(double) * s->nwells, cudaMemcpyDeviceToDevice, s->stream));
    if (m_known) {
        for (int c = 0; c < 3; c++) s->m_start[c] = m_known[c];
    } else if (k_component_mass(s, s->m_start) != SIM_OK) {
        return s->err;
    }
    return k_accumulation(s, s->x, s->ph, s->mold);
}

sim_status sim_set_state(sim_t *s, const double *p, const double *sw, const double *x3, const int8_t *phase) {
    CHECK_HANDLE(s);
    if (!p || !sw || (s->b == 3 && (!x3 || !phase))) return sim_fail(s, SIM_EINVAL, "NULL state array");
    const int N = s->N;
    // staged in a work vector and checked before the accepted state is touched
    double *st = s->w;
    SIM_CK(s, cudaMemcpyAsync(st, p, sizeof(double) * N, cudaMemcpyHostToDevice, s->stream));
    SIM_CK(s, cudaMemcpyAsync(st + N, sw, sizeof(double) * N, cudaMemcpyHostToDevice, s->stream));
    if (s->b == 3) SIM_CK(s, cudaMemcpyAsync(st + 2L * N, x3, sizeof(double) * N, cudaMemcpyHostToDevice, s->stream));
    int ok = 1;
    if (k_finite(s, st, (long)N * s->b, &ok) != SIM_OK) return s->err;
    if (!ok) return sim_fail(s, SIM_ENAN, "sim_set_state: non-finite value in the state (state left unchanged)");
    SIM_CK(s, cudaMemcpyAsync(s->x, st, sizeof(double) * N * s->b, cudaMemcpyDeviceToDevice, s->stream));
    if (s->b == 3) {
        SIM_CK(s, cudaMemcpyAsync(s->ph, phase, N, cudaMemcpyHostToDevice, s->stream));
    } else {
        SIM_CK(s, cudaMemsetAsync(s->ph, 1, N, s->stream));
    }
    s->cum_well[0] = s->cum_well[1] = s->cum_well[2] = 0.0;
    if (begin_step(s) != SIM_OK) return s->err;
    SIM_CK(s, cudaStreamSynchronize(s->stream));
    return SIM_OK;
}

sim_status sim_get_state(sim_t *s, double *p, double *sw, double *x3, int8_t *phase) {
    CHECK_HANDLE(s);
    const int N = s->N;
    if (p) SIM_CK(s, cudaMemcpyAsync(p, s->x, sizeof(double) * N, cudaMemcpyDeviceToHost, s->stream));
    if (sw) SIM_CK(s, cudaMemcpyAsync(sw, s->x + N, sizeof(double) * N, cudaMemcpyDeviceToHost, s->stream));
    if (x3) {
        if (s->b == 3) SIM_CK(s, cudaMemcpyAsync(x3, s->x + 2L * N, sizeof(double) * N, cudaMemcpyDeviceToHost, s->stream));
        else memset(x3, 0, sizeof(double) * N);
    }
    if (phase) SIM_CK(s, cudaMemcpyAsync(phase, s->ph, N, cudaMemcpyDeviceToHost, s->stream));
    SIM_CK(s, cudaStreamSynchronize(s->stream));
    return SIM_OK;
}

sim_status sim_set_iterate(sim_t *s, const double *x, const int8_t *phase) {
    CHECK_HANDLE(s);
    if (!x || !phase) return sim_fail(s, SIM_EINVAL, "NULL iterate");
    const long n = (long)s->N * s->b;
    SIM_CK(s, cudaMemcpyAsync(s->w, x, sizeof(double) * n, cudaMemcpyHostToDevice, s->stream));
    int ok = 1;
    if (k_finite(s, s->w, n, &ok) != SIM_OK) return s->err;
    if (!ok) return sim_fail(s, SIM_ENAN, "sim_set_iterate: non-finite value in the iterate (iterate left unchanged)");
    SIM_CK(s, cudaMemcpyAsync(s->x, s->w, sizeof(double) * n, cudaMemcpyDeviceToDevice, s->stream));
    SIM_CK(s, cudaMemcpyAsync(s->ph, phase, s->N, cudaMemcpyHostToDevice, s->stream));
    SIM_CK(s, cudaStreamSynchronize(s->stream));
    return SIM_OK;
}

sim_status sim_get_iterate(sim_t *s, double *x, int8_t *phase) {
    CHECK_HANDLE(s);
    if (x) SIM_CK(s, cudaMemcpyAsync(x, s->x, sizeof(double) * s->N * s->b, cudaMemcpyDeviceToHost, s->stream));
    if (phase) SIM_CK(s, cudaMemcpyAsync(phase, s->ph, s->N, cudaMemcpyDeviceToHost, s->stream));
    SIM_CK(s, cudaStreamSynchronize(s->stream));
    return SIM_OK;
}

// ---------------------------------------------------------------------------
// Newton (Algorithm 1) and time stepping
// ---------------------------------------------------------------------------
sim_status sim_assemble(sim_t *s, double dt) {
    CHECK_HANDLE(s);
    if (!(dt > 0)) return sim_fail(s, SIM_EINVAL, "dt must be positive");
    if (k_assemble(s, dt) != SIM_OK) return s->err;
    SIM_CK(s, cudaStreamSynchronize(s->stream));
    return SIM_OK;
}

sim_status sim_cnv(sim_t *s, double dt, double *cnv) {
    CHECK_HANDLE(s);
    return k_cnv(s, dt, cnv);
}

// forcing state of one Newton solve (Algorithm 1, Eq. 14)
struct Forcing {
    int l = 0;                      // Newton iteration within the solve
    double bprev = 0.0, rprev = 0.0, theta = 0.0;
};

// theta_l from ||b^l||, the previous ||b^{l-1}||, ||r^{l-1}|| and theta_{l-1}.
// Choice 2 takes the absolute value of its numerator; the first iteration
// uses theta_max; the Eisenstat-Walker safeguards keep theta from falling
// below theta_{l-1}^((1+sqrt 5)/2) (choices 1, 2) or gamma theta_{l-1}^beta
// (choice 3) while that bound exceeds 0.1; lin_tol <= theta <= theta_max.
static sim_status forcing_term(sim_t *s, const Forcing &f, double bnorm, double *theta) {
    const sim_options &o = s->opt;
    if (o.forcing == SIM_FORCING_FIXED) { *theta = o.lin_tol; return SIM_OK; }
    if (f.l == 0) { *theta = o.theta_max; return SIM_OK; }
    double th, guard;
    if (o.forcing == SIM_FORCING_EW1) {
        double d;
        if (k_diff_norm2(s, s->bl, s->rlin, (long)s->N * s->b, &d) != SIM_OK) return s->err;
        th = d / f.bprev;
        guard = pow(f.theta, 0.5 * (1.0 + sqrt(5.0)));
    } else if (o.forcing == SIM_FORCING_EW2) {
        th = fabs(bnorm - f.rprev) / f.bprev;
        guard = pow(f.theta, 0.5 * (1.0 + sqrt(5.0)));
    } else {
        th = o.ew_gamma * pow(bnorm / f.bprev, o.ew_beta);
        guard = o.ew_gamma * pow(f.theta, o.ew_beta);
    }
    if (guard > 0.1 && guard > th) th = guard;
    if (th > o.theta_max) th = o.theta_max;
    if (th < o.lin_tol) th = o.lin_tol;
    *theta = th;
    return SIM_OK;
}

// ---- per-phase figures of a Newton iteration (sim_phase_info) ----------------
// algorithmic bytes from the sizes and the levels' entries (the model stated in sim.h)
static double apply_bytes_per_value(const sim_t *s) { return sim_mixed(s) ? 4.0 : 8.0; }

static double bytes_assembly(const sim_t *s) {
    const double N = s->N, b = s->b;
    return N * (7 * b * b + 3 * b + 4) * 8;
}

static double bytes_update(const sim_t *s) { return 3.0 * s->b * (double)s->N * 8; }

static double bytes_setup(const sim_t *s) {
    const double N = s->N, b = s->b, t = apply_bytes_per_value(s);
    double v = N * (7 * b * b * (8 + 2 * t) + 7 * 8 + b * b * t);
    const int nl = (int)s->lev.size();
    for (int l = 0; l + 1 < nl; l++) {
        v += 4 * s->lev[l].entries * 12 + s->lev[l + 1].entries * 12 + 4.0 * s->lev[l].n;
    }
    return v;
}

// one CPR application (two-stage; the three-stage form adds one stage F and
// its residual)
static double bytes_apply(const sim_t *s) {
    const double N = s->N, b = s->b, t = apply_bytes_per_value(s);
    double v = N * (8 * b + b * t + t);                       // restriction
    const int nl = (int)s->lev.size();
    for (int l = 0; l < nl; l++) {
        const double n = s->lev[l].n;
        if (l + 1 == nl) { v += n * n * 8 + 2 * n * t; break; }   // dense coarsest product
        v += 3 * s->lev[l].entries * (l == 0 ? t : 4 + t) + 6 * n * t;      // smoothing, residual, prolongation
    }
    const double stage_f = N * (8 * b + b * b * t + 7 * b * t + t + b * t)      // r - Ahat x1 (pressure columns)
                         + N * (7 * b * b * t + b * b * t + 3 * b * t + b * t); // red-black ILU(0) sweeps
    v += stage_f;
    if (s->opt.cpr_stages == 3) v += stage_f + N * 7 * b * b * t;
    return v;
}

static double bytes_solve(const sim_t *s, const sim_linear_info &li) {
    const double N = s->N, b = s->b, n = b * N;
    const double tz = sim_mixed(s) ? 4.0 : 8.0;
    const double spmv = (7 * b * b + b) * 8 * N + b * N * tz;
    const double apply = s->opt.precond == SIM_PRECOND_CPR ? bytes_apply(s) : N * (b * b * 8 + 2 * b * 8);
    if (s->opt.krylov == SIM_KRYLOV_BICGSTAB)
        return li.iterations * (2 * spmv + 2 * apply + 12 * n * 8) + (li.restarts + 1) * (spmv + 3 * n * 8);
    double v = 0.0;
    int left = li.iterations;
    const int cycles = li.restarts + 1;
    for (int c = 0; c < cycles; c++) {
        const int k = (c + 1 == cycles) ? left : (left < s->m ? left : s->m);
        for (int j = 0; j < k; j++) v += spmv + apply + (3.0 * (j + 1) + 7) * n * 8;
        v += k * n * tz + 2 * n * 8 + spmv + 3 * n * 8;    // x += Z y, then r = b - J x
        left -= k;
    }
    return v;
}

static void phase_add(sim_phase_info *a, const sim_phase_info &b) {
    a->assemble_us += b.assemble_us; a->setup_us += b.setup_us; a->solve_us += b.solve_us; a->update_us += b.update_us;
    a->assemble_bytes += b.assemble_bytes; a->setup_bytes += b.setup_bytes;
    a->solve_bytes += b.solve_bytes; a->update_bytes += b.update_bytes;
}

static double event_us(cudaEvent_t a, cudaEvent_t b) {
    float ms = 0.f;
    if (cudaEventElapsedTime(&ms, a, b) != cudaSuccess) { (void)cudaGetLastError(); return 0.0; }
    return 1e3 * ms;
}

// assemble and test CNV, with the assembly phase marked by pev[0], pev[1]
static sim_status assemble_and_test(sim_t *s, double dt, double *cnv, double *wcnv, sim_phase_info *ph) {
    NvtxRange range("assemble");
    SIM_CK(s, cudaEventRecord(s->pev[0], s->stream));
    if (k_assemble(s, dt) != SIM_OK) return s->err;
    if (k_cnv(s, dt, cnv, wcnv) != SIM_OK) return s->err;
    SIM_CK(s, cudaEventRecord(s->pev[1], s->stream));
    SIM_CK(s, cudaEventSynchronize(s->pev[1]));
    ph->assemble_us += event_us(s->pev[0], s->pev[1]);
    ph->assemble_bytes += bytes_assembly(s);
    return SIM_OK;
}

// solve J dx = -R and update; *lin receives the linear info.  With a forcing
// state the tolerance is its theta_l, else lin_tol.  The preconditioner
// setup, the solve and the update are marked by pev[1..4] into *ph.
static sim_status solve_and_update(sim_t *s, sim_linear_info *lin, bool *finite_ok, sim_phase_info *ph,
                                   Forcing *f = nullptr) {
    const long n = (long)s->N * s->b;
    SIM_CK(s, cudaEventRecord(s->pev[1], s->stream));
    if (!s->precond_ready) {
        NvtxRange range("cpr_setup");
        if (cpr_setup(s) != SIM_OK) return s->err;
        ph->setup_bytes += s->opt.precond == SIM_PRECOND_CPR ? bytes_setup(s)
                                                             : (double)s->N * s->b * s->b * 8 * 9;   // block Jacobi
    }
    SIM_CK(s, cudaEventRecord(s->pev[2], s->stream));
    negate_kernel<<<SIM_RED_BLOCKS, SIM_THREADS, 0, s->stream>>>(s->R, s->bl, n);
    SIM_LAUNCHED(s);
    if (k_well_rhs(s, s->bl) != SIM_OK) return s->err;
    double bnorm = 0.0;
    s->theta = s->opt.lin_tol;
    if (f && s->opt.forcing != SIM_FORCING_FIXED) {
        if (k_norm2(s, s->bl, n, &bnorm) != SIM_OK) return s->err;
        if (forcing_term(s, *f, bnorm, &s->theta) != SIM_OK) return s->err;
    }
    sim_status st;
    {
        NvtxRange range("linear_solve");
        st = k_linear_solve(s, s->bl, s->dx, lin);
    }
    SIM_CK(s, cudaEventRecord(s->pev[3], s->stream));
    ph->solve_bytes += bytes_solve(s, *lin);
    const double theta_used = s->theta;
    s->theta = s->opt.lin_tol;
    if (f && s->opt.forcing != SIM_FORCING_FIXED && st == SIM_OK) {
        f->bprev = bnorm; f->rprev = lin->r_norm; f->theta = theta_used; f->l++;
        SIM_CK(s, cudaMemcpyAsync(s->rlin, s->r, sizeof(double) * n, cudaMemcpyDeviceToDevice, s->stream));
    }
    if (st != SIM_OK) {
        if (s->err == SIM_ENAN) { sim_clear_error(s); *finite_ok = false; return SIM_OK; }
        return s->err;
    }
    NvtxRange range("update");
    int ok = 1;
    if (k_finite(s, s->dx, n, &ok) != SIM_OK) return s->err;
    *finite_ok = ok != 0;
    if (!ok) return SIM_OK;
    if (k_well_update(s, s->dx) != SIM_OK) return s->err;
    if (k_newton_update(s, s->dx) != SIM_OK) return s->err;
    SIM_CK(s, cudaEventRecord(s->pev[4], s->stream));
    SIM_CK(s, cudaEventSynchronize(s->pev[4]));
    ph->setup_us += event_us(s->pev[1], s->pev[2]);
    ph->solve_us += event_us(s->pev[2], s->pev[3]);
    ph->update_us += event_us(s->pev[3], s->pev[4]);
    ph->update_bytes += bytes_update(s);
    s->newton_total++;
    return SIM_OK;
}

sim_status sim_newton_step(sim_t *s, double dt, sim_newton_info *info) {
    CHECK_HANDLE(s);
    if (!(dt > 0)) return sim_fail(s, SIM_EINVAL, "dt must be positive");
    sim_newton_info ni;
    memset(&ni, 0, sizeof(ni));
    double cnv, wcnv;
    if (assemble_and_test(s, dt, &cnv, &wcnv, &ni.phase) != SIM_OK) return s->err;
    ni.cnv = cnv;
    if (cnv <= s->opt.newton_tol && wcnv <= s->opt.newton_tol) {
        ni.converged = 1;
        phase_add(&s->run_phase, ni.phase);
        if (info) *info = ni;
        return SIM_OK;
    }
    sim_linear_info li;
    bool fin = true;
    if (solve_and_update(s, &li, &fin, &ni.phase) != SIM_OK) return s->err;
    ni.newton_iterations = 1;
    ni.linear_iterations = li.iterations;
    ni.linear_failures = !li.converged;
    ni.lin_residual = li.b_norm > 0 ? li.r_norm / li.b_norm : 0.0;
    s->run_lin_failures += !li.converged;
    phase_add(&s->run_phase, ni.phase);
    if (info) *info = ni;
    return fin ? SIM_OK : SIM_ENAN;
}

}  // extern "C"

// ---- the pieces of a Newton iteration, for the ensemble runtime -------------
// (the steps newton_solve and sim_step take, in the same order, so that a
// member advanced by the batch computes what sim_step computes)
sim_status nl_assemble_test(sim_t *s, double dt, int *state, sim_phase_info *ph) {
    double cnv, wcnv;
    if (assemble_and_test(s, dt, &cnv, &wcnv, ph) != SIM_OK) return s->err;
    if (!(cnv == cnv) || !(wcnv == wcnv)) *state = 2;
    else if (cnv <= s->opt.newton_tol && wcnv <= s->opt.newton_tol) *state = 1;
    else *state = 0;
    return SIM_OK;
}

// right-hand side -R (+ the rate wells' term) into bl, the preconditioner set up
sim_status nl_prepare_solve(sim_t *s, sim_phase_info *ph) {
    const long n = (long)s->N * s->b;
    SIM_CK(s, cudaEventRecord(s->pev[1], s->stream));
    if (!s->precond_ready) {
        if (cpr_setup(s) != SIM_OK) return s->err;
        ph->setup_bytes += bytes_setup(s);
    }
    SIM_CK(s, cudaEventRecord(s->pev[2], s->stream));
    negate_kernel<<<SIM_RED_BLOCKS, SIM_THREADS, 0, s->stream>>>(s->R, s->bl, n);
    SIM_LAUNCHED(s);
    if (k_well_rhs(s, s->bl) != SIM_OK) return s->err;
    s->theta = s->opt.lin_tol;
    SIM_CK(s, cudaEventSynchronize(s->pev[2]));
    ph->setup_us += event_us(s->pev[1], s->pev[2]);
    SIM_CK(s, cudaStreamSynchronize(s->stream));
    return SIM_OK;
}

// after the (batched) solve of dx: finiteness, the wells' and cells' update
sim_status nl_finish_solve(sim_t *s, const sim_linear_info &li, bool *finite_ok, sim_phase_info *ph) {
    const long n = (long)s->N * s->b;
    ph->solve_bytes += bytes_solve(s, li);
    *finite_ok = li.r_norm == li.r_norm;
    if (!*finite_ok) return SIM_OK;
    SIM_CK(s, cudaEventRecord(s->pev[3], s->stream));
    int ok = 1;
    if (k_finite(s, s->dx, n, &ok) != SIM_OK) return s->err;
    *finite_ok = ok != 0;
    if (!ok) return SIM_OK;
    if (k_well_update(s, s->dx) != SIM_OK) return s->err;
    if (k_newton_update(s, s->dx) != SIM_OK) return s->err;
    SIM_CK(s, cudaEventRecord(s->pev[4], s->stream));
    SIM_CK(s, cudaEventSynchronize(s->pev[4]));
    ph->update_us += event_us(s->pev[3], s->pev[4]);
    ph->update_bytes += bytes_update(s);
    s->newton_total++;
    return SIM_OK;
}

// the start of the step again (a failed Newton solve, before the step is halved)
sim_status nl_restore(sim_t *s) {
    SIM_CK(s, cudaMemcpyAsync(s->x, s->x_old, sizeof(double) * s->N * s->b, cudaMemcpyDeviceToDevice, s->stream));
    SIM_CK(s, cudaMemcpyAsync(s->ph, s->ph_old, s->N, cudaMemcpyDeviceToDevice, s->stream));
    if (s->nwells)
        SIM_CK(s, cudaMemcpyAsync(s->wp, s->wp_old, sizeof(double) * s->nwells, cudaMemcpyDeviceToDevice, s->stream));
    return SIM_OK;
}

// the current iterate becomes the accepted state of a step of length dt
sim_status accept_step(sim_t *s, double dt) {
    SIM_CK(s, cudaMemcpyAsync(s->h_pinned, s->qtot, sizeof(double) * 3, cudaMemcpyDeviceToHost, s->stream));
    SIM_CK(s, cudaStreamSynchronize(s->stream));
    double q[3], m[3];
    for (int c = 0; c < 3; c++) q[c] = s->h_pinned[c];
    for (int c = 0; c < 3; c++) s->cum_well[c] += dt * q[c];
    // mass balance of the substep: the masses in place against the start's plus the wells' inflow
    if (k_component_mass(s, m) != SIM_OK) return s->err;
    double total = 0.0, worst = 0.0;
    for (int c = 0; c < s->b; c++) {
        total += m[c];
        worst = fmax(worst, fabs(m[c] - s->m_start[c] - dt * q[c]));
    }
    s->last_mb = total > 0.0 ? worst / total : worst;
    s->run_max_mb = fmax(s->run_max_mb, s->last_mb);
    s->run_substeps++;
    s->run_days += dt;
    return begin_step(s, m);
}

void run_record_step(sim_t *s, const sim_step_info &si, sim_status st) {
    if (st == SIM_OK) s->run_steps++;
    else s->run_failed_steps++;
    s->run_cuts += si.cuts;
    phase_add(&s->run_phase, si.phase);
}

extern "C" {

// Newton loop; returns 0 converged, 1 not converged, 2 non-finite
static int newton_solve(sim_t *s, double dt, sim_newton_info *ni) {
    memset(ni, 0, sizeof(*ni));
    Forcing f;
    for (int l = 0;; l++) {
        double cnv, wcnv;
        if (assemble_and_test(s, dt, &cnv, &wcnv, &ni->phase) != SIM_OK) return -1;
        ni->cnv = cnv;
        if (!(cnv == cnv) || !(wcnv == wcnv)) return 2;
        if (cnv <= s->opt.newton_tol && wcnv <= s->opt.newton_tol) { ni->converged = 1; return 0; }
        if (l >= s->opt.newton_max) return 1;
        sim_linear_info li;
        bool fin = true;
        if (solve_and_update(s, &li, &fin, &ni->phase, &f) != SIM_OK) return -1;
        ni->newton_iterations++;
        ni->linear_iterations += li.iterations;
        ni->linear_failures += !li.converged;
        ni->lin_residual = fmax(ni->lin_residual, li.b_norm > 0 ? li.r_norm / li.b_norm : 0.0);
        s->run_lin_failures += !li.converged;
        if (!fin) return 2;
    }
}

sim_status sim_newton_solve(sim_t *s, double dt, sim_newton_info *info) {
    CHECK_HANDLE(s);
    if (!(dt > 0)) return sim_fail(s, SIM_EINVAL, "dt must be positive");
    sim_newton_info ni;
    const int rc = newton_solve(s, dt, &ni);
    if (info) *info = ni;
    if (rc < 0) return s->err;
    phase_add(&s->run_phase, ni.phase);
    return rc == 0 ? SIM_OK : (rc == 2 ? SIM_ENAN : SIM_ENOCONV_NEWTON);
}


sim_status sim_accept_step(sim_t *s, double dt) {
    CHECK_HANDLE(s);
    if (!(dt > 0)) return sim_fail(s, SIM_EINVAL, "dt must be positive");
    if (accept_step(s, dt) != SIM_OK) return s->err;
    SIM_CK(s, cudaStreamSynchronize(s->stream));
    return SIM_OK;
}

sim_status sim_step(sim_t *s, double dt, sim_step_info *info) {
    CHECK_HANDLE(s);
    if (!(dt > 0)) return sim_fail(s, SIM_EINVAL, "dt must be positive");
    NvtxRange range("sim_step");
    sim_step_info si;
    memset(&si, 0, sizeof(si));
    double remaining = dt, h = dt;
    sim_status st = SIM_OK;
    while (remaining > 1e-12 * dt) {
        if (h > remaining) h = remaining;
        sim_newton_info ni;
        const int rc = newton_solve(s, h, &ni);
        if (rc < 0) return s->err;
        phase_add(&si.phase, ni.phase);
        si.newton_iterations += ni.newton_iterations;
        si.linear_iterations += ni.linear_iterations;
        if (rc == 0) {
            if (accept_step(s, h) != SIM_OK) return s->err;
            remaining -= h;
            si.substeps++;
            si.mb_error = fmax(si.mb_error, s->last_mb);
        } else {
            if (nl_restore(s) != SIM_OK) return s->err;
            si.cuts++;
            if (si.cuts > s->opt.max_cuts) { st = SIM_ENOCONV_NEWTON; break; }
            h *= 0.5;
        }
    }
    SIM_CK(s, cudaStreamSynchronize(s->stream));
    si.ok = st == SIM_OK;
    run_record_step(s, si, st);
    if (info) *info = si;
    return st;
}

sim_status sim_linear_solve(sim_t *s, const double *b_dev, double *x_dev, sim_linear_info *info) {
    CHECK_HANDLE(s);
    if (!b_dev || !x_dev || b_dev == x_dev) return sim_fail(s, SIM_EINVAL, "bad vector pointers");
    sim_linear_info li;
    if (k_linear_solve(s, b_dev, x_dev, &li) != SIM_OK) return s->err;
    if (info) *info = li;
    return li.converged ? SIM_OK : SIM_ENOCONV_LINEAR;
}

// ---------------------------------------------------------------------------
// inspection
// ---------------------------------------------------------------------------
sim_status sim_get_residual(sim_t *s, double *R) {
    CHECK_HANDLE(s);
    SIM_CK(s, cudaMemcpyAsync(R, s->R, sizeof(double) * s->N * s->b, cudaMemcpyDeviceToHost, s->stream));
    SIM_CK(s, cudaStreamSynchronize(s->stream));
    return SIM_OK;
}
sim_status sim_get_jacobian(sim_t *s, double *J) {
    CHECK_HANDLE(s);
    SIM_CK(s, cudaMemcpyAsync(J, s->J, sizeof(double) * 7 * s->b * s->b * (size_t)s->N, cudaMemcpyDeviceToHost, s->stream));
    SIM_CK(s, cudaStreamSynchronize(s->stream));
    return SIM_OK;
}
sim_status sim_set_jacobian(sim_t *s, const double *J) {
    CHECK_HANDLE(s);
    SIM_CK(s, cudaMemcpyAsync(s->J, J, sizeof(double) * 7 * s->b * s->b * (size_t)s->N, cudaMemcpyHostToDevice, s->stream));
    SIM_CK(s, cudaStreamSynchronize(s->stream));
    s->precond_ready = false;
    return SIM_OK;
}
sim_status sim_spmv(sim_t *s, const double *x_dev, double *y_dev) {
    CHECK_HANDLE(s);
    if (k_spmv(s, x_dev, y_dev) != SIM_OK) return s->err;
    SIM_CK(s, cudaStreamSynchronize(s->stream));
    return SIM_OK;
}
sim_status sim_time_op(sim_t *s, int32_t which, int32_t reps, double *us) {
    CHECK_HANDLE(s);
    if (!us || reps < 1 || which < 0 || which > 2) return sim_fail(s, SIM_EINVAL, "sim_time_op: bad arguments");
    const int nv = s->m < 16 ? s->m : 16;
    const long n = (long)s->N * s->b;
    if (which == 1 && !s->precond_ready && cpr_setup(s) != SIM_OK) return s->err;
    // a buffer twice the L2 size, rewritten before every timed launch, so that
    // each launch starts with its operands out of the cache
    const size_t flush_bytes = 256u << 20;
    void *flush = sim_alloc(s, flush_bytes);
    if (!flush) return s->err;
    SIM_CK(s, cudaMemsetAsync(s->V, 0, sizeof(double) * n * (which == 2 ? nv + 1 : 1), s->stream));
    if (which == 2) SIM_CK(s, cudaMemsetAsync(s->w, 0, sizeof(double) * n, s->stream));
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    sim_status st = SIM_OK;
    if (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess) st = SIM_ECUDA;
    double total_ms = 0.0;
    for (int r = 0; r < reps && st == SIM_OK; r++) {
        float ms = 0.f;
        if (which == 2 &&   // no convergence test may stop the step: done = 0, tol = NaN
            (cudaMemsetAsync(&s->ctl->done, 0, sizeof(int), s->stream) != cudaSuccess ||
             cudaMemsetAsync(&s->ctl->tol, 0xff, sizeof(double), s->stream) != cudaSuccess)) { st = SIM_ECUDA; break; }
        if (cudaMemsetAsync(flush, r & 0xff, flush_bytes, s->stream) != cudaSuccess ||
            cudaEventRecord(e0, s->stream) != cudaSuccess) { st = SIM_ECUDA; break; }
        st = which == 0 ? k_spmv(s, s->V, s->w) : which == 1 ? cpr_apply(s, s->V, s->Z, nullptr) : k_orth_step(s, nv);
        if (st != SIM_OK) break;
        if (cudaEventRecord(e1, s->stream) != cudaSuccess || cudaEventSynchronize(e1) != cudaSuccess ||
            cudaEventElapsedTime(&ms, e0, e1) != cudaSuccess) { st = SIM_ECUDA; break; }
        total_ms += ms;
    }
    if (e0) cudaEventDestroy(e0);
    if (e1) cudaEventDestroy(e1);
    sim_free(s, flush);
    if (st != SIM_OK) return s->err != SIM_OK ? s->err : sim_fail(s, SIM_ECUDA, "sim_time_op: event timing failed");
    *us = 1e3 * total_ms / reps;
    return SIM_OK;
}

sim_status sim_precond_setup(sim_t *s) {
    CHECK_HANDLE(s);
    if (cpr_setup(s) != SIM_OK) return s->err;
    SIM_CK(s, cudaStreamSynchronize(s->stream));
    return SIM_OK;
}
sim_status sim_precond_apply(sim_t *s, const double *r_dev, double *z_dev) {
    CHECK_HANDLE(s);
    const long n = (long)s->N * s->b;
    void *z = sim_mixed(s) ? s->Z : (void *)z_dev;
    if (cpr_apply(s, r_dev, z, nullptr) != SIM_OK) return s->err;
    if (sim_mixed(s)) {   // widen the FP32 result into the caller's FP64 buffer
        widen_kernel<<<SIM_RED_BLOCKS, SIM_THREADS, 0, s->stream>>>((const float *)s->Z, z_dev, n);
        SIM_LAUNCHED(s);
    }
    SIM_CK(s, cudaStreamSynchronize(s->stream));
    return SIM_OK;
}
sim_status sim_get_qi(sim_t *s, double *w, double *ap) {
    CHECK_HANDLE(s);
    if (!s->precond_ready) return sim_fail(s, SIM_EINVAL, "preconditioner not set up");
    if (w) SIM_CK(s, cudaMemcpyAsync(w, s->qiw, sizeof(double) * s->N * s->b, cudaMemcpyDeviceToHost, s->stream));
    if (ap) SIM_CK(s, cudaMemcpyAsync(ap, s->ap, sizeof(double) * 7 * (size_t)s->N, cudaMemcpyDeviceToHost, s->stream));
    SIM_CK(s, cudaStreamSynchronize(s->stream));
    return SIM_OK;
}
int32_t sim_amg_levels(sim_t *s) { return s ? (int32_t)s->lev.size() : 0; }
sim_status sim_amg_level_info(sim_t *s, int32_t level, int32_t *n, int32_t *width) {
    CHECK_HANDLE(s);
    if (level < 0 || level >= (int)s->lev.size()) return sim_fail(s, SIM_EINVAL, "level out of range");
    if (n) *n = s->lev[level].n;
    if (width) *width = s->lev[level].width;
    return SIM_OK;
}
sim_status sim_amg_level_agg(sim_t *s, int32_t level, int32_t *agg) {
    CHECK_HANDLE(s);
    if (level < 0 || level + 1 >= (int)s->lev.size()) return sim_fail(s, SIM_EINVAL, "level has no aggregates");
    SIM_CK(s, cudaMemcpyAsync(agg, s->lev[level].agg, sizeof(int) * s->lev[level].n, cudaMemcpyDeviceToHost, s->stream));
    SIM_CK(s, cudaStreamSynchronize(s->stream));
    return SIM_OK;
}
sim_status sim_amg_level_ell(sim_t *s, int32_t level, int32_t *col, double *val) {
    CHECK_HANDLE(s);
    return cpr_copy_level_ell(s, level, col, val);
}
sim_status sim_component_mass(sim_t *s, double *m3) {
    CHECK_HANDLE(s);
    return k_component_mass(s, m3);
}
sim_status sim_cumulative_well_mass(sim_t *s, double *m3) {
    CHECK_HANDLE(s);
    for (int c = 0; c < 3; c++) m3[c] = s->cum_well[c];
    return SIM_OK;
}
sim_status sim_well_rates(sim_t *s, double *q3) {
    CHECK_HANDLE(s);
    SIM_CK(s, cudaMemcpyAsync(s->h_pinned, s->qtot, sizeof(double) * 3, cudaMemcpyDeviceToHost, s->stream));
    SIM_CK(s, cudaStreamSynchronize(s->stream));
    for (int c = 0; c < 3; c++) q3[c] = s->h_pinned[c];
    return SIM_OK;
}

int32_t sim_perforations(sim_t *s) { return s ? s->nperf : 0; }

sim_status sim_get_well_bhp(sim_t *s, double *bhp) {
    CHECK_HANDLE(s);
    if (!bhp) return sim_fail(s, SIM_EINVAL, "NULL array");
    if (s->nwells) SIM_CK(s, cudaMemcpyAsync(bhp, s->wp, sizeof(double) * s->nwells, cudaMemcpyDeviceToHost, s->stream));
    SIM_CK(s, cudaStreamSynchronize(s->stream));
    return SIM_OK;
}

sim_status sim_set_well_bhp(sim_t *s, const double *bhp) {
    CHECK_HANDLE(s);
    if (!bhp) return sim_fail(s, SIM_EINVAL, "NULL array");
    if (s->nwells) SIM_CK(s, cudaMemcpyAsync(s->wp, bhp, sizeof(double) * s->nwells, cudaMemcpyHostToDevice, s->stream));
    SIM_CK(s, cudaStreamSynchronize(s->stream));
    return SIM_OK;
}

sim_status sim_well_component_rates(sim_t *s, double *q) {
    CHECK_HANDLE(s);
    if (!q) return sim_fail(s, SIM_EINVAL, "NULL array");
    const int nw = s->nwells;
    if (!nw) return SIM_OK;
    std::vector<double> t(3 * (size_t)nw);
    SIM_CK(s, cudaMemcpyAsync(t.data(), s->qwell, sizeof(double) * 3 * nw, cudaMemcpyDeviceToHost, s->stream));
    SIM_CK(s, cudaStreamSynchronize(s->stream));
    for (int w = 0; w < nw; w++)
        for (int c = 0; c < 3; c++) q[w * 3 + c] = t[(size_t)c * nw + w];
    return SIM_OK;
}

sim_status sim_get_well_system(sim_t *s, double *Rw, double *Apw, double *Awp, double *Aww) {
    CHECK_HANDLE(s);
    const int nw = s->nwells, np = s->nperf, b = s->b;
    if (!nw) return SIM_OK;
    std::vector<double> a(3 * (size_t)np), c(3 * (size_t)np);
    if (Rw) SIM_CK(s, cudaMemcpyAsync(Rw, s->rw, sizeof(double) * nw, cudaMemcpyDeviceToHost, s->stream));
    if (Aww) SIM_CK(s, cudaMemcpyAsync(Aww, s->aww, sizeof(double) * nw, cudaMemcpyDeviceToHost, s->stream));
    SIM_CK(s, cudaMemcpyAsync(a.data(), s->apw, sizeof(double) * 3 * np, cudaMemcpyDeviceToHost, s->stream));
    SIM_CK(s, cudaMemcpyAsync(c.data(), s->awp, sizeof(double) * 3 * np, cudaMemcpyDeviceToHost, s->stream));
    SIM_CK(s, cudaStreamSynchronize(s->stream));
    for (int q = 0; q < np; q++)
        for (int k = 0; k < b; k++) {
            if (Apw) Apw[q * b + k] = a[(size_t)k * np + q];
            if (Awp) Awp[q * b + k] = c[(size_t)k * np + q];
        }
    return SIM_OK;
}

sim_status sim_set_well_system(sim_t *s, const double *Rw, const double *Apw, const double *Awp, const double *Aww) {
    CHECK_HANDLE(s);
    if (!Rw || !Apw || !Awp || !Aww) return sim_fail(s, SIM_EINVAL, "NULL array");
    const int nw = s->nwells, np = s->nperf, b = s->b;
    if (!nw) return SIM_OK;
    std::vector<double> a(3 * (size_t)np, 0.0), c(3 * (size_t)np, 0.0);
    for (int q = 0; q < np; q++)
        for (int k = 0; k < b; k++) { a[(size_t)k * np + q] = Apw[q * b + k]; c[(size_t)k * np + q] = Awp[q * b + k]; }
    SIM_CK(s, cudaMemcpyAsync(s->rw, Rw, sizeof(double) * nw, cudaMemcpyHostToDevice, s->stream));
    SIM_CK(s, cudaMemcpyAsync(s->aww, Aww, sizeof(double) * nw, cudaMemcpyHostToDevice, s->stream));
    SIM_CK(s, cudaMemcpyAsync(s->apw, a.data(), sizeof(double) * 3 * np, cudaMemcpyHostToDevice, s->stream));
    SIM_CK(s, cudaMemcpyAsync(s->awp, c.data(), sizeof(double) * 3 * np, cudaMemcpyHostToDevice, s->stream));
    SIM_CK(s, cudaStreamSynchronize(s->stream));
    s->precond_ready = false;
    return SIM_OK;
}
sim_status sim_set_learned_stage(sim_t *s, sim_net_t *net, int32_t enable) {
    CHECK_HANDLE(s);
    if (enable && !net) return sim_fail(s, SIM_EINVAL, "learned stage enabled without a network");
    if (net && net_cells(net) != s->N) return sim_fail(s, SIM_EINVAL, "network grid differs from the simulator grid");
    if (enable && !s->lfeat) {
        const size_t tsz = sim_mixed(s) ? sizeof(float) : sizeof(double);
        s->lfeat = (float *)sim_alloc(s, sizeof(float) * 3 * (size_t)s->N);
        s->lx = (float *)sim_alloc(s, sizeof(float) * 4 * (size_t)s->N);
        s->ly = (float *)sim_alloc(s, sizeof(float) * (size_t)s->N);
        s->lres = sim_alloc(s, tsz * s->N);
        s->lep = sim_alloc(s, tsz * s->N);
        s->lrms = (double *)sim_alloc(s, sizeof(double) * 2);
        if (!s->lfeat || !s->lx || !s->ly || !s->lres || !s->lep || !s->lrms) return s->err;
    }
    if (s->lfeat && cpr_learned_features(s) != SIM_OK) return s->err;
    s->net = net;
    s->learned_on = enable ? 1 : 0;
    SIM_CK(s, cudaStreamSynchronize(s->stream));
    return SIM_OK;
}

sim_status sim_learned_pairs(sim_t *s, int32_t k, float *x_dev, float *y_dev) {
    CHECK_HANDLE(s);
    if (!x_dev || !y_dev || k < 1 || k > s->last_cycle_k + 1 || k > s->m + 1)
        return SIM_EINVAL;   /* not sticky: the handle stays usable */
    if (!s->lfeat) {
        s->lfeat = (float *)sim_alloc(s, sizeof(float) * 3 * (size_t)s->N);
        s->lrms = (double *)sim_alloc(s, sizeof(double) * 2);
        if (!s->lfeat || !s->lrms) return s->err;
        if (cpr_learned_features(s) != SIM_OK) return s->err;
    }
    if (!s->lres) {
        s->lres = sim_alloc(s, (sim_mixed(s) ? sizeof(float) : sizeof(double)) * (size_t)s->N);
        if (!s->lres) return s->err;
    }
    if (cpr_learned_pairs(s, k, x_dev, y_dev) != SIM_OK) return s->err;
    SIM_CK(s, cudaStreamSynchronize(s->stream));
    return SIM_OK;
}

int64_t sim_learned_fallbacks(sim_t *s) { return s ? s->learned_fallbacks : 0; }
int32_t sim_learned_available(sim_t *s) { return s ? (s->last_cycle_k + 1 < s->m + 1 ? s->last_cycle_k + 1 : s->m + 1) : 0; }

sim_status sim_probe_fma_rates(double *fp64_fma_per_s, double *fp32_fma_per_s) {
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return sim_fail(nullptr, SIM_ECUDA, "sim_probe_fma_rates: no CUDA device");
    const int max_blocks = sms * 8, threads = 256;
    void *buf = nullptr;
    if (cudaMalloc(&buf, sizeof(double) * max_blocks * threads) != cudaSuccess)
        return sim_fail(nullptr, SIM_ENOMEM, "sim_probe_fma_rates: allocation failed");
    // the best of several shapes (chains per thread, blocks per SM): the rate of
    // the pipe, not of one shape's latency or tail
    double f64 = 0.0, f32 = 0.0;
    for (int bps : {4, 8}) {
        const int blocks = sms * bps;
        f64 = std::max(f64, probe_rate<double, 8>((double *)buf, blocks, threads, 8192));
        f64 = std::max(f64, probe_rate<double, 16>((double *)buf, blocks, threads, 4096));
        f32 = std::max(f32, probe_rate<float, 8>((float *)buf, blocks, threads, 32768));
        f32 = std::max(f32, probe_rate<float, 16>((float *)buf, blocks, threads, 16384));
    }
    if (fp64_fma_per_s) *fp64_fma_per_s = f64;
    if (fp32_fma_per_s) *fp32_fma_per_s = f32;
    cudaFree(buf);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return sim_fail(nullptr, SIM_ECUDA, std::string("sim_probe_fma_rates: ") + cudaGetErrorString(e));
    return SIM_OK;
}

sim_status sim_probe_fp64_pipe(double *fma_per_s, double *sm_mhz, double *fma_per_clk_per_sm) {
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return sim_fail(nullptr, SIM_ECUDA, "sim_probe_fp64_pipe: no CUDA device");
    const int threads = 256;
    double best = 0.0, best_mhz = 0.0;
    void *buf = nullptr, *st = nullptr;
    if (cudaMalloc(&buf, sizeof(double) * sms * 8 * threads) != cudaSuccess ||
        cudaMalloc(&st, sizeof(long long) * 2 * sms * 8) != cudaSuccess) {
        cudaFree(buf);
        return sim_fail(nullptr, SIM_ENOMEM, "sim_probe_fp64_pipe: allocation failed");
    }
    std::vector<long long> h(2 * sms * 8);
    for (int bps : {4, 8}) {
        const int blocks = sms * bps;
        for (int nc : {8, 16}) {
            const double r = nc == 8 ? probe_rate<double, 8>((double *)buf, blocks, threads, 8192, (long long *)st)
                                     : probe_rate<double, 16>((double *)buf, blocks, threads, 4096, (long long *)st);
            if (cudaMemcpy(h.data(), st, sizeof(long long) * 2 * blocks, cudaMemcpyDeviceToHost) != cudaSuccess) break;
            std::vector<double> mhz;
            for (int k = 0; k < blocks; k++)
                if (h[2 * k + 1] > 0) mhz.push_back(1e3 * (double)h[2 * k] / (double)h[2 * k + 1]);
            if (mhz.empty() || r <= best) continue;
            std::nth_element(mhz.begin(), mhz.begin() + mhz.size() / 2, mhz.end());
            best = r;
            best_mhz = mhz[mhz.size() / 2];
        }
    }
    cudaFree(buf);
    cudaFree(st);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return sim_fail(nullptr, SIM_ECUDA, std::string("sim_probe_fp64_pipe: ") + cudaGetErrorString(e));
    if (fma_per_s) *fma_per_s = best;
    if (sm_mhz) *sm_mhz = best_mhz;
    if (fma_per_clk_per_sm) *fma_per_clk_per_sm = best_mhz > 0 ? best / (sms * best_mhz * 1e6) : 0.0;
    return SIM_OK;
}

// ---- run report ----------------------------------------------------------------
}  // extern "C"

namespace {
struct Json {
    std::string out;
    bool first = true;
    void key(const char *k) {
        if (!first) out += ", ";
        first = false;
        out += '"';
        out += k;
        out += "\": ";
    }
    void num(const char *k, double v, const char *fmt = "%.17g") {
        char b[64];
        snprintf(b, sizeof b, fmt, v);
        key(k);
        out += (v == v && v - v == 0.0) ? b : "null";
    }
    void integer(const char *k, long long v) {
        key(k);
        out += std::to_string(v);
    }
    void str(const char *k, const char *v) {
        key(k);
        out += '"';
        out += v;
        out += '"';
    }
    void open(const char *k) {
        key(k);
        out += '{';
        first = true;
    }
    void close() {
        out += '}';
        first = false;
    }
};
void phase_json(Json &j, const char *name, double us, double bytes) {
    j.open(name);
    j.num("us", us, "%.3f");
    j.num("bytes", bytes, "%.0f");
    j.num("achieved_gbs", us > 0 ? bytes / us / 1e3 : 0.0, "%.1f");
    j.close();
}
}  // namespace

extern "C" {

sim_status sim_run_report(sim_t *s, char *buf, int64_t cap, int64_t *len) {
    if (!s || !len || (cap > 0 && !buf) || cap < 0) return SIM_EINVAL;
    const sim_options &o = s->opt;
    Json j;
    j.out = "{";
    j.open("grid");
    j.integer("nx", s->gd.nx);
    j.integer("ny", s->gd.ny);
    j.integer("nz", s->gd.nz);
    j.integer("cells", s->N);
    j.close();
    j.str("model", s->fc.model == 3 ? "black_oil" : "oil_water");
    j.integer("unknowns_per_cell", s->b);
    j.integer("wells", s->nwells);
    j.integer("rate_controlled_wells", s->nrate);
    j.open("options");
    j.str("precision", o.precision == SIM_PRECISION_MIXED ? "fp32_preconditioner" : "fp64");
    j.str("krylov", o.krylov == SIM_KRYLOV_BICGSTAB ? "bicgstab" : "fgmres");
    j.integer("gmres_m", o.gmres_m);
    j.integer("gmres_max_restarts", o.gmres_max_restarts);
    j.str("precond", o.precond == SIM_PRECOND_CPR ? "cpr" : o.precond == SIM_PRECOND_BJACOBI ? "block_jacobi" : "none");
    j.integer("cpr_stages", o.cpr_stages);
    j.str("decouple", o.decouple == SIM_DECOUPLE_ABF ? "abf" : "quasi_impes");
    j.str("stage2", o.stage2 == SIM_STAGE2_ILU0_RB ? "ilu0_red_black" : "block_jacobi");
    j.integer("amg_cycles", o.amg_cycles);
    j.num("lin_tol", o.lin_tol);
    j.num("newton_tol", o.newton_tol);
    j.integer("newton_max", o.newton_max);
    j.integer("max_cuts", o.max_cuts);
    j.str("forcing", o.forcing == SIM_FORCING_EW1 ? "ew1" : o.forcing == SIM_FORCING_EW2 ? "ew2"
                     : o.forcing == SIM_FORCING_EW3 ? "ew3" : "fixed");
    j.integer("graphs", o.graphs);
    j.integer("orth", o.orth);
    j.close();
    j.open("learned_stage");
    j.integer("enabled", s->learned_on && s->net ? 1 : 0);
    j.integer("fallbacks", s->learned_fallbacks);
    j.close();
    j.open("counters");
    j.integer("time_steps", s->run_steps);
    j.integer("failed_time_steps", s->run_failed_steps);
    j.integer("substeps", s->run_substeps);
    j.integer("cuts", s->run_cuts);
    j.num("simulated_days", s->run_days);
    j.integer("newton_iterations", s->newton_total);
    j.integer("linear_iterations", s->linear_total);
    j.integer("linear_solves_not_converged", s->run_lin_failures);
    j.num("max_mass_balance_error", s->run_max_mb, "%.3e");
    j.integer("kernel_launches", s->launches);
    j.close();
    const sim_phase_info &p = s->run_phase;
    j.open("phases");
    phase_json(j, "assemble", p.assemble_us, p.assemble_bytes);
    phase_json(j, "setup", p.setup_us, p.setup_bytes);
    phase_json(j, "solve", p.solve_us, p.solve_bytes);
    phase_json(j, "update", p.update_us, p.update_bytes);
    j.close();
    j.integer("device_bytes", (long long)s->bytes);
    j.open("launch_shapes");
    j.integer("spmv_block", s->tune_spmv);
    j.integer("amg_block", s->tune_amg);
    j.integer("stage_block", s->tune_stage);
    j.close();
    j.out += '}';
    *len = (int64_t)j.out.size();
    if (cap < *len + 1) return SIM_EINVAL;   // not sticky: the caller retries with *len + 1 bytes
    memcpy(buf, j.out.c_str(), j.out.size() + 1);
    return SIM_OK;
}

sim_status sim_get_stats(sim_t *s, sim_stats *st) {
    if (!s || !st) return SIM_EINVAL;
    st->kernel_launches = s->launches;
    st->newton_iterations = s->newton_total;
    st->linear_iterations = s->linear_total;
    st->device_bytes = (int64_t)s->bytes;
    st->spmv_block = s->tune_spmv;
    st->amg_block = s->tune_amg;
    st->stage_block = s->tune_stage;
    return SIM_OK;
}

sim_status sim_autotune(sim_t *s, double dt) {
    CHECK_HANDLE(s);
    if (!(dt > 0)) return sim_fail(s, SIM_EINVAL, "dt must be positive");
    if (k_assemble(s, dt) != SIM_OK) return s->err;
    const long n = (long)s->N * s->b;
    static const int spmv_cand[] = {64, 128, 256, 512};
    float best = 1e30f;
    int pick = s->tune_spmv;
    for (int bs : spmv_cand) {
        const float ms = time_launches(s, 5, [&] { k_spmv_block(s, s->bl, s->w, bs); });
        if (ms < best) { best = ms; pick = bs; }
    }
    s->tune_spmv = pick;
    if (s->opt.precond == SIM_PRECOND_CPR) {
        if (cpr_setup(s) != SIM_OK) return s->err;
        SIM_CK(s, cudaMemsetAsync(s->bl, 0, sizeof(double) * n, s->stream));
        static const int amg_cand[] = {64, 128, 256};
        best = 1e30f;
        pick = s->tune_amg;
        for (int bs : amg_cand) {
            s->tune_amg = bs;
            const float ms = time_launches(s, 3, [&] { cpr_apply(s, s->bl, s->Z, nullptr); });
            if (ms < best) { best = ms; pick = bs; }
        }
        s->tune_amg = pick;
        static const int stage_cand[] = {32, 64, 128, 256};
        best = 1e30f;
        pick = s->tune_stage;
        for (int bs : stage_cand) {
            s->tune_stage = bs;
            const float ms = time_launches(s, 3, [&] { cpr_apply(s, s->bl, s->Z, nullptr); });
            if (ms < best) { best = ms; pick = bs; }
        }
        s->tune_stage = pick;
    }
    s->setup_gen++;   // the captured restart cycle used the old launch shapes
    SIM_CK(s, cudaGetLastError());
    SIM_CK(s, cudaStreamSynchronize(s->stream));
    return SIM_OK;
}

// ---- launch shapes cached in a JSON file ---------------------------------
// one entry per line, {"b<b>_<fp64|mixed>_<nx>x<ny>x<nz>": {"spmv": S, "amg": A, "stage": F}}
static std::string tune_key(const sim_t *s) {
    char k[128];
    snprintf(k, sizeof(k), "b%d_%s_%dx%dx%d", s->b, sim_mixed(s) ? "mixed" : "fp64", s->gd.nx, s->gd.ny, s->gd.nz);
    return k;
}

struct TuneEntry { std::string key; int spmv, amg, stage; };

static std::vector<TuneEntry> read_tune_file(const char *path) {
    std::vector<TuneEntry> out;
    FILE *f = fopen(path, "r");
    if (!f) return out;
    char line[512], key[160];
    int a, b, c;
    while (fgets(line, sizeof(line), f)) {
        if (sscanf(line, " \"%159[^\"]\": {\"spmv\": %d, \"amg\": %d, \"stage\": %d}", key, &a, &b, &c) == 4)
            out.push_back(TuneEntry{key, a, b, c});
    }
    fclose(f);
    return out;
}

static bool shape_ok(int v, int lo, int hi) { return v >= lo && v <= hi && (v & (v - 1)) == 0; }

sim_status sim_autotune_cached(sim_t *s, double dt, const char *json_path, int32_t *from_cache) {
    CHECK_HANDLE(s);
    if (!json_path) return sim_fail(s, SIM_EINVAL, "sim_autotune_cached: NULL path");
    const std::string key = tune_key(s);
    std::vector<TuneEntry> tab = read_tune_file(json_path);
    for (const TuneEntry &e : tab) {
        if (e.key == key && shape_ok(e.spmv, 32, 512) && shape_ok(e.amg, 32, 1024) && shape_ok(e.stage, 32, 1024)) {
            s->tune_spmv = e.spmv; s->tune_amg = e.amg; s->tune_stage = e.stage;
            s->setup_gen++;
            if (from_cache) *from_cache = 1;
            return SIM_OK;
        }
    }
    if (sim_autotune(s, dt) != SIM_OK) return s->err;
    if (from_cache) *from_cache = 0;
    bool found = false;
    for (TuneEntry &e : tab)
        if (e.key == key) { e.spmv = s->tune_spmv; e.amg = s->tune_amg; e.stage = s->tune_stage; found = true; }
    if (!found) tab.push_back(TuneEntry{key, s->tune_spmv, s->tune_amg, s->tune_stage});
    // write a new file and move it over the old one (readers never see half a file)
    const std::string tmp = std::string(json_path) + ".tmp";
    FILE *f = fopen(tmp.c_str(), "w");
    if (!f) return sim_fail(s, SIM_EINVAL, std::string("sim_autotune_cached: cannot write ") + tmp);
    fprintf(f, "{\n");
    for (size_t i = 0; i < tab.size(); i++)
        fprintf(f, "\"%s\": {\"spmv\": %d, \"amg\": %d, \"stage\": %d}%s\n", tab[i].key.c_str(), tab[i].spmv,
                tab[i].amg, tab[i].stage, i + 1 < tab.size() ? "," : "");
    fprintf(f, "}\n");
    const bool ok = fclose(f) == 0 && rename(tmp.c_str(), json_path) == 0;
    if (!ok) return sim_fail(s, SIM_EINVAL, std::string("sim_autotune_cached: cannot replace ") + json_path);
    return SIM_OK;
}

}  // extern "C"
