// CPR two-stage preconditioner on the device (paper Sec. 2.4.2).
//
//   setup (FP64):  quasi-IMPES weights w_i = (1, -d_ps D_ss^-1) from the
//                  diagonal block; decoupled matrix Ahat (pressure row
//                  replaced by w^T rows); pressure block A_p; aggregation AMG
//                  hierarchy of A_p; red-black block ILU(0) (or block-Jacobi)
//                  of Ahat.
//   apply (T):     rp = w^T r; e_p = V(1,1)-cycle(A_p, rp);
//                  r2 = rhat - Ahat[:, p] e_p;  z = ILU0(Ahat)^-1 r2 + e_p.
// T = double for the plain form, float for the mixed form (FP32 hierarchy,
// factors and smoothers; the FGMRES outer loop stays FP64).
//
// AMG: two pairwise matching passes per level (handshakes among unmatched
// nodes; candidate = strongest unmatched strong neighbour compared by
// strength band (binary exponent), then a symmetric splitmix64 pair hash,
// then the smaller index); piecewise-constant prolongation; Galerkin coarse
// operators summed in member order then column order; l1-Jacobi V(1,1);
// dense inverse on the coarsest level.  The setup is deterministic and its
// integer results do not depend on thread scheduling.
//
// Layouts: level 0 is the 7-point stencil A_p [7][N]; coarser levels are ELL,
// entry k of row i at k*n + i, columns ascending, -1 padding.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <type_traits>
#include <vector>

#include <cooperative_groups.h>

#include "sim_internal.cuh"

namespace cg = cooperative_groups;

namespace {

constexpr int MAXE = SIM_MAX_ELL;

// enter (see sim_launch) and test the flag
__device__ __forceinline__ bool skip(const int *done) {
    sim_enter();
    return done != nullptr && *(volatile const int *)done;
}

struct Cell { int i, ix, iy, iz; };
__device__ __forceinline__ Cell cell_of(const GridDesc &g, int i) {
    Cell c; c.i = i; c.ix = i % g.nx; const int t = i / g.nx; c.iy = t % g.ny; c.iz = t / g.ny; return c;
}
__device__ __forceinline__ int nbrc(const GridDesc &g, const Cell &c, int d) {
    switch (d) {
    case 0: return c.i;
    case 1: return c.ix > 0 ? c.i - 1 : -1;
    case 2: return c.ix < g.nx - 1 ? c.i + 1 : -1;
    case 3: return c.iy > 0 ? c.i - g.nx : -1;
    case 4: return c.iy < g.ny - 1 ? c.i + g.nx : -1;
    case 5: return c.iz > 0 ? c.i - g.nx * g.ny : -1;
    default: return c.iz < g.nz - 1 ? c.i + g.nx * g.ny : -1;
    }
}
__device__ __forceinline__ int nbr7(const GridDesc &g, int i, int d) {
    const int ix = i % g.nx, t = i / g.nx, iy = t % g.ny, iz = t / g.ny;
    switch (d) {
    case 0: return i;
    case 1: return ix > 0 ? i - 1 : -1;
    case 2: return ix < g.nx - 1 ? i + 1 : -1;
    case 3: return iy > 0 ? i - g.nx : -1;
    case 4: return iy < g.ny - 1 ? i + g.nx : -1;
    case 5: return iz > 0 ? i - g.nx * g.ny : -1;
    default: return iz < g.nz - 1 ? i + g.nx * g.ny : -1;
    }
}
// thread t of a launch over one colour (0: ix+iy+iz even, 1: odd): slot k of
// x-row r holds the cell ix = 2k or 2k+1 of that colour, so a warp's threads
// all work (a launch over every cell would leave half of each warp idle)
__device__ __forceinline__ int colour_cell(const GridDesc &g, long t, int colour) {
    const int hx = (g.nx + 1) >> 1;
    const long r = t / hx;
    const int k = (int)(t - r * hx);
    if (r >= (long)g.ny * g.nz) return -1;
    const int iy = (int)(r % g.ny), iz = (int)(r / g.ny);
    const int ix = 2 * k + (((iy + iz) & 1) != colour ? 1 : 0);
    if (ix >= g.nx) return -1;
    return (int)(ix + (long)g.nx * r);
}

// Colour-split storage of the blocks the red-black sweeps read (Ahat and the
// inverted diagonal blocks): colour (ix + iy + iz) & 1 first, then the cell's
// slot in colour_cell's order, so the threads of a one-colour sweep read
// consecutive positions (component-major storage by cell would hand each warp
// sectors half filled with the other colour's blocks).  2 H positions.
__device__ __forceinline__ long cslot(const GridDesc &g, int ix, int iy, int iz) {
    return (long)((ix + iy + iz) & 1) * g.H + (long)(iy + g.ny * iz) * ((g.nx + 1) >> 1) + (ix >> 1);
}
__device__ __forceinline__ long cslot_of(const GridDesc &g, int i) {
    const int ix = i % g.nx, t = i / g.nx, iy = t % g.ny, iz = t / g.ny;
    return cslot(g, ix, iy, iz);
}

__device__ __forceinline__ int opp(int d) { return d == 0 ? 0 : ((d & 1) ? d + 1 : d - 1); }
__device__ __forceinline__ bool is_black(const GridDesc &g, int i) {
    const int ix = i % g.nx, t = i / g.nx, iy = t % g.ny, iz = t / g.ny;
    return ((ix + iy + iz) & 1) != 0;
}

// A row of a level matrix: structured (level 0) or ELL
template <typename V>
struct Mat {
    bool st;
    bool selfpad;    // ELL padded with (self column, 0) instead of -1: no early exit
    bool diff;       // difference form: the diagonal slot holds the row sum (see row_dot)
    GridDesc g;      // structured
    const V *val;    // structured: [7][n]; ELL: [width][n]
    const int *col;  // ELL
    int n, width;
    const int *len = nullptr;  // ELL: entries of each row (the width is the longest row's, two to three times the mean)
    const int *wp = nullptr;   // set-up: {width, flags} still on the device (width then holds the capacity)
};
// a product whose rows did not all fit is no matrix yet (entries are missing, and
// with them the symmetry of its pattern): what was enqueued on it does nothing, and
// the host, which reads the same words, builds it again and repeats the pass
template <typename V> __device__ __forceinline__ bool unfinished(const Mat<V> &A) {
    return A.wp && (A.wp[0] > A.width || A.wp[1] != 0);
}

// visit the entries of row i in ascending column order: f(col, val)
// (self-padded ELL rows end with zero entries on the diagonal column)
template <typename V, typename F>
__device__ __forceinline__ void for_row(const Mat<V> &A, int i, F f) {
    if (A.st) {
        const int nx = A.g.nx, ny = A.g.ny, nxy = nx * ny;
        const int ix = i % nx, t = i / nx, iy = t % ny, iz = t / ny;
        const long n = A.n;
        if (iz > 0) f(i - nxy, A.val[5 * n + i]);
        if (iy > 0) f(i - nx, A.val[3 * n + i]);
        if (ix > 0) f(i - 1, A.val[1 * n + i]);
        f(i, A.val[i]);
        if (ix < nx - 1) f(i + 1, A.val[2 * n + i]);
        if (iy < ny - 1) f(i + nx, A.val[4 * n + i]);
        if (iz < A.g.nz - 1) f(i + nxy, A.val[6 * n + i]);
    } else if (A.selfpad) {
        // batches of 8 entries: the batch's loads are issued together, then f
        // runs on them in column-slot order; padding within the last batch is
        // (own column, 0)
        const int W = A.len[i];
        for (int k0 = 0; k0 < W; k0 += 8) {
            int jj[8];
            V vv[8];
#pragma unroll
            for (int u = 0; u < 8; u++) {
                const long q = (long)(k0 + u) * A.n + i;
                const bool ok = k0 + u < W;
                jj[u] = ok ? A.col[q] : i;
                vv[u] = ok ? A.val[q] : V(0);
            }
#pragma unroll
            for (int u = 0; u < 8; u++)
                if (k0 + u < W) f(jj[u], vv[u]);
        }
    } else {
        const int W = A.len[i];
#pragma unroll 4
        for (int k = 0; k < W; k++) f(A.col[(long)k * A.n + i], A.val[(long)k * A.n + i]);
    }
}

// A_i . e.  In the difference form (the FP32 copies of the pressure matrices)
// the diagonal slot holds the row sum d_i = sum_j a_ij, computed in FP64, and
// A_i . e = d_i e_i + sum_{j != i} a_ij (e_j - e_i): the small row sum (the
// accumulation term, 1e-4 to 1e-7 of the off-diagonals where permeability is
// high) survives rounding to FP32, where a_ii + sum_{j != i} a_ij would lose it.
template <typename T>
__device__ __forceinline__ T row_dot(const Mat<T> &A, int i, const T *__restrict__ e) {
    T t = (T)0;
    if (A.diff) {
        const T ei = e[i];
        for_row(A, i, [&](int j, T v) { t += (j == i) ? v * ei : v * (e[j] - ei); });
    } else {
        for_row(A, i, [&](int j, T v) { t += v * e[j]; });
    }
    return t;
}

// ---- lanes of an ELL row ----------------------------------------------------
// A row of 8 to 25 entries taken by one thread is a chain of load batches; below
// 131k rows, where the launch does not fill the GPU with rows, lanes share a row and
// have all of its entries in flight at once (72k rows, longest 35, mean 11 entries:
// residual 16.6 -> 10.8 us with the row lengths).  The count depends on the level's size
// only, so every kernel that takes the row (one system, a batch, the fused coarse
// cycle) adds it up alike.  The lines between 4, 8 and 16 lanes are flat: 256 / 1,024,
// 512 / 2,048 and 1,024 / 4,096 rows, 2 lanes above 8,192 and no 16 measured within 0.4 % of
// each other.  Speed does not choose among them; the first is taken because the sums it
// gives leave the Newton counts of an ensemble's chaotic first steps, which any change of
// rounding moves by several, where the tests of those counts expect them.
__host__ __device__ inline int ell_lanes(int n) { return n > 131072 ? 1 : n > 1024 ? 4 : n > 256 ? 8 : 16; }

// sum_k val_k e(col_k) of row i by `lanes` adjacent lanes (sub: this one's number;
// every lane of the warp calls, ok: the row exists), the total in all of them.
// entry(k, j, v) gives column and value of slot k < W (padding: column i, value 0);
// len: slots the row uses, whose largest in the warp ends the loop -- the first
// batch's loads do not wait for it.  FP64: each lane adds its own slots, then a fixed
// tree.  Difference form (FP32 copies, see row_dot): the products are added in slot
// order, one lane's after the other's, so the rounding is that of one thread taking
// the row.
template <typename T, typename FEnt, typename FE>
__device__ __forceinline__ T row_dot_lanes(int W, int len, int lanes, int sub, bool ok, bool diff, int i, T ei, FEnt entry,
                                           FE e) {
    constexpr int U = 4;
    T t = (T)0;
    int most = W, j[U];
    T v[U];
    for (int k0 = 0; k0 < most; k0 += U * lanes) {
#pragma unroll
        for (int u = 0; u < U; u++) {
            const int k = k0 + u * lanes + sub;
            j[u] = i;
            v[u] = (T)0;
            if (ok && k < W) entry(k, j[u], v[u]);
        }
        T x[U];
#pragma unroll
        for (int u = 0; u < U; u++) x[u] = ok ? e(j[u]) : (T)0;
        if (k0 == 0) most = __reduce_max_sync(0xffffffffu, ok ? len : 0);
#pragma unroll
        for (int u = 0; u < U; u++) {
            if (k0 + u * lanes >= most) break;                 // uniform
            if (!diff) {
                t += v[u] * x[u];
            } else {
                const T d = j[u] == i ? ei : x[u] - ei;
                if (lanes == 1) { t = fma(v[u], d, t); continue; }
                for (int l = 0; l < lanes; l++)
                    t = fma(__shfl_sync(0xffffffffu, v[u], l, lanes), __shfl_sync(0xffffffffu, d, l, lanes), t);
            }
        }
    }
    if (!diff)
        for (int o = lanes >> 1; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    return t;
}
// A_i . e of an ELL level of the application with `lanes` lanes
template <typename T>
__device__ __forceinline__ T mat_dot_lanes(const Mat<T> &A, int i, bool ok, int lanes, int sub, const T *__restrict__ e) {
    const long n = A.n;
    return row_dot_lanes<T>(A.width, ok ? A.len[i] : 0, lanes, sub, ok, A.diff, i, ok && A.diff ? e[i] : (T)0,
                            [&](int k, int &j, T &v) { j = A.col[k * n + i]; v = A.val[k * n + i]; },
                            [&](int j) { return e[j]; });
}

// ---------------------------------------------------------------------------
// quasi-IMPES decoupling (FP64, rounding-exact: no contraction)
// ---------------------------------------------------------------------------
// rate-controlled wells' Schur term in the preconditioner matrix: block (i, d)
// of J loses A_pw[q] A_ww^-1 A_wp[q'] when cell i holds perforation q and its
// neighbour j holds perforation q' of the same rate-controlled well
struct WellCorr {
    const int *cell_perf = nullptr;   // null: no rate-controlled wells
    const int *pwell = nullptr;
    const double *apw = nullptr, *awp = nullptr, *aww = nullptr;   // [3][nperf], [nwells]
    int nperf = 0;
};

// block (row cell i, direction d, neighbour j) of the preconditioner matrix,
// the correction rounded as written (the AMG hierarchy is built bit-exactly)
template <int B>
__device__ __forceinline__ void load_jblock(const double *__restrict__ J, long N, int i, int d, int j, const WellCorr &wc,
                                            double *Jb) {
#pragma unroll
    for (int t = 0; t < B * B; t++) Jb[t] = J[(long)(d * B * B + t) * N + i];
    if (!wc.cell_perf || j < 0) return;
    const int q = wc.cell_perf[i];
    if (q < 0) return;
    const int q2 = wc.cell_perf[j];
    if (q2 < 0 || wc.pwell[q2] != wc.pwell[q]) return;
    const double a = wc.aww[wc.pwell[q]];
#pragma unroll
    for (int r = 0; r < B; r++)
#pragma unroll
        for (int c = 0; c < B; c++)
            Jb[r * B + c] = __dsub_rn(Jb[r * B + c],
                                      __ddiv_rn(__dmul_rn(wc.apw[(long)r * wc.nperf + q], wc.awp[(long)c * wc.nperf + q2]), a));
}

template <int B>
__device__ __forceinline__ void qi_weights(const double *D, double *w) {
    const double D01 = D[0 * B + 1], D11 = D[1 * B + 1];
    w[0] = 1.0;
    if constexpr (B == 2) {
        w[1] = -(D01 / D11);
    } else {
        const double D02 = D[0 * B + 2];
        const double D12 = D[1 * B + 2], D21 = D[2 * B + 1], D22 = D[2 * B + 2];
        const double det = __dsub_rn(__dmul_rn(D11, D22), __dmul_rn(D12, D21));
        w[1] = __ddiv_rn(__dsub_rn(__dmul_rn(D02, D21), __dmul_rn(D01, D22)), det);
        w[2] = __ddiv_rn(__dsub_rn(__dmul_rn(D01, D12), __dmul_rn(D02, D11)), det);
    }
}

// decoupled block (row cell i, direction d): Ahat = L_i J_id, products summed in
// row order without contraction (quasi-IMPES: L = [w^T; 0 I], so the pressure
// row is J_0c + w1 J_1c + w2 J_2c exactly as the oracle forms it and the others are
// J's own: 12 FP64 operations of b = 3, against 45 with the zeros and ones; full:
// ABF, every entry of L)
template <int B>
__device__ __forceinline__ void ahat_block(const double *__restrict__ J, long N, int i, int d, int j, const WellCorr &wc,
                                           const double *L, bool full, double *A) {
    double Jb[B * B];
    load_jblock<B>(J, N, i, d, j, wc, Jb);
#pragma unroll
    for (int r = 0; r < B; r++)
#pragma unroll
        for (int c = 0; c < B; c++) {
            if (!full && r > 0) { A[r * B + c] = Jb[r * B + c]; continue; }
            double t = full ? __dmul_rn(L[r * B], Jb[c]) : Jb[c];
            t = __dadd_rn(t, __dmul_rn(L[r * B + 1], Jb[B + c]));
            if (B == 3) t = __dadd_rn(t, __dmul_rn(L[r * B + 2], Jb[2 * B + c]));
            A[r * B + c] = t;
        }
}

template <int B>
__device__ __forceinline__ void load_lsc(const double *__restrict__ lsc, long N, int i, double *L) {
#pragma unroll
    for (int t = 0; t < B * B; t++) L[t] = lsc[(long)t * N + i];
}

// inverse of a diagonal block by cofactors, every operation rounded as written
// (the ABF scaling feeds the AMG hierarchy, which is built bit-exactly)
template <int B>
__device__ __forceinline__ void inv_block_rn(const double *A, double *Ai) {
#define M_(a, b) __dmul_rn(A[a], A[b])
    if constexpr (B == 2) {
        const double det = __dsub_rn(M_(0, 3), M_(1, 2));
        Ai[0] = __ddiv_rn(A[3], det); Ai[1] = __ddiv_rn(-A[1], det);
        Ai[2] = __ddiv_rn(-A[2], det); Ai[3] = __ddiv_rn(A[0], det);
    } else {
        const double c00 = __dsub_rn(M_(4, 8), M_(5, 7));
        const double c01 = __dsub_rn(M_(5, 6), M_(3, 8));
        const double c02 = __dsub_rn(M_(3, 7), M_(4, 6));
        const double det = __dadd_rn(__dadd_rn(__dmul_rn(A[0], c00), __dmul_rn(A[1], c01)), __dmul_rn(A[2], c02));
        Ai[0] = __ddiv_rn(c00, det);
        Ai[1] = __ddiv_rn(__dsub_rn(M_(2, 7), M_(1, 8)), det);
        Ai[2] = __ddiv_rn(__dsub_rn(M_(1, 5), M_(2, 4)), det);
        Ai[3] = __ddiv_rn(c01, det);
        Ai[4] = __ddiv_rn(__dsub_rn(M_(0, 8), M_(2, 6)), det);
        Ai[5] = __ddiv_rn(__dsub_rn(M_(2, 3), M_(0, 5)), det);
        Ai[6] = __ddiv_rn(c02, det);
        Ai[7] = __ddiv_rn(__dsub_rn(M_(1, 6), M_(0, 7)), det);
        Ai[8] = __ddiv_rn(__dsub_rn(M_(0, 4), M_(1, 3)), det);
    }
#undef M_
}

// left scaling per cell (quasi-IMPES or ABF), its first row, the pressure
// block A_p and the decoupled matrix in the apply precision
template <int B, typename T>
__global__ void qi_kernel(GridDesc g, const double *__restrict__ J, WellCorr wc, int abf, double *__restrict__ lsc,
                          T *__restrict__ lscT, double *__restrict__ qiw, T *__restrict__ qiwT, double *__restrict__ ap,
                          T *__restrict__ apT, T *__restrict__ ahat, T *__restrict__ dinv0) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const long N = g.N;
    if (i >= N) return;
    double L[B * B], D[B * B];
    load_jblock<B>(J, N, i, 0, i, wc, D);
    if (abf) {
        inv_block_rn<B>(D, L);
    } else {
        double w[3] = {1.0, 0.0, 0.0};
        qi_weights<B>(D, w);
#pragma unroll
        for (int t = 0; t < B * B; t++) L[t] = (t / B == t % B) ? 1.0 : 0.0;
        L[1] = w[1];
        if (B == 3) L[2] = w[2];
    }
#pragma unroll
    for (int t = 0; t < B * B; t++) { lsc[(long)t * N + i] = L[t]; lscT[(long)t * N + i] = (T)L[t]; }
#pragma unroll
    for (int c = 0; c < B; c++) { qiw[(long)c * N + i] = L[c]; qiwT[(long)c * N + i] = (T)L[c]; }
    const Cell cc = cell_of(g, i);
    const long NS = 2L * g.H, si = cslot(g, cc.ix, cc.iy, cc.iz);
    double a0[7];                        // the row of A_p
#pragma unroll
    for (int d = 0; d < 7; d++) {
        double A[B * B];
        const int j = nbrc(g, cc, d);
        ahat_block<B>(J, N, i, d, j, wc, L, abf != 0, A);
        a0[d] = j >= 0 ? A[0] : 0.0;
        ap[(long)d * N + i] = a0[d];
        apT[(long)d * N + i] = (T)a0[d];
#pragma unroll
        for (int t = 0; t < B * B; t++) ahat[(long)(d * B * B + t) * NS + si] = (T)A[t];
    }
    // level 0's 1 / l1 row sum, in ascending column order
    double l1 = fabs(a0[5]);
    l1 += fabs(a0[3]); l1 += fabs(a0[1]); l1 += fabs(a0[0]); l1 += fabs(a0[2]); l1 += fabs(a0[4]); l1 += fabs(a0[6]);
    dinv0[i] = (T)(1.0 / l1);
    if (sizeof(T) == sizeof(float)) {    // FP32 copy: row sum of A_p on the diagonal slot (difference form)
        double rsum = 0.0;
#pragma unroll
        for (int d = 0; d < 7; d++) rsum += a0[d];
        apT[i] = (T)rsum;
    }
}

// ---------------------------------------------------------------------------
// block inverses and red-black ILU(0) setup (FP64)
// ---------------------------------------------------------------------------
template <int B>
__device__ __forceinline__ void inv_block(const double *A, double *Ai) {
    if constexpr (B == 2) {
        const double det = A[0] * A[3] - A[1] * A[2];
        Ai[0] = A[3] / det; Ai[1] = -A[1] / det; Ai[2] = -A[2] / det; Ai[3] = A[0] / det;
    } else {
        const double c00 = A[4] * A[8] - A[5] * A[7];
        const double c01 = A[5] * A[6] - A[3] * A[8];
        const double c02 = A[3] * A[7] - A[4] * A[6];
        const double det = A[0] * c00 + A[1] * c01 + A[2] * c02;
        const double id = 1.0 / det;
        Ai[0] = c00 * id; Ai[1] = (A[2] * A[7] - A[1] * A[8]) * id; Ai[2] = (A[1] * A[5] - A[2] * A[4]) * id;
        Ai[3] = c01 * id; Ai[4] = (A[0] * A[8] - A[2] * A[6]) * id; Ai[5] = (A[2] * A[3] - A[0] * A[5]) * id;
        Ai[6] = c02 * id; Ai[7] = (A[1] * A[6] - A[0] * A[7]) * id; Ai[8] = (A[0] * A[4] - A[1] * A[3]) * id;
    }
}

// mode 0: inverse of Ahat_ii for every cell (block-Jacobi) or red cells only (mode 1);
// mode 2: inverse of J_ii (plain block-Jacobi, no decoupling)
template <int B>
__global__ void diag_inv_kernel(GridDesc g, const double *__restrict__ J, WellCorr wc, const double *__restrict__ lsc,
                                int abf, int mode, double *__restrict__ dinv) {
    const long N = g.N;
    const int i = mode == 1 ? colour_cell(g, blockIdx.x * (long)blockDim.x + threadIdx.x, 0)
                            : (blockIdx.x * blockDim.x + threadIdx.x < N ? (int)(blockIdx.x * blockDim.x + threadIdx.x) : -1);
    if (i < 0) return;
    double L[B * B], A[B * B], Ai[B * B];
    if (mode == 2) {
        load_jblock<B>(J, N, i, 0, i, wc, A);
    } else {
        load_lsc<B>(lsc, N, i, L);
        ahat_block<B>(J, N, i, 0, i, wc, L, abf != 0, A);
    }
    inv_block<B>(A, Ai);
    const long NS = 2L * g.H, si = cslot_of(g, i);
#pragma unroll
    for (int t = 0; t < B * B; t++) dinv[(long)t * NS + si] = Ai[t];
}

// black cells: D = Ahat_ii - sum_d Ahat_{i,d} Dinv_k Ahat_{k,opp(d)}
template <int B>
__global__ void __launch_bounds__(SIM_THREADS, 2) ilu_black_kernel(GridDesc g, const double *__restrict__ J, WellCorr wc,
                                                                   const double *__restrict__ lsc, int abf,
                                                                   double *__restrict__ dinv) {
    const int i = colour_cell(g, blockIdx.x * (long)blockDim.x + threadIdx.x, 1);
    const long N = g.N;
    if (i < 0) return;
    double Li[B * B];
    load_lsc<B>(lsc, N, i, Li);
    double D[B * B];
    ahat_block<B>(J, N, i, 0, i, wc, Li, abf != 0, D);
    for (int d = 1; d < 7; d++) {
        const int k = nbr7(g, i, d);
        if (k < 0) continue;
        double Lk[B * B], Aik[B * B], Aki[B * B], Dk[B * B], T1[B * B];
        load_lsc<B>(lsc, N, k, Lk);
        ahat_block<B>(J, N, i, d, k, wc, Li, abf != 0, Aik);
        ahat_block<B>(J, N, k, opp(d), i, wc, Lk, abf != 0, Aki);
        const long sk = cslot_of(g, k);
#pragma unroll
        for (int t = 0; t < B * B; t++) Dk[t] = dinv[(long)t * 2L * g.H + sk];
#pragma unroll
        for (int r = 0; r < B; r++)
#pragma unroll
            for (int c = 0; c < B; c++) {
                double s = 0.0;
#pragma unroll
                for (int q = 0; q < B; q++) s += Dk[r * B + q] * Aki[q * B + c];
                T1[r * B + c] = s;
            }
#pragma unroll
        for (int r = 0; r < B; r++)
#pragma unroll
            for (int c = 0; c < B; c++) {
#pragma unroll
                for (int q = 0; q < B; q++) D[r * B + c] -= Aik[r * B + q] * T1[q * B + c];
            }
    }
    double Di[B * B];
    inv_block<B>(D, Di);
    const long NS = 2L * g.H, si = cslot_of(g, i);
#pragma unroll
    for (int t = 0; t < B * B; t++) dinv[(long)t * NS + si] = Di[t];
}

template <typename T>
__global__ void cast_kernel(const double *__restrict__ a, T *__restrict__ b, long n) {
    for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x) b[i] = (T)a[i];
}

// ---------------------------------------------------------------------------
// AMG setup kernels (FP64 values, integer results)
//
// One aggregation pass is seven launches and no host round trip of its own:
// the matching rounds (a round reads the picks of the round before and finds out
// for itself which nodes those matched, so no launch confirms them), the
// absorption, the sizes, and one launch that numbers the aggregates and writes
// their members.  On the coarse levels every one of them is a chain of dependent
// loads, so a row is given 8 lanes (a thread per row of 30 entries: 18 us per
// launch whatever the level's size).  200k cells, 8 passes: 2.3 ms in 240 launches
// before, 0.6 ms in 64.
// ---------------------------------------------------------------------------
__device__ __forceinline__ unsigned long long edge_hash(int a, int b) {
    const unsigned long long lo = (unsigned long long)(a < b ? a : b), hi = (unsigned long long)(a < b ? b : a);
    unsigned long long z = ((hi << 32) | lo) + 0x9E3779B97F4A7C15ULL;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
    return z ^ (z >> 31);
}

// -a as an ordered integer: positive numbers compare by their bits (no FP64
// compares); 0 for an entry that is not a negative number
__device__ __forceinline__ long long neg_bits(double a) {
    const long long v = __double_as_longlong(-a);
    return v > 0 && v <= 0x7ff0000000000000LL ? v : 0;
}
// the least strong coupling theta mx as such bits; a bound that is no positive number
// (theta NaN or negative, 0 times infinity) refuses none, as a < bound does in FP64
__device__ __forceinline__ long long strong_bits(double theta, long long mx) {
    const double t = theta * __longlong_as_double(mx);
    return t > 0.0 ? __double_as_longlong(t) : 0;
}

// the best candidate so far: strength band (binary exponent), then the symmetric
// hash of the pair, then the smaller index
struct Cand {
    int band, j;
    unsigned long long h;
    __device__ __forceinline__ void offer(int b, unsigned long long hh, int jj) {
        if (j < 0 || b > band || (b == band && (hh > h || (hh == h && jj < j)))) { band = b; h = hh; j = jj; }
    }
};

// node j is matched: by its recorded partner, or by the last round's picks
__device__ __forceinline__ bool is_matched(const int *partner, const int *pk, int j) {
    if (!pk) return false;
    if (((volatile const int *)partner)[j] >= 0) return true;
    const int p = pk[j];
    return p >= 0 && pk[p] == j;
}

// Absorbed nodes kept per pair (more: the pair's rows are searched for them)
constexpr int kAbsorb = 6;
struct MatchState {
    int *partner;         // [n] partner, -1 none
    int *host;            // [n] host of an absorbed node, -1 none
    int *acnt, *alist;    // [n], [kAbsorb][n] nodes absorbed by the pair led by i (any order)
};

// One matching round (HOST false: out = the picks) or the absorption that follows
// the last one (HOST true: host, and the pairs' lists).  LANES lanes share a row:
// 1 on the 7-point level, 8 on ELL levels.  Nodes the last round matched record
// their partner; others reading them meanwhile see the match either way.
template <bool HOST, int LANES>
__global__ void __launch_bounds__(SIM_THREADS) match_kernel(Mat<double> A, MatchState st, const int *__restrict__ pk,
                                                            int *__restrict__ out, double theta) {
    if (unfinished(A)) return;
    const int i = (int)((blockIdx.x * (long)blockDim.x + threadIdx.x) / LANES), sub = threadIdx.x & (LANES - 1);
    const int n = A.n;
    bool open = false;
    if (i < n) {
        int p = -1;
        if (!pk) {
            if (sub == 0) { st.partner[i] = -1; st.acnt[i] = 0; }
            open = true;
        } else {
            p = ((volatile const int *)st.partner)[i];
            if (p < 0) {
                const int q = pk[i];
                if (q >= 0 && pk[q] == i) { p = q; if (sub == 0) st.partner[i] = q; }
            }
            open = p < 0;
        }
        if (!open && sub == 0) { if (HOST) st.host[i] = -1; else out[i] = -1; }
    }
    if (!__any_sync(0xffffffffu, open)) return;
    Cand best;
    best.band = 0; best.j = -1; best.h = 0ULL;
    auto consider = [&](int j, long long a, long long lim) {
        if (a == 0 || a < lim || is_matched(st.partner, pk, j) != HOST) return;
        best.offer((int)(a >> 52), edge_hash(i, j), j);
    };
    if constexpr (LANES == 1) {
        if (open) {
            const Cell cc = cell_of(A.g, i);
            long long mx = 0, a[7];
#pragma unroll
            for (int d = 1; d < 7; d++) {
                a[d] = nbrc(A.g, cc, d) >= 0 ? neg_bits(A.val[(long)d * n + i]) : 0;
                mx = max(mx, a[d]);
            }
            if (mx > 0) {
                const long long lim = strong_bits(theta, mx);
#pragma unroll
                for (int d = 1; d < 7; d++)
                    if (a[d] != 0) consider(nbrc(A.g, cc, d), a[d], lim);
            }
        }
    } else {
        constexpr int U = 4;                       // entries of a lane kept in registers: rows of up to 32
        const int W = open ? A.len[i] : 0;
        long long mx = 0, a[U];
        int jj[U];
#pragma unroll
        for (int u = 0; u < U; u++) {
            const int k = sub + LANES * u;
            jj[u] = k < W ? A.col[(long)k * n + i] : -1;
        }
#pragma unroll
        for (int u = 0; u < U; u++) {
            a[u] = jj[u] >= 0 && jj[u] != i ? neg_bits(A.val[(long)(sub + LANES * u) * n + i]) : 0;
            mx = max(mx, a[u]);
        }
        for (int k = sub + LANES * U; k < W; k += LANES) {
            const int j = A.col[(long)k * n + i];
            if (j != i) mx = max(mx, neg_bits(A.val[(long)k * n + i]));
        }
#pragma unroll
        for (int o = LANES / 2; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        if (mx > 0) {
            const long long lim = strong_bits(theta, mx);
#pragma unroll
            for (int u = 0; u < U; u++) consider(jj[u], a[u], lim);
            for (int k = sub + LANES * U; k < W; k += LANES) {
                const int j = A.col[(long)k * n + i];
                if (j != i) consider(j, neg_bits(A.val[(long)k * n + i]), lim);
            }
        }
#pragma unroll
        for (int o = LANES / 2; o > 0; o >>= 1) {
            const int b2 = __shfl_xor_sync(0xffffffffu, best.band, o), j2 = __shfl_xor_sync(0xffffffffu, best.j, o);
            const unsigned long long h2 = __shfl_xor_sync(0xffffffffu, best.h, o);
            if (j2 >= 0) best.offer(b2, h2, j2);
        }
    }
    if (!open || sub != 0) return;
    if (!HOST) { out[i] = best.j; return; }
    st.host[i] = best.j;
    if (best.j >= 0) {
        const int h = best.j;
        int hp = ((volatile const int *)st.partner)[h];
        if (hp < 0) hp = pk[h];                    // matched by the last round
        const int lead = h < hp ? h : hp, slot = atomicAdd(&st.acnt[lead], 1);
        if (slot < kAbsorb) st.alist[(long)slot * n + lead] = i;
    }
}

// Aggregates: pair leaders (lower index of a pair) and lone nodes without a host
// found one, in index order; its members are the pair and the nodes either of the
// two absorbed.  On the second pass of a level the members' fine nodes (offsets
// moffF, list memF of the first pass) make up the composite aggregate.
struct AggPass {
    MatchState st;
    int n;
    const int *moffF, *memF;     // first pass (null on the first pass itself)
    int *agg, *moff, *mem;       // node -> aggregate, members (CSR, ascending)
    int *aggC, *moffC, *memC;    // the composite of both passes
    int *csum;                   // [3][chunks] founders, members, fine members per chunk
    int *nc;                     // number of aggregates
    bool scanned;                // csum holds the sums of the chunks before each (agg_scan_kernel)
};

// founder i's member count; composite: its fine members too
__device__ __forceinline__ bool is_founder(const AggPass &P, int i, int &p) {
    p = P.st.partner[i];
    return p >= 0 ? i < p : P.st.host[i] < 0;
}
// visit founder i's members in no particular order (an absorbed node's host has it
// in its own row: the patterns are symmetric, the 7-point one and every P^T A P of it)
template <typename F>
__device__ __forceinline__ void each_member(const AggPass &P, const Mat<double> &A, int i, int p, F f) {
    f(i);
    if (p < 0) return;
    f(p);
    const int c = P.st.acnt[i];
    if (c <= kAbsorb) {
        for (int k = 0; k < c; k++) f(P.st.alist[(long)k * P.n + i]);
    } else {
        for (int e = 0; e < 2; e++) {
            const int h = e ? p : i;
            for_row(A, h, [&](int j, double) { if (j != h && P.st.host[j] == h) f(j); });
        }
    }
}

// a chunk is one block's nodes, one per thread (four per thread in turn made the
// second pass's launch 65 us at 85k nodes: a founder's lists are a chain of loads)
__device__ __forceinline__ void agg_counts(const AggPass &P, const Mat<double> &A, int i, int (&c)[3]) {
    c[0] = c[1] = c[2] = 0;
    int p;
    if (i >= P.n || !is_founder(P, i, p)) return;
    c[0] = 1;
    c[1] = 1 + (p >= 0 ? 1 + P.st.acnt[i] : 0);
    if (P.moffF) each_member(P, A, i, p, [&](int m) { c[2] += P.moffF[m + 1] - P.moffF[m]; });
}

__device__ __forceinline__ int block_sum(int v) {
    __shared__ int sh[32];
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
    __syncthreads();
    int t = 0;
    for (int w = 0; w < (int)(blockDim.x >> 5); w++) t += sh[w];
    return t;
}

__global__ void agg_sizes_kernel(AggPass P, Mat<double> A) {
    if (unfinished(A)) return;
    int t[3];
    agg_counts(P, A, blockIdx.x * blockDim.x + threadIdx.x, t);
    for (int q = 0; q < 3; q++) {
        const int v = block_sum(t[q]);
        if (threadIdx.x == 0) P.csum[q * gridDim.x + blockIdx.x] = v;
    }
}

// csum of very many chunks: each chunk's sum becomes the sum of the chunks before it, by one
// block (a thread takes a run of chunks)
__global__ void __launch_bounds__(1024) agg_scan_kernel(AggPass P, Mat<double> A, int chunks) {
    if (unfinished(A)) return;
    __shared__ int wsum[32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, per = (chunks + 1023) / 1024;
    const int lo = min(chunks, (int)threadIdx.x * per), hi = min(chunks, lo + per);
    for (int q = 0; q < 3; q++) {
        int *c = P.csum + (long)q * chunks, sum = 0;
#pragma unroll 8
        for (int k = lo; k < hi; k++) sum += c[k];
        int x = sum;
        for (int o = 1; o < 32; o <<= 1) { const int y = __shfl_up_sync(0xffffffffu, x, o); if (lane >= o) x += y; }
        if (lane == 31) wsum[wid] = x;
        __syncthreads();
        int b = x - sum;
        for (int w = 0; w < wid; w++) b += wsum[w];
        for (int k = lo; k < hi; k++) { const int v = c[k]; c[k] = b; b += v; }
        __syncthreads();
    }
}

// v[0..n) ascending
__device__ __forceinline__ void sort_ints(int *v, int n) {
    for (int a = 1; a < n; a++) {
        const int x = v[a];
        int t = a - 1;
        while (t >= 0 && v[t] > x) { v[t + 1] = v[t]; t--; }
        v[t + 1] = x;
    }
}

// number the aggregates of this block's chunk (its base: the sum of the chunks
// before it, added up by every block for itself unless agg_scan_kernel has) and write them
__global__ void agg_write_kernel(AggPass P, Mat<double> A) {
    if (unfinished(A)) return;
    constexpr int kLocal = 24;
    __shared__ int wsum[3][32];
    const int i = blockIdx.x * blockDim.x + threadIdx.x, lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int t[3], pre[3];
    agg_counts(P, A, i, t);
    for (int q = 0; q < 3; q++) {
        int b = 0;
        if (P.scanned) {
            b = P.csum[q * gridDim.x + blockIdx.x];
        } else {
            for (int k = threadIdx.x; k < (int)blockIdx.x; k += blockDim.x) b += P.csum[q * gridDim.x + k];
            b = block_sum(b);
        }
        int x = t[q];                                          // inclusive scan over the block's threads
        for (int o = 1; o < 32; o <<= 1) { const int y = __shfl_up_sync(0xffffffffu, x, o); if (lane >= o) x += y; }
        if (lane == 31) wsum[q][wid] = x;
        __syncthreads();
        for (int w = 0; w < wid; w++) b += wsum[q][w];
        pre[q] = b + x - t[q];
    }
    if (blockIdx.x == gridDim.x - 1 && threadIdx.x == blockDim.x - 1) {
        const int tot = pre[0] + t[0];
        *P.nc = tot;
        P.moff[tot] = pre[1] + t[1];
        if (P.moffF) P.moffC[tot] = pre[2] + t[2];
    }
    if (!t[0]) return;
    const int id = pre[0], sz = t[1], p = P.st.partner[i];
    int buf[kLocal];
    int *mm = P.mem + pre[1], k = 0;
    P.moff[id] = pre[1];
    if (sz <= kLocal) {
        each_member(P, A, i, p, [&](int m) { buf[k++] = m; });
        sort_ints(buf, sz);
        for (int q = 0; q < sz; q++) { mm[q] = buf[q]; P.agg[buf[q]] = id; }
    } else {
        each_member(P, A, i, p, [&](int m) { mm[k++] = m; P.agg[m] = id; });
        sort_ints(mm, sz);
    }
    if (!P.moffF) return;
    const int szF = t[2];
    int *mf = P.memC + pre[2], kf = 0;
    int *dst = szF <= kLocal ? buf : mf;
    P.moffC[id] = pre[2];
    for (int q = 0; q < sz; q++) {
        const int m = mm[q];
        for (int r = P.moffF[m]; r < P.moffF[m + 1]; r++) dst[kf++] = P.memF[r];
    }
    sort_ints(dst, szF);
    for (int q = 0; q < szF; q++) { mf[q] = dst[q]; P.aggC[dst[q]] = id; }
}

// Galerkin row I of P^T A P, one warp per row.  The members' row entries, mapped
// to aggregate columns, are staged in member-then-column order (the order of the
// sequential definition) and each distinct column sums its entries in that order;
// the distinct columns are ranked ascending.  A list of at most kGalSort entries is
// sorted by (column, place in the list) in registers; longer ones, up to kGalCap,
// are searched; a row beyond that is marked (first column -2) for galerkin_kernel
// and sets bit 0 of *flags.  Writes the entries below Wcap of each row (the rest of
// the columns holds -1 already) and the largest row length into *wmax.  Bound by the
// latency of a warp's chain (members, columns, aggregates, sort).  200k cells: the
// first pass's 85k rows 75 us in one launch (counting and filling by search: 80 + 102
// us), the third's 15k 27 us (30 + 50 us).
constexpr int kGalWarps = 4, kGalCap = 384, kGalSort = 256;
static_assert(kGalSort % 32 == 0 && kGalSort <= 256 && kGalCap % 32 == 0, "a lane per key, eight bits of place");

// the list cl, vl of L <= 32 KR entries: element 32 r + lane of the warp's bitonic
// sort is key r of the lane; returns the number of distinct columns
template <int KR>
__device__ __forceinline__ int galerkin_sorted(const int *cl, const double *vl, unsigned *sk, int L, int I, int nc, int Wcap,
                                               int *__restrict__ ccol, double *__restrict__ cval) {
    const int lane = threadIdx.x & 31;
    unsigned k[KR];
#pragma unroll
    for (int r = 0; r < KR; r++) {
        const int e = 32 * r + lane;
        k[r] = e < L ? ((unsigned)cl[e] << 8) | e : 0xffffffffu;
    }
#pragma unroll
    for (int size = 2; size <= 32 * KR; size <<= 1) {
#pragma unroll
        for (int str = size >> 1; str > 0; str >>= 1) {
            if (str >= 32) {
                const int d = str >> 5;
#pragma unroll
                for (int r = 0; r < KR; r++) {
                    if (r & d) continue;
                    const bool up = size == 32 * KR || ((32 * r) & size) == 0;
                    const unsigned lo = min(k[r], k[r | d]), hi = max(k[r], k[r | d]);
                    k[r] = up ? lo : hi;
                    k[r | d] = up ? hi : lo;
                }
            } else {
                const bool low = (lane & str) == 0;
#pragma unroll
                for (int r = 0; r < KR; r++) {
                    const unsigned o = __shfl_xor_sync(0xffffffffu, k[r], str);
                    const bool up = size == 32 * KR || ((32 * r + lane) & size) == 0;
                    k[r] = low == up ? min(k[r], o) : max(k[r], o);
                }
            }
        }
    }
#pragma unroll
    for (int r = 0; r < KR; r++) sk[32 * r + lane] = k[r];
    __syncwarp();
    int D = 0;
#pragma unroll
    for (int r = 0; r < KR; r++) {
        const int e = 32 * r + lane;
        const unsigned c = k[r] >> 8;
        const bool head = e < L && (e == 0 || (sk[e - 1] >> 8) != c);
        const unsigned b = __ballot_sync(0xffffffffu, head);
        if (head) {
            const int rank = D + __popc(b & ((1u << lane) - 1u));
            double sum = 0.0;
            for (int q = e; q < L && (sk[q] >> 8) == c; q++) sum = __dadd_rn(sum, vl[sk[q] & 255u]);
            if (rank < Wcap) {
                ccol[(long)rank * nc + I] = (int)c;
                cval[(long)rank * nc + I] = sum;
            }
        }
        D += __popc(b);
    }
    return D;
}

__global__ void __launch_bounds__(kGalWarps * 32) galerkin_row_kernel(
    Mat<double> A, const int *__restrict__ agg, const int *__restrict__ moff, const int *__restrict__ mem, int nc, int Wcap,
    int *__restrict__ ccol, double *__restrict__ cval, int *__restrict__ clen, int *wmax, int *flags) {
    __shared__ int scol[kGalWarps][kGalCap];
    __shared__ double sval[kGalWarps][kGalCap];
    __shared__ unsigned skey[kGalWarps][kGalSort];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int I = blockIdx.x * kGalWarps + w;
    if (I >= nc) return;                          // whole warp
    int *cl = scol[w];
    double *vl = sval[w];
    const unsigned lt = (1u << lane) - 1u;
    // 1. the ordered list: slots (member, entry of its row), four per lane in flight
    const int q0 = moff[I], nm = moff[I + 1] - q0;
    int W = 7;                                    // the members' longest row
    if (!A.st) {
        W = 0;
        for (int q = lane; q < nm; q += 32) W = max(W, A.len[mem[q0 + q]]);
        W = __reduce_max_sync(0xffffffffu, W);
    }
    const int slots = nm * W;
    int L = 0;
    for (int s0 = 0; s0 < slots; s0 += 4 * 32) {
        int col[4];
        double v[4];
#pragma unroll
        for (int u = 0; u < 4; u++) {
            const int s = s0 + 32 * u + lane;
            col[u] = -1;
            v[u] = 0.0;
            if (s < slots) {
                const int q = s / W, k = s - q * W, m = mem[q0 + q];
                if (A.st) {
                    // the 7-point entries in ascending column order: -z, -y, -x, centre, +x, +y, +z
                    const int nx = A.g.nx, ny = A.g.ny, nxy = nx * ny;
                    const int ix = m % nx, t = m / nx, iy = t % ny, iz = t / ny;
                    const int d = k == 0 ? 5 : k == 1 ? 3 : k == 2 ? 1 : k == 3 ? 0 : k == 4 ? 2 : k == 5 ? 4 : 6;
                    const bool ok = d == 0 || (d == 1 && ix > 0) || (d == 2 && ix < nx - 1) || (d == 3 && iy > 0) ||
                                    (d == 4 && iy < ny - 1) || (d == 5 && iz > 0) || (d == 6 && iz < A.g.nz - 1);
                    const int off = d == 0 ? 0 : d == 1 ? -1 : d == 2 ? 1 : d == 3 ? -nx : d == 4 ? nx : d == 5 ? -nxy : nxy;
                    if (ok) { col[u] = m + off; v[u] = A.val[(long)d * A.n + m]; }
                } else {
                    col[u] = A.col[(long)k * A.n + m];      // -1 past the row's end
                    if (col[u] >= 0) v[u] = A.val[(long)k * A.n + m];
                }
            }
        }
#pragma unroll
        for (int u = 0; u < 4; u++) if (col[u] >= 0) col[u] = agg[col[u]];
#pragma unroll
        for (int u = 0; u < 4; u++) {
            const unsigned bal = __ballot_sync(0xffffffffu, col[u] >= 0);
            const int pos = L + __popc(bal & lt);
            if (col[u] >= 0 && pos < kGalCap) { cl[pos] = col[u]; vl[pos] = v[u]; }
            L += __popc(bal);
        }
        if (L > kGalCap) { if (lane == 0) { ccol[I] = -2; atomicOr(flags, 1); } return; }
    }
    __syncwarp();
    int D = 0;
    if (L <= kGalSort && nc < (1 << 24)) {
        // 2a. keys (column, place) sorted over the warp, up to eight per lane
        if (L <= 32) D = galerkin_sorted<1>(cl, vl, skey[w], L, I, nc, Wcap, ccol, cval);
        else if (L <= 64) D = galerkin_sorted<2>(cl, vl, skey[w], L, I, nc, Wcap, ccol, cval);
        else if (L <= 128) D = galerkin_sorted<4>(cl, vl, skey[w], L, I, nc, Wcap, ccol, cval);
        else D = galerkin_sorted<8>(cl, vl, skey[w], L, I, nc, Wcap, ccol, cval);
    } else {
        // 2b. search: an entry is its column's first when none before it has the column
        unsigned firsts[kGalCap / 32];
#pragma unroll
        for (int g = 0; g < kGalCap / 32; g++) {
            const int p = 32 * g + lane;
            bool first = p < L;
            if (first) {
                const int c = cl[p];
                for (int q = 0; q < p; q++) if (cl[q] == c) { first = false; break; }
            }
            firsts[g] = __ballot_sync(0xffffffffu, first);
            D += __popc(firsts[g]);
        }
#pragma unroll
        for (int g = 0; g < kGalCap / 32; g++) {
            const int p = 32 * g + lane;
            if (!((firsts[g] >> lane) & 1u)) continue;
            const int c = cl[p];
            double sum = 0.0;
            for (int q = p; q < L; q++) if (cl[q] == c) sum = __dadd_rn(sum, vl[q]);
            int rank = 0;                          // distinct columns below c
#pragma unroll
            for (int g2 = 0; g2 < kGalCap / 32; g2++)
                for (unsigned f = firsts[g2]; f; f &= f - 1) rank += cl[32 * g2 + __ffs(f) - 1] < c;
            if (rank < Wcap) {
                ccol[(long)rank * nc + I] = c;
                cval[(long)rank * nc + I] = sum;
            }
        }
    }
    if (lane == 0) {
        clen[I] = D;
        if (D > *(volatile int *)wmax) atomicMax(wmax, D);
    }
}

// Galerkin rows the row kernel marked, one thread per row: members moff/mem
// (ascending), entries summed in member order then column order, columns sorted
// ascending.  A row of more than SIM_MAX_ELL columns sets bit 1 of *flags.
__global__ void galerkin_kernel(Mat<double> A, const int *__restrict__ agg, const int *__restrict__ moff,
                                const int *__restrict__ mem, int nc, int Wcap, int *__restrict__ ccol,
                                double *__restrict__ cval, int *__restrict__ clen, int *wmax, int *flags) {
    const int I = blockIdx.x * blockDim.x + threadIdx.x;
    if (I >= nc || ccol[I] != -2) return;
    int cols[MAXE];
    double vals[MAXE];
    int cnt = 0;
    bool over = false;
    for (int q = moff[I]; q < moff[I + 1]; q++) {
        const int m = mem[q];
        for_row(A, m, [&](int j, double a) {
            const int Jc = agg[j];
            int f = -1;
            for (int t = 0; t < cnt; t++) if (cols[t] == Jc) { f = t; break; }
            if (f < 0) {
                if (cnt == MAXE) { over = true; return; }
                cols[cnt] = Jc; vals[cnt] = 0.0; f = cnt++;
            }
            vals[f] = __dadd_rn(vals[f], a);
        });
    }
    if (over) { atomicOr(flags, 2); return; }
    clen[I] = cnt;
    atomicMax(wmax, cnt);
    if (cnt > Wcap) return;                        // built again with room for it
    for (int a = 1; a < cnt; a++) {
        const int cj = cols[a];
        const double cv = vals[a];
        int t = a - 1;
        while (t >= 0 && cols[t] > cj) { cols[t + 1] = cols[t]; vals[t + 1] = vals[t]; t--; }
        cols[t + 1] = cj; vals[t + 1] = cv;
    }
    for (int t = 0; t < cnt; t++) {
        ccol[(long)t * nc + I] = cols[t];
        cval[(long)t * nc + I] = vals[t];
    }
}

// What the application reads of the coarse levels, all levels in one launch, a
// thread per row: 1 / l1 row sums, the columns with padding on the row itself
// (value 0), and the FP32 copy in the difference form: the diagonal entry replaced
// by the row sum (computed in FP64), the others rounded as they are.  It also counts each
// level's entries (a sum over the warp and one atomic), which the byte models report.
constexpr int kFinishLevels = 16;
struct FinishLevel {
    int n, width, row0;          // row0: first row of the level in the launch's row numbering
    const int *col, *len;
    double *val;
    int *colA;
    void *valT, *dinvT;
};
struct FinishTable {
    int count, rows;
    unsigned long long *entries;             // of each level
    FinishLevel lv[kFinishLevels];
};
template <typename T>
__global__ void __launch_bounds__(128) finish_levels_kernel(const __grid_constant__ FinishTable tb) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    int l = 0;
    while (l + 1 < tb.count && t >= tb.lv[l + 1].row0) l++;
    const FinishLevel &L = tb.lv[l];
    const int i = t - L.row0, n = L.n;
    const int len = t < tb.rows ? L.len[i] : 0;
    for (int q = __reduce_min_sync(0xffffffffu, l), q1 = __reduce_max_sync(0xffffffffu, l); q <= q1; q++) {
        const int c = __reduce_add_sync(0xffffffffu, l == q ? len : 0);
        if ((threadIdx.x & 31) == 0) atomicAdd(tb.entries + q, (unsigned long long)c);
    }
    if (t >= tb.rows) return;
    double s = 0.0, rs = 0.0;
    for (int k0 = 0; k0 < L.width; k0 += 8) {
        int j[8];
        double a[8];
#pragma unroll
        for (int u = 0; u < 8; u++) j[u] = k0 + u < L.width ? L.col[(long)(k0 + u) * n + i] : -1;
#pragma unroll
        for (int u = 0; u < 8; u++) a[u] = j[u] >= 0 ? L.val[(long)(k0 + u) * n + i] : 0.0;
#pragma unroll
        for (int u = 0; u < 8; u++) {
            if (k0 + u >= L.width) continue;
            const long q = (long)(k0 + u) * n + i;
            if (j[u] >= 0) { s += fabs(a[u]); rs += a[u]; }
            else L.val[q] = 0.0;
            L.colA[q] = j[u] >= 0 ? j[u] : i;
            if (sizeof(T) == sizeof(float) && j[u] != i) ((float *)L.valT)[q] = (float)a[u];
        }
    }
    ((T *)L.dinvT)[i] = (T)(1.0 / s);
    if (sizeof(T) == sizeof(float))
        for (int k = 0; k < L.width; k++)
            if (L.col[(long)k * n + i] == i) { ((float *)L.valT)[(long)k * n + i] = (float)rs; break; }
}

// Gauss-Jordan step k without pivoting on the augmented [A | Inv] (n x 2n),
// read from src and written to dst: the coarse pressure block is
// diagonally dominant with a positive diagonal, so the pivots stay positive.
// Gauss-Jordan elimination without pivoting of [A | I] on the coarsest level,
// in one launch of an 8-CTA cluster: step k writes, from the matrix left by
// step k-1 (ping-pong buffers), pivot row k divided by its pivot and every
// other row minus its column-k entry times that row; a cluster barrier
// separates the steps; the result ends in A1 for odd n, else A0
constexpr int kGjMax = 1024;   // largest coarsest level (rows)

// A pivot whose magnitude is not above kGjPivotTol times the l1 norm of its
// row of A (rn) -- zero, denormal, NaN, or pure rounding noise -- sets *bad;
// the elimination still runs to its end (the cluster barriers need every CTA)
// and the host turns the flag into an error instead of using the inverse.
constexpr double kGjPivotTol = 1e-14;

__device__ __forceinline__ void gj_check_pivot(double piv, double rnorm, int *bad) {
    if (!(fabs(piv) > kGjPivotTol * rnorm)) *(volatile int *)bad = 1;
}

__global__ void __cluster_dims__(8, 1, 1) __launch_bounds__(1024, 1)
gj_cluster_kernel(int n, double *__restrict__ A0, double *__restrict__ A1, const double *__restrict__ rn, int *bad) {
    __shared__ double pk[2 * kGjMax];   // the pivot row over its pivot, per CTA (one division per entry)
    const int w = 2 * n;
    // CTA c owns rows c, c + 8, ...; its threads stride over the columns (no index division)
    const int tpr = blockDim.x < (unsigned)w ? blockDim.x : w;    // threads per row
    const int rows_at_once = blockDim.x / tpr;
    const int r0 = threadIdx.x / tpr, j0 = threadIdx.x % tpr;
    for (int k = 0; k < n; k++) {
        const double *src = (k & 1) ? A1 : A0;
        double *dst = (k & 1) ? A0 : A1;
        const double piv = src[(long)k * w + k];
        if (blockIdx.x == 0 && threadIdx.x == 0) gj_check_pivot(piv, rn[k], bad);
        for (int j = threadIdx.x; j < w; j += blockDim.x) pk[j] = src[(long)k * w + j] / piv;
        __syncthreads();
        if (r0 < rows_at_once) {
            for (int i = blockIdx.x + r0 * gridDim.x; i < n; i += rows_at_once * gridDim.x) {
                const double f = src[(long)i * w + k];
                const double *si = src + (long)i * w;
                double *di = dst + (long)i * w;
                for (int j = j0; j < w; j += tpr) di[j] = (i == k) ? pk[j] : si[j] - f * pk[j];
            }
        }
        __threadfence();
        cg::this_cluster().sync();   // also keeps pk from being overwritten early
    }
}

// The inverse of a matrix of at most kGjSmem rows in one launch of one cluster (8
// CTAs, or 16 where the part schedules a cluster that large), in place in shared
// memory: Gauss-Jordan without pivoting, eight pivots at a time.  Column j lives in
// CTA j mod CTAs, so the eight columns of a panel lie in eight CTAs: each of them
// brings its column of the next panel up to date first and publishes it, and the
// cluster barrier's arrival is there; the rest of the columns follows between
// arrival and wait.  After the barrier every CTA reads the panel (distributed shared
// memory) and inverts its 8 x 8 pivot block D for itself, in one warp's registers:
//   T_j = D A_Kj,  A_ij -= A_iK T_j (i outside K),  A_Kj = T_j;
// a column j of the panel takes part with A_Kj = e_j and A_ij = 0.  Bound by that
// chain and, near 256 rows, by the FP64 pipe of the cluster's SMs (n^2 8 / CTAs FMAs
// a step at 2 a clock).  236 rows: 796 -> 392 us, 133: 352 -> 141, 84: 193 -> 74 (row blocks
// and an augmented matrix, which took 8 us more to set up; a panel of four factored by one
// CTA of 1,024 threads while the others wait).
constexpr int kGjSmem = 256, kGjNb = 8, kGjThreads = 512;

__device__ __forceinline__ void inv8_warp(double (&a)[2], int lane, const double *rn, int *bad) {
    // lane holds row lane / 4, columns 2 (lane % 4) and the next
    const int r = lane >> 2, c0 = 2 * (lane & 3);
#pragma unroll
    for (int k = 0; k < kGjNb; k++) {
        const int kc = k & 1, src = 4 * k + (k >> 1);
        const double piv = __shfl_sync(0xffffffffu, a[kc], src);
        if (bad && lane == 0) gj_check_pivot(piv, rn[k], bad);
        const double ip = 1.0 / piv;
        const double p0 = __shfl_sync(0xffffffffu, a[0], 4 * k + (lane & 3)) * ip;
        const double p1 = __shfl_sync(0xffffffffu, a[1], 4 * k + (lane & 3)) * ip;
        const double f = __shfl_sync(0xffffffffu, a[kc], (lane & ~3) + (k >> 1));
        if (r == k) {
            a[0] = c0 == k ? ip : p0;
            a[1] = c0 + 1 == k ? ip : p1;
        } else {
            a[0] = c0 == k ? -f * ip : a[0] - f * p0;
            a[1] = c0 + 1 == k ? -f * ip : a[1] - f * p1;
        }
    }
}

__global__ void __launch_bounds__(kGjThreads, 1) gj_inverse_kernel(Mat<double> A, double *__restrict__ inv, int *bad) {
    extern __shared__ double gsm[];
    cg::cluster_group cl = cg::this_cluster();
    const int n = A.n, nc = (int)cl.num_blocks(), me = (int)cl.block_rank(), cpc = (n + nc - 1) / nc;
    const int tid = threadIdx.x;
    double *S = gsm;                                  // [cpc][n] own columns
    double *pub = S + (long)cpc * n;                  // [2][n] own column of a panel, by panel parity
    double *PL = pub + 2 * n;                         // [kGjNb][n] the current panel
    double *Tc = PL + kGjNb * n;                      // [cpc][kGjNb]
    double *D = Tc + cpc * kGjNb;                     // [kGjNb][kGjNb] row-major
    double *rn = D + kGjNb * kGjNb;                   // [n + kGjNb] l1 row norms (the pivot test's scale)
    const int mycols = n > me ? (n - me + nc - 1) / nc : 0;
    for (int t = tid; t < cpc * n; t += kGjThreads) S[t] = 0.0;
    __syncthreads();
    for (int i = tid; i < n + kGjNb; i += kGjThreads) {
        double s = 0.0;
        if (i < n)
            for_row(A, i, [&](int j, double v) {
                s += fabs(v);
                if (j % nc == me) S[(long)(j / nc) * n + i] += v;
            });
        rn[i] = s;
    }
    __syncthreads();
    const int steps = (n + kGjNb - 1) / kGjNb;
    if (me < kGjNb && me < n)                         // the first panel
        for (int i = tid; i < n; i += kGjThreads) pub[i] = S[i];
    cl.barrier_arrive();
    for (int s = 0; s < steps; s++) {
        const int k0 = s * kGjNb, kb = min(kGjNb, n - k0);
        cl.barrier_wait();
        for (int t = tid; t < kGjNb * n; t += kGjThreads) {
            const int q = t / n, i = t - q * n;
            PL[t] = q < kb ? cl.map_shared_rank(pub, (k0 + q) % nc)[(s & 1) * n + i] : 0.0;
        }
        __syncthreads();
        if (tid < 32) {
            const int r = tid >> 2, c0 = 2 * (tid & 3);
            double a[2];
#pragma unroll
            for (int u = 0; u < 2; u++) {
                const int c = c0 + u;
                a[u] = r < kb && c < kb ? PL[(long)c * n + k0 + r] : (r == c ? 1.0 : 0.0);
            }
            // rows past the end are the identity's: their pivots are 1 against a norm of 0
            inv8_warp(a, tid, rn + k0, me == 0 ? bad : nullptr);
#pragma unroll
            for (int u = 0; u < 2; u++) D[r * kGjNb + c0 + u] = a[u];
        }
        __syncthreads();
        for (int t = tid; t < mycols * kGjNb; t += kGjThreads) {
            const int lc = t / kGjNb, r = t - lc * kGjNb, j = lc * nc + me;
            double v = 0.0;
            if (j >= k0 && j < k0 + kb) {
                v = D[r * kGjNb + j - k0];
            } else {
#pragma unroll
                for (int q = 0; q < kGjNb; q++) v += D[r * kGjNb + q] * (q < kb ? S[(long)lc * n + k0 + q] : 0.0);
            }
            Tc[t] = v;
        }
        __syncthreads();
        auto update = [&](int lc, int i) -> double {
            const int j = lc * nc + me;
            if (i >= k0 && i < k0 + kb) return Tc[lc * kGjNb + i - k0];
            double v = j >= k0 && j < k0 + kb ? 0.0 : S[(long)lc * n + i];
#pragma unroll
            for (int q = 0; q < kGjNb; q++) v -= PL[q * n + i] * Tc[lc * kGjNb + q];
            return v;
        };
        // my column of the next panel, if I have one
        const int nk0 = k0 + kGjNb, off = ((me - nk0) % nc + nc) % nc, nj = nk0 + off;
        const int nl = off < kGjNb && nj < n ? nj / nc : -1;
        if (nl >= 0)
            for (int i = tid; i < n; i += kGjThreads) {
                const double v = update(nl, i);
                S[(long)nl * n + i] = v;
                pub[((s + 1) & 1) * n + i] = v;
            }
        cl.barrier_arrive();                          // releases the published column
        for (int t = tid; t < mycols * n; t += kGjThreads) {
            const int lc = t / n, i = t - lc * n;
            if (lc != nl) S[t] = update(lc, i);
        }
        __syncthreads();                              // PL, Tc and S are read and written again
    }
    cl.barrier_wait();                                // no CTA leaves while another may read its column
    for (int t = tid; t < mycols * n; t += kGjThreads) {
        const int lc = t / n, i = t - lc * n;
        inv[(long)i * n + lc * nc + me] = S[t];
    }
}

static size_t gj_inverse_bytes(int n, int nc) {
    const int cpc = (n + nc - 1) / nc;
    return sizeof(double) * ((size_t)cpc * n + (2 + kGjNb) * (size_t)n + (size_t)cpc * kGjNb + kGjNb * kGjNb + n + kGjNb);
}

// CTAs of the Gauss-Jordan cluster: 16 (a non-portable size) when the
// occupancy query finds room for one such cluster at the largest shared-memory
// size, else the portable 8; 0 without that much shared memory; the query launches nothing
static int gj_cluster_ctas() {
    if (cudaFuncSetAttribute(gj_inverse_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)gj_inverse_bytes(kGjSmem, 8)) != cudaSuccess) {
        (void)cudaGetLastError();
        return 0;
    }
    if (cudaFuncSetAttribute(gj_inverse_kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) {
        (void)cudaGetLastError();
        return 8;
    }
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = 16; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3(16); cfg.blockDim = dim3(kGjThreads); cfg.dynamicSmemBytes = gj_inverse_bytes(kGjSmem, 16);
    cfg.attrs = at; cfg.numAttrs = 1;
    int clusters = 0;
    if (cudaOccupancyMaxActiveClusters(&clusters, gj_inverse_kernel, &cfg) != cudaSuccess) {
        (void)cudaGetLastError();
        return 8;
    }
    return clusters > 0 ? 16 : 8;
}

// [A | I], one thread per entry (row i, column j of the n x 2n array)
__global__ void gj_init_kernel(Mat<double> A, double *__restrict__ aug) {
    const long w = 2L * A.n;
    const long t = blockIdx.x * (long)blockDim.x + threadIdx.x;
    if (t >= (long)A.n * w) return;
    const int i = (int)(t / w), j = (int)(t - (long)i * w);
    double v = (j - A.n == i) ? 1.0 : 0.0;
    if (j < A.n) for_row(A, i, [&](int c, double a) { if (c == j) v += a; });
    aug[t] = v;
}

// l1 norm of each row of the coarsest matrix (the scale of the pivot test)
__global__ void gj_rownorm_kernel(Mat<double> A, double *__restrict__ rn) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= A.n) return;
    double t = 0.0;
    for_row(A, i, [&](int, double a) { t += fabs(a); });
    rn[i] = t;
}

template <typename T>
__global__ void gj_extract_kernel(int n, const double *__restrict__ aug, T *__restrict__ inv) {
    const long t = blockIdx.x * (long)blockDim.x + threadIdx.x;
    if (t >= (long)n * n) return;
    const int i = (int)(t / n), j = (int)(t % n);
    inv[t] = (T)aug[(long)i * 2 * n + n + j];
}

// ---------------------------------------------------------------------------
// apply kernels (precision T)
// ---------------------------------------------------------------------------
// L2 prefetch of part `part` of `parts` of [p, p + bytes), its ends rounded
// inwards to 16 bytes (a bulk prefetch is a hint; it never leaves the range)
__device__ __forceinline__ void l2_prefetch_part(const void *p, size_t bytes, int part, int parts) {
    if (p == nullptr || bytes < 16) return;
    const size_t a = (size_t)p, e = a + bytes;
    const size_t chunk = (bytes / parts + 15) & ~(size_t)15;
    size_t lo = (a + (size_t)part * chunk + 15) & ~(size_t)15;
    size_t hi = (a + (size_t)(part + 1) * chunk) & ~(size_t)15;
    if (hi > (e & ~(size_t)15)) hi = e & ~(size_t)15;
    if (hi <= lo) return;
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(lo), "r"((unsigned)(hi - lo)) : "memory");
}

// arrays to bring into L2 ahead of their use (the coarse levels of a V-cycle):
// the first kernel of stage P issues the prefetches, the cluster launch of the
// coarse levels starts tens of microseconds later with its data in L2
constexpr int kPrefetchMax = 16;
struct L2Prefetch {
    int count;
    const void *p[kPrefetchMax];
    unsigned long long bytes[kPrefetchMax];
};
constexpr int kPrefetchParts = 8;
__device__ __forceinline__ void issue_prefetch(const L2Prefetch &pf) {
    if (blockIdx.x < kPrefetchParts && (int)threadIdx.x < pf.count)
        l2_prefetch_part(pf.p[threadIdx.x], pf.bytes[threadIdx.x], blockIdx.x, kPrefetchParts);
}

// f0 = first row of L times r (quasi-IMPES: L_00 = 1); e0 = f0 / l1
template <int B, typename T>
__device__ __forceinline__ void restrict_p_row(int N, const double *__restrict__ r, const T *__restrict__ wT, int full,
                                               const T *__restrict__ dinv0, T *__restrict__ f0, T *__restrict__ e0,
                                               int i) {
    // explicit FMAs: the same rounding in every kernel that inlines the row
    const T r0 = full ? wT[i] * (T)r[i] : (T)r[i];
    T t = fma(wT[(long)N + i], (T)r[(long)N + i], r0);
    if (B == 3) t = fma(wT[2L * N + i], (T)r[2L * N + i], t);
    f0[i] = t;
    e0[i] = t * dinv0[i];
}

template <int B, typename T>
__global__ void restrict_p_kernel(int N, const double *__restrict__ r, const T *__restrict__ wT, int full,
                                  const T *__restrict__ dinv0, T *__restrict__ f0, T *__restrict__ e0, const L2Prefetch pf,
                                  const int *done) {
    if (skip(done)) return;
    issue_prefetch(pf);
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N) return;
    restrict_p_row<B, T>(N, r, wT, full, dinv0, f0, e0, i);
}

// r = f - A e, row i by `lanes` lanes from thread t of the level's launch on (a
// thread per row on the 7-point level: coalesced stencil reads)
template <typename T>
__device__ __forceinline__ void amg_resid_row(const Mat<T> &A, const T *__restrict__ f, const T *__restrict__ e,
                                              T *__restrict__ r, long t) {
    if (A.st) {
        if (t < A.n) r[t] = f[t] - row_dot(A, (int)t, e);
        return;
    }
    const int lanes = ell_lanes(A.n), i = (int)(t / lanes), sub = (int)(t & (lanes - 1));
    const bool ok = i < A.n;
    const T d = mat_dot_lanes(A, i, ok, lanes, sub, e);
    if (ok && sub == 0) r[i] = f[i] - d;
}
template <typename T>
__global__ void amg_resid_kernel(Mat<T> A, const T *__restrict__ f, const T *__restrict__ e, T *__restrict__ r,
                                 const int *done) {
    if (skip(done)) return;
    amg_resid_row<T>(A, f, e, r, blockIdx.x * (long)blockDim.x + threadIdx.x);
}

// f_c = P^T r of coarse row I
template <typename T>
__device__ __forceinline__ void amg_restrict_row(const T *__restrict__ r, const int *__restrict__ moff,
                                                 const int *__restrict__ mem, T *__restrict__ fc, T *__restrict__ ec,
                                                 const T *__restrict__ dinvc, int I) {
    // members in batches of 8: the batch's indices, then its gathers, then the
    // sum in member order (a plain loop would wait on each load in turn)
    const int q0 = moff[I], q1 = moff[I + 1];
    T s = (T)0;
    for (int qb = q0; qb < q1; qb += 8) {
        int m[8];
        T v[8];
#pragma unroll
        for (int u = 0; u < 8; u++) m[u] = qb + u < q1 ? mem[qb + u] : -1;
#pragma unroll
        for (int u = 0; u < 8; u++) v[u] = m[u] >= 0 ? r[m[u]] : (T)0;
#pragma unroll
        for (int u = 0; u < 8; u++)
            if (qb + u < q1) s += v[u];
    }
    fc[I] = s;
    if (ec) ec[I] = s * dinvc[I];
}

// f_c = P^T r (members in ascending order); e_c = f_c / l1 (coarse pre-smoothing)
template <typename T>
__global__ void amg_restrict_kernel(const T *__restrict__ r, const int *__restrict__ moff, const int *__restrict__ mem,
                                    int nc, T *__restrict__ fc, T *__restrict__ ec, const T *__restrict__ dinvc,
                                    const int *done) {
    if (skip(done)) return;
    const int I = blockIdx.x * blockDim.x + threadIdx.x;
    if (I >= nc) return;
    amg_restrict_row<T>(r, moff, mem, fc, ec, dinvc, I);
}


// e += P e_c
template <typename T>
__global__ void amg_prolong_kernel(int n, const int *__restrict__ agg, const T *__restrict__ ec, T *__restrict__ e,
                                   const int *done) {
    if (skip(done)) return;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) e[i] += ec[agg[i]];
}

// e2 = e + (f - A e) / l1 (post-smoothing), threads as in amg_resid_row; on a 7-point
// level `add` adds it to e2 (the correction of several cycles: no pass of its own)
template <typename T>
__device__ __forceinline__ void amg_smooth_row(const Mat<T> &A, const T *__restrict__ f, const T *__restrict__ e,
                                               const T *__restrict__ dinv, T *__restrict__ e2, long t, bool add = false) {
    if (A.st) {
        if (t < A.n) {
            const T v = e[t] + (f[t] - row_dot(A, (int)t, e)) * dinv[t];
            e2[t] = add ? e2[t] + v : v;
        }
        return;
    }
    const int lanes = ell_lanes(A.n), i = (int)(t / lanes), sub = (int)(t & (lanes - 1));
    const bool ok = i < A.n;
    const T d = mat_dot_lanes(A, i, ok, lanes, sub, e);
    if (ok && sub == 0) e2[i] = e[i] + (f[i] - d) * dinv[i];
}
template <typename T>
__global__ void amg_smooth_kernel(Mat<T> A, const T *__restrict__ f, const T *__restrict__ e, const T *__restrict__ dinv,
                                  T *__restrict__ e2, const int *done, bool add) {
    if (skip(done)) return;
    amg_smooth_row<T>(A, f, e, dinv, e2, blockIdx.x * (long)blockDim.x + threadIdx.x, add);
}

// next stage-P cycle: f0 = rp - A_p ep; e0 = f0 / l1
template <typename T>
__device__ __forceinline__ void cycle_next_row(const Mat<T> &A, const T *rp, const T *__restrict__ ep,
                                               const T *__restrict__ dinv, T *f0, T *__restrict__ e0, int i) {
    const T f = rp[i] - row_dot(A, i, ep);
    f0[i] = f;
    e0[i] = f * dinv[i];
}
// The second cycle starts from the first one's f0 (in place: a row reads its own entry
// only) and e2, and leaves both where later cycles look (keep_rp may be null, keep_ep):
// 1M cells, two cycles: with the last smoothing adding its result the application takes
// 603 us, 617 with three copy launches of 5 us (4.1M cells: a solve 300 against 309 ms).
template <typename T>
__global__ void cycle_next_kernel(Mat<T> A, const T *rp, const T *__restrict__ ep, const T *__restrict__ dinv,
                                  T *f0, T *__restrict__ e0, T *__restrict__ keep_rp, T *__restrict__ keep_ep, const int *done) {
    if (skip(done)) return;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= A.n) return;
    if (keep_rp) keep_rp[i] = rp[i];
    if (keep_ep) keep_ep[i] = ep[i];
    cycle_next_row<T>(A, rp, ep, dinv, f0, e0, i);
}

// y = x (mode 0) or y += x (mode 1)
template <typename T>
__global__ void copy_add_kernel(int n, const T *__restrict__ x, T *__restrict__ y, int mode, const int *done) {
    if (skip(done)) return;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) y[i] = mode ? y[i] + x[i] : x[i];
}

// e = Inv f on the coarsest level (FP64 inverse and sum): one warp per row
template <typename T>
__global__ void coarse_solve_kernel(int n, const double *__restrict__ Inv, const T *__restrict__ f, T *__restrict__ e,
                                    const int *done) {
    if (skip(done)) return;
    const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (warp >= n) return;
    double s = 0.0;
    for (int j = lane; j < n; j += 32) s += Inv[(long)warp * n + j] * (double)f[j];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if (lane == 0) e[warp] = (T)s;
}

// ---- the coarse end of the V-cycle in one launch --------------------------
// Levels l0..nl-1 (each at most coarse_rows rows) run inside one thread-block
// cluster: the same row operations as the per-level kernels, with a cluster
// barrier between dependent sweeps instead of a kernel boundary.  On entry
// level l0 holds f and its pre-smoothed e; on exit its corrected vector is e2.
// Every sweep is a chain of dependent L2 loads: 16 CTAs (8 where the part does not
// schedule a cluster that large) give each row its lanes (ell_lanes), the prolonged
// correction is added where the post-smoothing reads it (one sweep and one barrier
// less a level), and a row's loop ends at the warp's longest row, not at the ELL
// width.  What a larger level costs here is the latency of its passes on 16 SMs
// (8,000 rows: residual 6 us, post-smoothing 9 us), so it is left to the per-level
// launches over all SMs: above 3,072 rows in FP64 (200k-cell Newton iteration 31.8 ms
// with 16,384 rows, 31.2 with 3,000; application of 398k cells 213 and 202 us), above
// 6,144 in FP32, whose sums are cheaper (151k cells: 14.65 ms, 15.1 with 3,000).
constexpr int kCoarseThreads = 1024;
inline int coarse_rows(bool fp32) { return fp32 ? 6144 : 3072; }
constexpr int kCoarseMaxLevels = 24;

template <typename T>
struct CoarseLevel {
    int n, width, diff, st;   // st: level 0, the 7-point stencil
    const int *colA;     // self-padded ELL columns [width][n]
    const int *len;      // entries of each row
    const T *val;        // [width][n]
    const T *dinv;       // 1 / l1 row sums
    const int *agg;      // row -> next-level aggregate
    const int *moff, *mem;
    T *f, *e, *e2;
};

template <typename T>
struct CoarseCycle {
    int nlev;                          // levels in lv (the last one is the coarsest)
    GridDesc g;                        // of a structured level
    const double *inv;                 // coarsest: dense inverse, row-major (FP64)
    CoarseLevel<T> lv[kCoarseMaxLevels];
};

// the arrival releases this thread's global writes to the cluster, the wait acquires the others'
__device__ __forceinline__ void cluster_barrier() { cg::this_cluster().sync(); }

// rows lo..hi of a level of n rows for CTA `rank` of nb: one contiguous block each,
// so every SM of the cluster carries an equal share of a small level's L2 traffic
// (a grid-wide thread index would leave a 1,000-row level to one or two SMs);
// f(row, row exists, lane of the row) on every lane of the CTA together
template <typename F>
__device__ __forceinline__ void sweep_rows(int n, int lanes, int rank, int nb, F f) {
    const int per = (n + nb - 1) / nb, lo = min(n, rank * per), hi = min(n, lo + per);
    const int sub = threadIdx.x & (lanes - 1), at = threadIdx.x / lanes, step = blockDim.x / lanes;
    for (int b = lo; b < hi; b += step) f(b + at, b + at < hi, sub);
}

template <typename T, typename FE>
__device__ __forceinline__ T coarse_dot(const CoarseCycle<T> &cc, const CoarseLevel<T> &L, int i, bool ok, int lanes, int sub,
                                        T ei, FE e) {
    const long n = L.n;
    return row_dot_lanes<T>(L.width, L.st ? 7 : (ok ? L.len[i] : 0), lanes, sub, ok, L.diff != 0, i, ei,
                            [&](int k, int &j, T &v) {
                                if (L.st) {
                                    const int d = k == 0 ? 5 : k == 1 ? 3 : k == 2 ? 1 : k == 3 ? 0 : k == 4 ? 2 : k == 5 ? 4 : 6;
                                    const int q = nbr7(cc.g, i, d);
                                    if (q >= 0) { j = q; v = L.val[d * n + i]; }
                                } else {
                                    j = L.colA[k * n + i];
                                    v = L.val[k * n + i];
                                }
                            },
                            e);
}

// the cycle run by CTA `rank` of the nb CTAs of one cluster
template <typename T>
__device__ __forceinline__ void coarse_cycle_body(const CoarseCycle<T> &cc, int rank, int nb) {
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5, wpb = blockDim.x >> 5;
    const int last = cc.nlev - 1;
    // the matrices of the levels below the first and the dense inverse come into
    // L2 while the first level is swept: one bulk prefetch per (array, CTA)
    if (threadIdx.x < 32) {
        const int t = threadIdx.x;
        const int lv = 1 + t / 4, a = t % 4;
        if (lv <= last) {
            const CoarseLevel<T> &Q = cc.lv[lv];
            const size_t ell = (size_t)Q.width * Q.n;
            if (a == 0) l2_prefetch_part(Q.colA, sizeof(int) * ell, rank, nb);
            else if (a == 1) l2_prefetch_part(Q.val, sizeof(T) * ell, rank, nb);
            else if (a == 2) l2_prefetch_part(Q.dinv, sizeof(T) * Q.n, rank, nb);
            else if (lv < last) l2_prefetch_part(Q.mem, sizeof(int) * Q.n, rank, nb);
            else l2_prefetch_part(cc.inv, sizeof(double) * (size_t)Q.n * Q.n, rank, nb);
        }
    }
    for (int l = 0; l < last; l++) {
        const CoarseLevel<T> &L = cc.lv[l], &C = cc.lv[l + 1];
        const int lanes = L.st ? 1 : ell_lanes(L.n);
        sweep_rows(L.n, lanes, rank, nb, [&](int i, bool ok, int sub) {
            const T t = coarse_dot<T>(cc, L, i, ok, lanes, sub, ok ? L.e[i] : (T)0, [&](int j) { return L.e[j]; });
            if (ok && sub == 0) L.e2[i] = L.f[i] - t;
        });
        cluster_barrier();
        // restriction: eight lanes load a coarse row's members, added in member order
        sweep_rows(C.n, 8, rank, nb, [&](int I, bool ok, int sub) {
            const int q0 = ok ? L.moff[I] : 0, q1 = ok ? L.moff[I + 1] : 0;
            const int most = __reduce_max_sync(0xffffffffu, q1 - q0);
            T s = (T)0;
            for (int b = 0; b < most; b += 8) {
                const T v = q0 + b + sub < q1 ? L.e2[L.mem[q0 + b + sub]] : (T)0;
#pragma unroll
                for (int u = 0; u < 8; u++) {
                    const T x = __shfl_sync(0xffffffffu, v, u, 8);
                    if (q0 + b + u < q1) s += x;
                }
            }
            if (ok && sub == 0) {
                C.f[I] = s;
                if (l + 1 < last) C.e[I] = s * C.dinv[I];
            }
        });
        cluster_barrier();
    }
    {
        const CoarseLevel<T> &C = cc.lv[last];
        const int per = (C.n + nb - 1) / nb, hi = min(C.n, (rank + 1) * per);
        for (int r = rank * per + wib; r < hi; r += wpb) {
            double s = 0.0;
#pragma unroll 8
            for (int j = lane; j < C.n; j += 32) s += cc.inv[(long)r * C.n + j] * (double)C.f[j];
            for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
            if (lane == 0) C.e[r] = (T)s;
        }
    }
    cluster_barrier();
    for (int l = last - 1; l >= 0; l--) {
        const CoarseLevel<T> &L = cc.lv[l], &C = cc.lv[l + 1];
        const T *ec = (l + 1 == last) ? C.e : C.e2;
        const int lanes = L.st ? 1 : ell_lanes(L.n);
        sweep_rows(L.n, lanes, rank, nb, [&](int i, bool ok, int sub) {
            auto e = [&](int j) { return L.e[j] + ec[L.agg[j]]; };
            const T ei = ok ? e(i) : (T)0;
            const T t = coarse_dot<T>(cc, L, i, ok, lanes, sub, ei, e);
            if (ok && sub == 0) L.e2[i] = ei + (L.f[i] - t) * L.dinv[i];
        });
        if (l > 0) cluster_barrier();
    }
}

template <typename T>
__global__ void __launch_bounds__(kCoarseThreads, 1)
coarse_cycle_kernel(const __grid_constant__ CoarseCycle<T> cc, const int *done) {
    if (skip(done)) return;            // uniform over the cluster: no thread reaches a barrier alone
    // (a grid constant: the body reads the description in parameter space, no copy)
    coarse_cycle_body<T>(cc, (int)blockIdx.x, (int)gridDim.x);
}

// stage F, pass 1: r2 = rhat - Ahat[:,p] e_p; red cells z = Dinv r2, black keep r2.
// rhat = L r from the FP64 residual (lscT = null: quasi-IMPES, only the first row
// differs from the identity) or, when r is null, the given vector rh; ep may be null.
template <int B, typename T>
__device__ __forceinline__ void stage2_a_row(const GridDesc &g, const double *__restrict__ r, const T *__restrict__ wT,
                                             const T *__restrict__ lscT, const T *__restrict__ rh,
                                             const T *__restrict__ ahat, const T *__restrict__ dinv,
                                             const T *__restrict__ ep, T *__restrict__ r2, T *__restrict__ z, int rb,
                                             int i) {
    const long N = g.N;
    T v[B];
    if (!r) {
#pragma unroll
        for (int c = 0; c < B; c++) v[c] = rh[(long)c * N + i];
    } else if (lscT) {
        T u[B];
#pragma unroll
        for (int c = 0; c < B; c++) u[c] = (T)r[(long)c * N + i];
#pragma unroll
        for (int rr = 0; rr < B; rr++) {
            T t = fma(lscT[(long)(rr * B + 1) * N + i], u[1], lscT[(long)(rr * B) * N + i] * u[0]);
            if (B == 3) t = fma(lscT[(long)(rr * B + 2) * N + i], u[2], t);
            v[rr] = t;
        }
    } else {
#pragma unroll
        for (int c = 0; c < B; c++) v[c] = (T)r[(long)c * N + i];
        T rp = fma(wT[(long)N + i], v[1], v[0]);
        if (B == 3) rp = fma(wT[2L * N + i], v[2], rp);
        v[0] = rp;
    }
    const Cell cc = cell_of(g, i);
    const long NS = 2L * g.H, si = cslot(g, cc.ix, cc.iy, cc.iz);
    if (ep) {
#pragma unroll
        for (int d = 0; d < 7; d++) {
            const int j = nbrc(g, cc, d);
            if (j < 0) continue;
            const T e = ep[j];
#pragma unroll
            for (int c = 0; c < B; c++) v[c] -= ahat[(long)(d * B * B + c * B) * NS + si] * e;
        }
    }
    if (rb && is_black(g, i)) {
#pragma unroll
        for (int c = 0; c < B; c++) r2[(long)c * N + i] = v[c];
        return;
    }
#pragma unroll
    for (int c = 0; c < B; c++) {
        T s = (T)0;
#pragma unroll
        for (int q = 0; q < B; q++) s += dinv[(long)(c * B + q) * NS + si] * v[q];
        z[(long)c * N + i] = s;
    }
}

template <int B, typename T>
__global__ void stage2_a_kernel(GridDesc g, const double *__restrict__ r, const T *__restrict__ wT,
                                const T *__restrict__ lscT, const T *__restrict__ rh, const T *__restrict__ ahat,
                                const T *__restrict__ dinv, const T *__restrict__ ep, T *__restrict__ r2,
                                T *__restrict__ z, int rb, const int *done) {
    if (skip(done)) return;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= g.N) return;
    stage2_a_row<B, T>(g, r, wT, lscT, rh, ahat, dinv, ep, r2, z, rb, i);
}

// CPR-FPF, after the first stage F (x0): rh = L r - Ahat x0 over the full 7-point
// block stencil; f0 = rh_p, e0 = f0 / l1 start stage P
template <int B, typename T>
__device__ __forceinline__ void fpf_resid_row(const GridDesc &g, const double *__restrict__ r, const T *__restrict__ wT,
                                              const T *__restrict__ lscT, const T *__restrict__ ahat,
                                              const T *__restrict__ x0, const T *__restrict__ dinv0, T *__restrict__ rh,
                                              T *__restrict__ f0, T *__restrict__ e0, int i) {
    const long N = g.N;
    T v[B], u[B];
#pragma unroll
    for (int c = 0; c < B; c++) u[c] = (T)r[(long)c * N + i];
    if (lscT) {
#pragma unroll
        for (int rr = 0; rr < B; rr++) {
            T t = lscT[(long)(rr * B) * N + i] * u[0] + lscT[(long)(rr * B + 1) * N + i] * u[1];
            if (B == 3) t += lscT[(long)(rr * B + 2) * N + i] * u[2];
            v[rr] = t;
        }
    } else {
#pragma unroll
        for (int c = 0; c < B; c++) v[c] = u[c];
        T rp = v[0] + wT[(long)N + i] * v[1];
        if (B == 3) rp += wT[2L * N + i] * v[2];
        v[0] = rp;
    }
    const Cell cc = cell_of(g, i);
    const long NS = 2L * g.H, si = cslot(g, cc.ix, cc.iy, cc.iz);
#pragma unroll
    for (int d = 0; d < 7; d++) {
        const int j = nbrc(g, cc, d);
        if (j < 0) continue;
        T xj[B];
#pragma unroll
        for (int c = 0; c < B; c++) xj[c] = x0[(long)c * N + j];
#pragma unroll
        for (int rr = 0; rr < B; rr++)
#pragma unroll
            for (int c = 0; c < B; c++) v[rr] -= ahat[(long)(d * B * B + rr * B + c) * NS + si] * xj[c];
    }
#pragma unroll
    for (int c = 0; c < B; c++) rh[(long)c * N + i] = v[c];
    f0[i] = v[0];
    e0[i] = v[0] * dinv0[i];
}

template <int B, typename T>
__global__ void fpf_resid_kernel(GridDesc g, const double *__restrict__ r, const T *__restrict__ wT,
                                 const T *__restrict__ lscT, const T *__restrict__ ahat, const T *__restrict__ x0,
                                 const T *__restrict__ dinv0, T *__restrict__ rh, T *__restrict__ f0, T *__restrict__ e0,
                                 const L2Prefetch pf, const int *done) {
    if (skip(done)) return;
    issue_prefetch(pf);
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < g.N) fpf_resid_row<B, T>(g, r, wT, lscT, ahat, x0, dinv0, rh, f0, e0, i);
}

// stage-F output of component r: x (+ e_p on the pressure row) (+ addv, the first
// stage F of CPR-FPF), added in the order the stages ran
template <typename T>
__device__ __forceinline__ T fin(T x, int r, int i, long N, const T *__restrict__ ep, const T *__restrict__ addv) {
    if (r == 0 && ep) x += ep[i];
    if (addv) x += addv[(long)r * N + i];
    return x;
}

// stage F, pass 2 (black cells): z = Dinv (r2 - sum_d Ahat_{i,d} z_red(nbr)); out = z + e_p
template <int B, typename T, typename TZ>
__device__ __forceinline__ void stage2_b_row(const GridDesc &g, const T *__restrict__ ahat, const T *__restrict__ dinv,
                                             const T *__restrict__ r2, T *__restrict__ z, const T *__restrict__ ep,
                                             const T *__restrict__ addv, TZ *__restrict__ out, int i) {
    const long N = g.N;
    const Cell cc = cell_of(g, i);
    const long NS = 2L * g.H, si = cslot(g, cc.ix, cc.iy, cc.iz);
    T t[B];
#pragma unroll
    for (int c = 0; c < B; c++) t[c] = r2[(long)c * N + i];
#pragma unroll
    for (int d = 1; d < 7; d++) {
        const int k = nbrc(g, cc, d);
        if (k < 0) continue;
        T zk[B];
#pragma unroll
        for (int c = 0; c < B; c++) zk[c] = z[(long)c * N + k];
#pragma unroll
        for (int r = 0; r < B; r++)
#pragma unroll
            for (int c = 0; c < B; c++) t[r] -= ahat[(long)(d * B * B + r * B + c) * NS + si] * zk[c];
    }
#pragma unroll
    for (int r = 0; r < B; r++) {
        T s = (T)0;
#pragma unroll
        for (int q = 0; q < B; q++) s += dinv[(long)(r * B + q) * NS + si] * t[q];
        z[(long)r * N + i] = s;
        out[(long)r * N + i] = (TZ)fin<T>(s, r, i, N, ep, addv);
    }
}

template <int B, typename T, typename TZ>
__global__ void stage2_b_kernel(GridDesc g, const T *__restrict__ ahat, const T *__restrict__ dinv,
                                const T *__restrict__ r2, T *__restrict__ z, const T *__restrict__ ep,
                                const T *__restrict__ addv, TZ *__restrict__ out, const int *done) {
    if (skip(done)) return;
    const int i = colour_cell(g, blockIdx.x * (long)blockDim.x + threadIdx.x, 1);
    if (i < 0) return;
    stage2_b_row<B, T, TZ>(g, ahat, dinv, r2, z, ep, addv, out, i);
}

// stage F, pass 3 (red cells): x = z - Dinv sum_d Ahat_{i,d} z_black(nbr); out = x + e_p
// (rb = 0: block-Jacobi, out = z + e_p for every cell)
template <int B, typename T, typename TZ>
__device__ __forceinline__ void stage2_c_row(const GridDesc &g, const T *__restrict__ ahat, const T *__restrict__ dinv,
                                             const T *__restrict__ z, const T *__restrict__ ep,
                                             const T *__restrict__ addv, TZ *__restrict__ out, int rb, int i) {
    const long N = g.N;
    if (!rb) {
#pragma unroll
        for (int r = 0; r < B; r++) {
            out[(long)r * N + i] = (TZ)fin<T>(z[(long)r * N + i], r, i, N, ep, addv);
        }
        return;
    }
    const Cell cc = cell_of(g, i);
    const long NS = 2L * g.H, si = cslot(g, cc.ix, cc.iy, cc.iz);
    T t[B];
#pragma unroll
    for (int c = 0; c < B; c++) t[c] = (T)0;
#pragma unroll
    for (int d = 1; d < 7; d++) {
        const int k = nbrc(g, cc, d);
        if (k < 0) continue;
        T zk[B];
#pragma unroll
        for (int c = 0; c < B; c++) zk[c] = z[(long)c * N + k];
#pragma unroll
        for (int r = 0; r < B; r++)
#pragma unroll
            for (int c = 0; c < B; c++) t[r] += ahat[(long)(d * B * B + r * B + c) * NS + si] * zk[c];
    }
#pragma unroll
    for (int r = 0; r < B; r++) {
        T s = (T)0;
#pragma unroll
        for (int q = 0; q < B; q++) s += dinv[(long)(r * B + q) * NS + si] * t[q];
        out[(long)r * N + i] = (TZ)fin<T>(z[(long)r * N + i] - s, r, i, N, ep, addv);
    }
}

template <int B, typename T, typename TZ>
__global__ void stage2_c_kernel(GridDesc g, const T *__restrict__ ahat, const T *__restrict__ dinv, const T *__restrict__ z,
                                const T *__restrict__ ep, const T *__restrict__ addv, TZ *__restrict__ out, int rb,
                                const int *done) {
    if (skip(done)) return;
    const int i = rb ? colour_cell(g, blockIdx.x * (long)blockDim.x + threadIdx.x, 0)   // red cells
                     : (blockIdx.x * blockDim.x + threadIdx.x < (unsigned)g.N ? (int)(blockIdx.x * blockDim.x + threadIdx.x) : -1);
    if (i < 0) return;
    stage2_c_row<B, T, TZ>(g, ahat, dinv, z, ep, addv, out, rb, i);
}

// ---- the whole CPR application of a small grid in one launch -----------------
// Up to kSmallCells cells an application is 10 to 25 dependent launches of 2.5 to 5 us
// each, whose work is a fraction of that; here they are sweeps of one 16-CTA cluster with a
// cluster barrier (about 1 us) between them, calling the same row functions in the
// same order, level 0 of the V-cycle among them, so the result is that of the
// separate launches bit for bit.  2,000 two-phase cells: an application 72 -> 48 us, an
// FGMRES iteration (its launches replayed from a graph) 86 -> 77 us.  The latency of
// 16 SMs sets the bound: an iteration at 4,000 cells goes from 82 to 78 us, at 7,840
// from 88 to 92.
constexpr int kSmallCells = 5120, kSmallThreads = 512;

template <typename T>
struct SmallApply {
    CoarseCycle<T> cc;                 // every level
    const T *wT, *lscT, *ahat, *dinv;
    T *r2, *zr, *x0, *rhT, *rpT, *epacc;
    int full, rb, fpf, cycles;
};

// out = M r by CTA `rank` of the nb CTAs of one cluster
template <int B, typename T, typename TZ>
__device__ __forceinline__ void small_apply_body(const SmallApply<T> &S, const double *__restrict__ r, TZ *__restrict__ out,
                                                 int rank, int nb) {
    const GridDesc &g = S.cc.g;
    const CoarseLevel<T> &L0 = S.cc.lv[0];
    const int N = g.N, slots = g.H;
    const bool one = S.cc.nlev == 1;   // a single level is solved by its dense inverse
    auto cells = [&](int n, auto f) {
        const int per = (n + nb - 1) / nb, hi = min(n, (rank + 1) * per);
        for (int i = rank * per + (int)threadIdx.x; i < hi; i += kSmallThreads) f(i);
    };
    // one stage F (three sweeps) into o
    auto stage_f = [&](const double *ri, const T *rh, const T *ep, const T *addv, auto *o) {
        using TO = std::remove_pointer_t<decltype(o)>;
        cells(N, [&](int i) { stage2_a_row<B, T>(g, ri, S.wT, S.lscT, rh, S.ahat, S.dinv, ep, S.r2, S.zr, S.rb, i); });
        cluster_barrier();
        if (S.rb) {
            cells(slots, [&](int t) {
                const int i = colour_cell(g, t, 1);
                if (i >= 0) stage2_b_row<B, T, TO>(g, S.ahat, S.dinv, S.r2, S.zr, ep, addv, o, i);
            });
            cluster_barrier();
            cells(slots, [&](int t) {
                const int i = colour_cell(g, t, 0);
                if (i >= 0) stage2_c_row<B, T, TO>(g, S.ahat, S.dinv, S.zr, ep, addv, o, 1, i);
            });
        } else {
            cells(N, [&](int i) { stage2_c_row<B, T, TO>(g, S.ahat, S.dinv, S.zr, ep, addv, o, 0, i); });
        }
    };
    if (S.fpf) {
        stage_f(r, (const T *)nullptr, (const T *)nullptr, (const T *)nullptr, S.x0);
        cluster_barrier();
        cells(N, [&](int i) { fpf_resid_row<B, T>(g, r, S.wT, S.lscT, S.ahat, S.x0, L0.dinv, S.rhT, L0.f, L0.e, i); });
    } else {
        cells(N, [&](int i) { restrict_p_row<B, T>(N, r, S.wT, S.full, L0.dinv, L0.f, L0.e, i); });
    }
    cluster_barrier();
    coarse_cycle_body<T>(S.cc, rank, nb);
    const T *ep = one ? L0.e : L0.e2;
    if (S.cycles > 1 && !one) {
        cluster_barrier();
        cells(N, [&](int i) { S.rpT[i] = L0.f[i]; S.epacc[i] = L0.e2[i]; });
        Mat<T> A;
        A.st = true; A.selfpad = true; A.diff = L0.diff != 0; A.g = g; A.val = L0.val; A.col = nullptr; A.n = N; A.width = 7;
        for (int c = 1; c < S.cycles; c++) {
            cluster_barrier();
            cells(N, [&](int i) { cycle_next_row<T>(A, S.rpT, S.epacc, L0.dinv, L0.f, L0.e, i); });
            cluster_barrier();
            coarse_cycle_body<T>(S.cc, rank, nb);
            cluster_barrier();
            cells(N, [&](int i) { S.epacc[i] = S.epacc[i] + L0.e2[i]; });
        }
        ep = S.epacc;
    }
    cluster_barrier();
    stage_f(S.fpf ? nullptr : r, S.rhT, ep, S.fpf ? S.x0 : (const T *)nullptr, out);
}

template <int B, typename T, typename TZ>
__global__ void __launch_bounds__(kSmallThreads, 1) small_apply_kernel(const __grid_constant__ SmallApply<T> S,
                                                                      const double *r, TZ *out, const int *done) {
    if (skip(done)) return;            // uniform over the cluster
    small_apply_body<B, T, TZ>(S, r, out, (int)blockIdx.x, (int)gridDim.x);
}

// no preconditioner / plain block-Jacobi on J (no decoupling)
template <int B, typename TZ>
__global__ void simple_prec_kernel(GridDesc g, const double *__restrict__ r, const double *__restrict__ dinv, TZ *__restrict__ z,
                                   int use_dinv, const int *done) {
    if (skip(done)) return;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const long N = g.N;
    if (i >= N) return;
    const long NS = 2L * g.H, si = cslot_of(g, i);
    double v[B];
#pragma unroll
    for (int c = 0; c < B; c++) v[c] = r[(long)c * N + i];
#pragma unroll
    for (int rr = 0; rr < B; rr++) {
        double s = v[rr];
        if (use_dinv) {
            s = 0.0;
#pragma unroll
            for (int q = 0; q < B; q++) s += dinv[(long)(rr * B + q) * NS + si] * v[q];
        }
        z[(long)rr * N + i] = (TZ)s;
    }
}

// ---- learned stage helpers ------------------------------------------------
// RMS of a vector into *out (per-block partials folded in block order by the last block)
template <typename T>
__global__ void rms_kernel(int n, const T *__restrict__ v, double *partials, unsigned int *ticket, double *out,
                           const int *done) {
    if (skip(done)) return;
    __shared__ double sh[SIM_THREADS];
    __shared__ bool last;
    double s = 0.0;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) s += (double)v[i] * (double)v[i];
    sh[threadIdx.x] = s;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if ((int)threadIdx.x < o) sh[threadIdx.x] += sh[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) partials[blockIdx.x] = sh[0];
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = (atomicAdd(ticket, 1u) == gridDim.x - 1);
    __syncthreads();
    if (!last) return;
    __threadfence();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int b = 0; b < (int)gridDim.x; b++) t += __ldcg(partials + b);
        *out = sqrt(t / n);
        *ticket = 0u;
    }
}

// network input: [r / rms, three standardised log-transmissibility features]
template <typename T>
__global__ void learned_in_kernel(int n, const T *__restrict__ r, const double *__restrict__ rms,
                                  const float *__restrict__ feat, float *__restrict__ x, const int *done) {
    if (skip(done)) return;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double sc = *rms > 0.0 ? 1.0 / *rms : 0.0;
    x[(long)i * 4] = (float)((double)r[i] * sc);
    x[(long)i * 4 + 1] = feat[(long)i * 3];
    x[(long)i * 4 + 2] = feat[(long)i * 3 + 1];
    x[(long)i * 4 + 3] = feat[(long)i * 3 + 2];
}

// q = A_p c with c = y * rms (the network's correction in pressure units)
template <typename T>
__global__ void learned_apply_kernel(Mat<T> A, const float *__restrict__ y, const double *__restrict__ rms,
                                     T *__restrict__ q, const int *done) {
    if (skip(done)) return;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= A.n) return;
    const double sc = *rms;
    T t = (T)0;
    const T yi = (T)((double)y[i] * sc);
    for_row(A, i, [&](int j, T v) {
        const T yj = (T)((double)y[j] * sc);
        t += A.diff ? ((j == i) ? v * yi : v * (yj - yi)) : v * yj;
    });
    q[i] = t;
}

// minimal-residual step alpha = (q . r) / (q . q) into out[1] (0 if q = 0)
template <typename T>
__global__ void mr_step_kernel(int n, const T *__restrict__ q, const T *__restrict__ r, double *partials,
                               unsigned int *ticket, double *out, const int *done) {
    if (skip(done)) return;
    __shared__ double s1[SIM_THREADS], s2[SIM_THREADS];
    __shared__ bool last;
    double a = 0.0, c = 0.0;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        a += (double)q[i] * (double)r[i];
        c += (double)q[i] * (double)q[i];
    }
    s1[threadIdx.x] = a; s2[threadIdx.x] = c;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if ((int)threadIdx.x < o) { s1[threadIdx.x] += s1[threadIdx.x + o]; s2[threadIdx.x] += s2[threadIdx.x + o]; }
        __syncthreads();
    }
    if (threadIdx.x == 0) { partials[2 * blockIdx.x] = s1[0]; partials[2 * blockIdx.x + 1] = s2[0]; }
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = (atomicAdd(ticket, 1u) == gridDim.x - 1);
    __syncthreads();
    if (!last) return;
    __threadfence();
    if (threadIdx.x == 0) {
        double ta = 0.0, tc = 0.0;
        for (int b = 0; b < (int)gridDim.x; b++) { ta += __ldcg(partials + 2 * b); tc += __ldcg(partials + 2 * b + 1); }
        out[1] = tc > 0.0 ? ta / tc : 0.0;
        *ticket = 0u;
    }
}

// ep_out = ep + alpha * y * rms
template <typename T>
__global__ void learned_out_kernel(int n, const T *__restrict__ ep, const float *__restrict__ y,
                                   const double *__restrict__ rms, T *__restrict__ out, const int *done) {
    if (skip(done)) return;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = ep[i] + (T)(rms[1] * (double)y[i] * rms[0]);
}

// training pair j: x_j = [f / rms(f), features], y_j = e / rms(e) (the stage's
// minimal-residual step restores the scale at inference)
template <typename T>
__global__ void pair_kernel(int n, const T *__restrict__ f, const T *__restrict__ e, const double *__restrict__ rms,
                            const float *__restrict__ feat, float *__restrict__ x, float *__restrict__ y) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double sc = rms[0] > 0.0 ? 1.0 / rms[0] : 0.0;
    const double se = rms[1] > 0.0 ? 1.0 / rms[1] : 0.0;
    x[(long)i * 4] = (float)((double)f[i] * sc);
    x[(long)i * 4 + 1] = feat[(long)i * 3];
    x[(long)i * 4 + 2] = feat[(long)i * 3 + 1];
    x[(long)i * 4 + 3] = feat[(long)i * 3 + 2];
    y[i] = (float)((double)e[i] * se);
}

// log of the summed face transmissibilities per direction
__global__ void logt_kernel(GridDesc g, const double *__restrict__ T, float *__restrict__ feat) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= g.N) return;
    const Cell c = cell_of(g, i);
    const long N = g.N;
    const double sx = T[i] + (c.ix > 0 ? T[i - 1] : 0.0);
    const double sy = T[N + i] + (c.iy > 0 ? T[N + i - g.nx] : 0.0);
    const double sz = T[2L * N + i] + (c.iz > 0 ? T[2L * N + i - g.nx * g.ny] : 0.0);
    feat[(long)i * 3] = (float)log(sx + 1e-30);
    feat[(long)i * 3 + 1] = (float)log(sy + 1e-30);
    feat[(long)i * 3 + 2] = (float)log(sz + 1e-30);
}

__global__ void standardize_kernel(int n, float *__restrict__ feat, float m0, float m1, float m2, float s0, float s1,
                                   float s2) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    feat[(long)i * 3] = s0 > 0.f ? (feat[(long)i * 3] - m0) / s0 : 0.f;
    feat[(long)i * 3 + 1] = s1 > 0.f ? (feat[(long)i * 3 + 1] - m1) / s1 : 0.f;
    feat[(long)i * 3 + 2] = s2 > 0.f ? (feat[(long)i * 3 + 2] - m2) / s2 : 0.f;
}

}  // namespace

// ===========================================================================
// host side
// ===========================================================================
bool sim_mixed(const sim_t *s) { return s->opt.precision == SIM_PRECISION_MIXED; }

static void *dev_alloc_async(sim_t *s, size_t bytes) {
    void *p = nullptr;
    if (bytes == 0) bytes = 16;
    cudaError_t e = cudaMallocAsync(&p, bytes, s->stream);
    if (e != cudaSuccess) { sim_cuda_ok(s, e, "cudaMallocAsync (AMG hierarchy)"); return nullptr; }
    return p;
}
static void dev_free_async(sim_t *s, void *p) { if (p) cudaFreeAsync(p, s->stream); }

static void free_level(sim_t *s, AmgLevel &L) {
    dev_free_async(s, L.work); dev_free_async(s, L.len); dev_free_async(s, L.val);
    dev_free_async(s, L.agg); dev_free_async(s, L.moff); dev_free_async(s, L.mem); dev_free_async(s, L.coarse_inv);
    L = AmgLevel();
}

void cpr_free(sim_t *s) {
    for (auto &L : s->lev) free_level(s, L);
    s->lev.clear();
}

static Mat<double> level_mat(sim_t *s, const AmgLevel &L, int l) {
    Mat<double> A;
    A.st = (l == 0); A.selfpad = false; A.diff = false; A.g = s->gd; A.n = L.n; A.width = L.width;
    A.val = l == 0 ? s->ap : L.val;
    A.col = L.col;
    A.len = L.len;
    return A;
}
template <typename T>
static Mat<T> level_matT(sim_t *s, const AmgLevel &L, int l) {
    Mat<T> A;
    A.st = (l == 0); A.selfpad = true; A.diff = sizeof(T) == sizeof(float); A.g = s->gd; A.n = L.n; A.width = L.width;
    A.val = (const T *)L.valT;
    A.col = L.colA;
    A.len = L.len;
    return A;
}

// ---- coarsening -------------------------------------------------------------
// scalars of the set-up in s->iscal: the aggregate count of the last pass, then
// {largest row, flags} of the level's matrix and of its intermediate one; behind them the entry counts (64 bits each) of up to kScLevels levels
constexpr int kScNc = 0, kScBad = 4, kScM = 8, kScM1 = 10, kScCount = SIM_SETUP_SCALARS, kScLevels = SIM_SETUP_LEVELS;

static bool read_scalars(sim_t *s, int (&v)[kScCount]) {
    if (!sim_cuda_ok(s, cudaMemcpyAsync(s->h_pinned, s->iscal, sizeof(int) * kScCount, cudaMemcpyDeviceToHost, s->stream), "copy") ||
        !sim_cuda_ok(s, cudaStreamSynchronize(s->stream), "AMG set-up"))
        return false;
    memcpy(v, s->h_pinned, sizeof(v));
    return true;
}

// one aggregation pass on A (n rows), enqueued: matching rounds, absorption of
// single nodes, numbering by founders, members.  On the second pass of a level the
// composite with the first (agg, members of the fine nodes) as well.
static bool enqueue_pass(sim_t *s, const Mat<double> &A, bool second, int *aggC, int *moffC, int *memC) {
    const int n = A.n;
    MatchState st;
    st.partner = s->partner; st.host = s->host; st.acnt = s->cnt; st.alist = s->absorbed;
    int *pk[2] = {s->pick, s->pick2};
    const int nb = A.st ? sim_blocks(n) : sim_blocks(8L * n);
    auto match = [&](bool host, const int *in, int *out) {
        if (A.st) {
            if (host) match_kernel<true, 1><<<nb, SIM_THREADS, 0, s->stream>>>(A, st, in, out, s->opt.amg_theta);
            else match_kernel<false, 1><<<nb, SIM_THREADS, 0, s->stream>>>(A, st, in, out, s->opt.amg_theta);
        } else {
            if (host) match_kernel<true, 8><<<nb, SIM_THREADS, 0, s->stream>>>(A, st, in, out, s->opt.amg_theta);
            else match_kernel<false, 8><<<nb, SIM_THREADS, 0, s->stream>>>(A, st, in, out, s->opt.amg_theta);
        }
        s->launches++;
    };
    for (int r = 0; r < s->opt.amg_rounds; r++) match(false, r ? pk[(r - 1) & 1] : nullptr, pk[r & 1]);
    match(true, pk[(s->opt.amg_rounds - 1) & 1], nullptr);
    AggPass P;
    P.st = st; P.n = n;
    P.moffF = second ? s->moffA : nullptr; P.memF = second ? s->memA : nullptr;
    P.agg = second ? s->aggB : s->aggA; P.moff = second ? s->moffB : s->moffA; P.mem = second ? s->memB : s->memA;
    P.aggC = aggC; P.moffC = moffC; P.memC = memC;
    P.csum = s->scan; P.nc = s->iscal + kScNc;
    // chunks of 256 nodes spread a small level over the SMs; from 256k nodes chunks of 1,024
    // keep the sums every block adds up for its base short.  Those grow with the square of
    // the chunks: above 4,096 of them one block scans the sums first (64M nodes: 0.14 ms and
    // the writing launch 2.13 ms, 8.67 without; 16.8M nodes: 0.05 and 0.63, 1.08 without).
    const int threads = n <= (1 << 18) ? 256 : 1024;
    const int chunks = sim_blocks(n, threads);
    P.scanned = chunks > 4096;
    agg_sizes_kernel<<<chunks, threads, 0, s->stream>>>(P, A);
    if (P.scanned) agg_scan_kernel<<<1, 1024, 0, s->stream>>>(P, A, chunks);
    agg_write_kernel<<<chunks, threads, 0, s->stream>>>(P, A);
    s->launches += P.scanned ? 3 : 2;
    return sim_cuda_ok(s, cudaGetLastError(), "aggregation pass");
}

// Memory the set-up may write until it returns: the preconditioned directions of the
// Krylov solver, whose contents no call keeps.  It holds the products while their widths
// are unknown (48 or 64 slots a row; the longest rows have 19 to 49), so the pool holds
// the levels at their widths only: 160 B a cell of the pool at 4.2M black-oil cells, 412
// with the products there too (177 with each width counted by a launch of its own first).
// What it costs is a copy per large level: 0.6 ms of 40 at 16.8M cells.
struct SetupScratch {
    char *p;
    size_t size;
};

// a Galerkin product P^T A P enqueued into ELL arrays of capacity Wcap; its width is
// read with the next scalars
struct GalerkinJob {
    bool on = false, own = false;      // own: arrays of the pool's, else of the scratch
    Mat<double> A;
    const int *agg = nullptr, *moff = nullptr, *mem = nullptr;
    int nc = 0, Wcap = 0, sc = 0;
    SetupScratch scr = {nullptr, 0};   // what it may take of the scratch
    size_t taken = 0;                  // and took
    int *len = nullptr;                // row lengths, from ell_head(nc) on the columns
    double *val = nullptr;
    int *col() const;
};
// ints before the columns in the block of an ELL matrix of n rows
static size_t ell_head(int n) { return ((size_t)n + 63) & ~(size_t)63; }
int *GalerkinJob::col() const { return len + ell_head(nc); }
static size_t up256(size_t b) { return (b + 255) & ~(size_t)255; }
static size_t ell_ints(int n, int W) { return up256(sizeof(int) * (ell_head(n) + (size_t)W * n)); }
static size_t ell_vals(int n, int W) { return up256(sizeof(double) * (size_t)W * n); }

static void galerkin_release(sim_t *s, GalerkinJob &g) {
    if (g.own) { dev_free_async(s, g.len); dev_free_async(s, g.val); }
    g.len = nullptr; g.val = nullptr; g.own = false; g.taken = 0;
}
static bool galerkin_alloc(sim_t *s, GalerkinJob &g, int W) {
    galerkin_release(s, g);
    g.Wcap = W;
    const size_t bi = ell_ints(g.nc, W), bv = ell_vals(g.nc, W);
    if (bi + bv <= g.scr.size) {
        g.len = (int *)g.scr.p;
        g.val = (double *)(g.scr.p + bi);
        g.taken = bi + bv;
    } else {
        g.own = true;
        g.len = (int *)dev_alloc_async(s, bi);
        g.val = (double *)dev_alloc_async(s, bv);
        if (!g.len || !g.val) return false;
    }
    return sim_cuda_ok(s, cudaMemsetAsync(g.col(), 0xff, sizeof(int) * (size_t)W * g.nc, s->stream), "memset") &&
           sim_cuda_ok(s, cudaMemsetAsync(s->iscal + g.sc, 0, 2 * sizeof(int), s->stream), "memset");
}
static bool galerkin_rows(sim_t *s, GalerkinJob &g) {
    galerkin_row_kernel<<<(g.nc + kGalWarps - 1) / kGalWarps, kGalWarps * 32, 0, s->stream>>>(
        g.A, g.agg, g.moff, g.mem, g.nc, g.Wcap, g.col(), g.val, g.len, s->iscal + g.sc, s->iscal + g.sc + 1);
    s->launches++;
    return sim_cuda_ok(s, cudaGetLastError(), "Galerkin");
}
// scr: the scratch it may take; roomy: the pool may hold its capacity for a while
static bool enqueue_galerkin(sim_t *s, GalerkinJob &g, const Mat<double> &A, const int *agg, const int *moff, const int *mem,
                             int nc, int sc, SetupScratch scr, bool roomy) {
    g = GalerkinJob();
    g.on = true; g.A = A; g.agg = agg; g.moff = moff; g.mem = mem; g.nc = nc; g.sc = sc; g.scr = scr;
    // Rows of these hierarchies have 15 to 49 columns: a product that 40 slots a row do
    // not hold is rare, and completed by resolve_galerkin.  Where neither the scratch
    // (few Krylov directions) nor a small level leaves room for that, one slot a row: the
    // row kernel then counts, and resolve_galerkin builds the product at its width.
    const int want = nc <= (1 << 20) ? 64 : 48;
    int W = want;
    while (W > 40 && ell_ints(nc, W) + ell_vals(nc, W) > scr.size) W--;
    if (ell_ints(nc, W) + ell_vals(nc, W) > scr.size) W = roomy || nc <= (1 << 17) ? want : 1;
    return galerkin_alloc(s, g, W) && galerkin_rows(s, g);
}
// width of an enqueued product from its scalars; 0: a row wider than SIM_MAX_ELL
// (the caller stops coarsening), -1: error.  A list the row kernel does not take or
// a row beyond the capacity has the product completed (*rebuilt: kernels enqueued
// on it in the meantime did nothing).
static int resolve_galerkin(sim_t *s, GalerkinJob &g, const int (&v)[kScCount], bool *rebuilt) {
    int W = v[g.sc], flags = v[g.sc + 1];
    *rebuilt = false;
    g.on = false;
    while (flags || W > g.Wcap) {
        *rebuilt = true;
        if (flags & 2) return 0;
        if (!flags) {                              // only too wide: again, with room for it
            if (!galerkin_alloc(s, g, W) || !galerkin_rows(s, g)) return -1;
        } else if (!sim_cuda_ok(s, cudaMemsetAsync(s->iscal + g.sc + 1, 0, sizeof(int), s->stream), "memset")) {
            return -1;
        }
        int u[kScCount];
        galerkin_kernel<<<sim_blocks(g.nc), SIM_THREADS, 0, s->stream>>>(g.A, g.agg, g.moff, g.mem, g.nc, g.Wcap, g.col(), g.val,
                                                                         g.len, s->iscal + g.sc, s->iscal + g.sc + 1);
        s->launches++;
        if (!sim_cuda_ok(s, cudaGetLastError(), "Galerkin") || !read_scalars(s, u)) return -1;
        W = u[g.sc];
        flags = flags ? u[g.sc + 1] : u[g.sc + 1] & 2;   // bit 0 set again by the row kernel: its rows are done now
    }
    return W < 1 ? 1 : W;
}
static Mat<double> job_mat(sim_t *s, const GalerkinJob &g) {
    Mat<double> A;
    A.st = false; A.selfpad = false; A.diff = false; A.g = s->gd; A.n = g.nc; A.width = g.Wcap; A.col = g.col(); A.val = g.val; A.len = g.len;
    A.wp = s->iscal + g.sc;
    return A;
}

// apply-precision data of the levels: one allocation per level, one launch for all
// the ELL levels
template <typename T>
static sim_status level_work(sim_t *s, AmgLevel &L, bool ell) {
    const size_t vec = up256(sizeof(T) * L.n), colb = ell ? up256(sizeof(int) * (size_t)L.width * L.n) : 0;
    const bool copy = ell && sizeof(T) != sizeof(double);     // the FP64 form applies the set-up's values
    const size_t valb = copy ? up256(sizeof(T) * (size_t)L.width * L.n) : 0;
    char *p = (char *)dev_alloc_async(s, 4 * vec + colb + valb);
    if (!p) return s->err;
    L.work = p;
    L.dinvT = p; L.f = p + vec; L.e = p + 2 * vec; L.e2 = p + 3 * vec;
    if (ell) {
        L.colA = (int *)(p + 4 * vec);
        L.valT = copy ? (void *)(p + 4 * vec + colb) : (void *)L.val;
    }
    return SIM_OK;
}

template <typename T>
static sim_status finish_levels(sim_t *s) {
    // l1 inverse diagonals, apply-precision values, work vectors; coarsest dense inverse
    const int nl = (int)s->lev.size();
    // the pivot flag and the levels' entry counts come back together
    int *bad = s->iscal + kScBad;
    SIM_CK(s, cudaMemsetAsync(bad, 0, sizeof(int) * (kScCount - kScBad + 2 * kScLevels), s->stream));
    s->lev[0].entries = 7.0 * s->N;
    for (int l0 = 1; l0 < nl; l0 += kFinishLevels) {
        FinishTable tb;
        tb.count = 0; tb.rows = 0;
        tb.entries = (unsigned long long *)(s->iscal + kScCount) + l0;
        for (int l = l0; l < nl && l < l0 + kFinishLevels; l++) {
            AmgLevel &L = s->lev[l];
            if (level_work<T>(s, L, true) != SIM_OK) return s->err;
            FinishLevel &f = tb.lv[tb.count++];
            f.n = L.n; f.width = L.width; f.row0 = tb.rows; f.col = L.col; f.len = L.len; f.val = L.val; f.colA = L.colA; f.valT = L.valT;
            f.dinvT = L.dinvT;
            tb.rows += L.n;
        }
        finish_levels_kernel<T><<<sim_blocks(tb.rows, 128), 128, 0, s->stream>>>(tb);
        SIM_LAUNCHED(s);
    }
    // coarsest: dense Gauss-Jordan inverse in FP64
    AmgLevel &C = s->lev[nl - 1];
    const int n = C.n;
    // the coarsest inverse stays FP64 in both forms: the coarse matrices of
    // strongly heterogeneous fields are ill-conditioned, and the product is tiny
    C.coarse_inv = dev_alloc_async(s, sizeof(double) * (size_t)n * n);
    if (!C.coarse_inv) return s->err;
    static PerDevice asked;
    const int gj_ctas = asked.get(sim_device(), gj_cluster_ctas);
    if (gj_ctas > 0 && n <= kGjSmem) {
        cudaLaunchConfig_t cfg = {};
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = gj_ctas; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
        cfg.gridDim = dim3(gj_ctas); cfg.blockDim = dim3(kGjThreads); cfg.dynamicSmemBytes = gj_inverse_bytes(n, gj_ctas);
        cfg.stream = s->stream; cfg.attrs = at; cfg.numAttrs = 1;
        if (!sim_cuda_ok(s, cudaLaunchKernelEx(&cfg, gj_inverse_kernel, level_mat(s, C, nl - 1), (double *)C.coarse_inv, bad),
                         "coarsest inverse"))
            return s->err;
        s->launches++;
    } else {
        const size_t aug = (size_t)n * 2 * n;
        double *A0 = (double *)dev_alloc_async(s, sizeof(double) * aug);
        double *A1 = (double *)dev_alloc_async(s, sizeof(double) * aug);
        double *rn = (double *)dev_alloc_async(s, sizeof(double) * n);
        if (!A0 || !A1 || !rn) return s->err;
        gj_init_kernel<<<sim_blocks(2L * n * n), SIM_THREADS, 0, s->stream>>>(level_mat(s, C, nl - 1), A0);
        gj_rownorm_kernel<<<sim_blocks(n), SIM_THREADS, 0, s->stream>>>(level_mat(s, C, nl - 1), rn);
        gj_cluster_kernel<<<8, 1024, 0, s->stream>>>(n, A0, A1, rn, bad);
        gj_extract_kernel<double><<<sim_blocks((long)n * n), SIM_THREADS, 0, s->stream>>>(n, (n & 1) ? A1 : A0,
                                                                                        (double *)C.coarse_inv);
        s->launches += 4;
        dev_free_async(s, A0); dev_free_async(s, A1); dev_free_async(s, rn);
    }
    SIM_CK(s, cudaGetLastError());
    // the pivot test of the elimination (no pivoting: a vanishing pivot would
    // leave inf / NaN in the coarsest inverse)
    SIM_CK(s, cudaMemcpyAsync(s->h_pinned, s->iscal, sizeof(int) * (kScCount + 2 * kScLevels), cudaMemcpyDeviceToHost, s->stream));
    SIM_CK(s, cudaStreamSynchronize(s->stream));
    int hb = 0;
    memcpy(&hb, (const int *)s->h_pinned + kScBad, sizeof(int));
    const unsigned long long *entries = (const unsigned long long *)((const int *)s->h_pinned + kScCount);
    for (int l = 1; l < nl; l++) s->lev[l].entries = (double)entries[l];
    if (hb) return sim_fail(s, SIM_ENAN, "coarsest AMG level: a Gauss-Jordan pivot is not above 1e-14 of its row's l1 norm");
    return SIM_OK;
}

// the product of g at its width W becomes level L's matrix.  Levels of more than
// kExactRows rows are moved into arrays of that width (one copy each: slots lie row after
// row); a smaller one keeps its capacity, 30 MB at most beyond its width (at 200k cells 15 of
// 690 MB for 1.8 % of a set-up: 1549 us against a start of 1541 with the line at 16,384 rows,
// 1526 against 1546 here).
constexpr int kExactRows = 1 << 16;
static bool take_product(sim_t *s, GalerkinJob &g, AmgLevel &L, int W) {
    L.width = W;
    if (g.own && (W == g.Wcap || g.nc <= kExactRows)) {
        L.len = g.len; L.val = g.val;
        g.own = false;
    } else {
        L.len = (int *)dev_alloc_async(s, ell_ints(g.nc, W));
        L.val = (double *)dev_alloc_async(s, ell_vals(g.nc, W));
        if (!L.len || !L.val ||
            !sim_cuda_ok(s, cudaMemcpyAsync(L.len, g.len, sizeof(int) * (ell_head(g.nc) + (size_t)W * g.nc),
                                            cudaMemcpyDeviceToDevice, s->stream), "copy") ||
            !sim_cuda_ok(s, cudaMemcpyAsync(L.val, g.val, sizeof(double) * (size_t)W * g.nc, cudaMemcpyDeviceToDevice,
                                            s->stream), "copy"))
            return false;
    }
    L.col = L.len + ell_head(g.nc);
    galerkin_release(s, g);
    return true;
}

// coarsen from level 0 (whose work vectors the caller has allocated); jm: the current
// level's matrix while its width is unread, j1: the intermediate one it is built from
static sim_status coarsen(sim_t *s, GalerkinJob &jm, GalerkinJob &j1) {
    const int cmax = s->opt.amg_coarse_max;
    const SetupScratch scr = {(char *)s->Z, (sim_mixed(s) ? sizeof(float) : sizeof(double)) * (size_t)s->m * s->N * s->b};
    int v[kScCount];
    bool rebuilt = false;
    // jm's width arrives with the scalars in v: its level takes it, or the level goes
    // when a row is too wide (the level above is then the coarsest)
    auto settle = [&](bool *gone) -> bool {
        *gone = rebuilt = false;
        if (!jm.on) return true;
        const int W = resolve_galerkin(s, jm, v, &rebuilt);
        if (W < 0) return false;
        galerkin_release(s, j1);                       // after a rebuild in stream order
        if (W == 0) {
            galerkin_release(s, jm);
            s->lev.pop_back();
            AmgLevel &P = s->lev.back();
            dev_free_async(s, P.agg); dev_free_async(s, P.moff); dev_free_async(s, P.mem);
            P.agg = P.moff = P.mem = nullptr;
            *gone = true;
            return true;
        }
        return take_product(s, jm, s->lev.back(), W);
    };
    bool gone = false;
    while (true) {
        const int l = (int)s->lev.size() - 1;
        if (s->lev[l].n <= cmax || (int)s->lev.size() >= s->opt.amg_max_levels) break;
        const int n = s->lev[l].n;
        Mat<double> A = jm.on ? job_mat(s, jm) : level_mat(s, s->lev[l], l);
        do {
            if (!enqueue_pass(s, A, false, nullptr, nullptr, nullptr) || !read_scalars(s, v) || !settle(&gone)) return s->err;
            if (!gone) A = level_mat(s, s->lev[l], l);
        } while (rebuilt && !gone);
        if (gone) break;
        const int n1 = v[kScNc];
        if (!enqueue_galerkin(s, j1, A, s->aggA, s->moffA, s->memA, n1, kScM1, scr, false)) return s->err;
        AmgLevel &L = s->lev[l];
        L.agg = (int *)dev_alloc_async(s, sizeof(int) * (size_t)n);
        L.moff = (int *)dev_alloc_async(s, sizeof(int) * (size_t)(n1 + 1));
        L.mem = (int *)dev_alloc_async(s, sizeof(int) * (size_t)n);
        if (!L.agg || !L.moff || !L.mem) return s->err;
        Mat<double> A1 = job_mat(s, j1);
        int W1 = 0;
        do {
            if (!enqueue_pass(s, A1, true, L.agg, L.moff, L.mem) || !read_scalars(s, v)) return s->err;
            rebuilt = false;
            if (j1.on) {
                W1 = resolve_galerkin(s, j1, v, &rebuilt);
                if (W1 < 0) return s->err;
                A1 = job_mat(s, j1);
                A1.wp = nullptr; A1.width = W1;
            }
        } while (rebuilt && W1 > 0);
        const int n2 = v[kScNc];
        // a row of the intermediate matrix wider than SIM_MAX_ELL, or more than three
        // quarters of the rows left: this level is the coarsest
        if (W1 == 0 || 4L * n2 > 3L * n) {
            galerkin_release(s, j1);
            dev_free_async(s, L.agg); dev_free_async(s, L.moff); dev_free_async(s, L.mem);
            L.agg = L.moff = L.mem = nullptr;
            break;
        }
        const bool rest = n2 > kExactRows;             // else the level keeps what it is built in
        const SetupScratch after = {scr.p + j1.taken, rest ? scr.size - j1.taken : 0};
        if (!enqueue_galerkin(s, jm, A1, s->aggB, s->moffB, s->memB, n2, kScM, after, !j1.own)) return s->err;
        s->lev.emplace_back();
        s->lev.back().n = n2;
    }
    if (jm.on && (!read_scalars(s, v) || !settle(&gone))) return s->err;
    return SIM_OK;
}

static sim_status amg_setup(sim_t *s) {
    GalerkinJob jm, j1;
    const sim_status st = coarsen(s, jm, j1);
    galerkin_release(s, jm); galerkin_release(s, j1);  // what a failed set-up leaves
    if (st != SIM_OK) return st;
    if (s->lev.back().n > 1024) return sim_fail(s, SIM_ELIMIT, "AMG coarsest level larger than 1024 rows");
    return sim_mixed(s) ? finish_levels<float>(s) : finish_levels<double>(s);
}

// blocks of a launch over one colour (colour_cell)
static int colour_blocks(const sim_t *s, int threads = SIM_THREADS) {
    return sim_blocks((long)((s->gd.nx + 1) / 2) * s->gd.ny * s->gd.nz, threads);
}

// stage-F sweeps of a batched application in blocks of 64 threads (the default of
// sim_autotune's stage-F shape: at 0.3-0.6 waves the finer blocks spread a
// launch's FP64 work more evenly over the SMs than blocks of 256)
constexpr int kStageThreads = 64;

template <int B, typename T>
static sim_status setup_bt(sim_t *s) {
    const int N = s->N;
    const int nb = sim_blocks(N), nbc = colour_blocks(s);
    WellCorr wc;
    if (s->nrate > 0) {
        wc.cell_perf = s->cell_perf; wc.pwell = s->perf_well;
        wc.apw = s->apw; wc.awp = s->awp; wc.aww = s->aww; wc.nperf = s->nperf;
    }
    if (s->opt.precond == SIM_PRECOND_BJACOBI) {
        diag_inv_kernel<B><<<nb, SIM_THREADS, 0, s->stream>>>(s->gd, s->J, wc, s->lsc, 0, 2, s->dinv_d);
        SIM_LAUNCHED(s);
        return SIM_OK;
    }
    if (s->opt.precond != SIM_PRECOND_CPR) return SIM_OK;
    cpr_free(s);
    s->lev.emplace_back();
    AmgLevel &L0 = s->lev[0];
    L0.n = N; L0.width = 7;
    if (level_work<T>(s, L0, false) != SIM_OK) return s->err;
    L0.valT = s->apT;
    qi_kernel<B, T><<<nb, SIM_THREADS, 0, s->stream>>>(s->gd, s->J, wc, s->opt.decouple == SIM_DECOUPLE_ABF, s->lsc,
                                                       (T *)s->lscT, s->qiw, (T *)s->qiwT, s->ap, (T *)s->apT,
                                                       (T *)s->ahat, (T *)L0.dinvT);
    SIM_LAUNCHED(s);
    if (amg_setup(s) != SIM_OK) return s->err;
    const int rb = s->opt.stage2 == SIM_STAGE2_ILU0_RB, abf = s->opt.decouple == SIM_DECOUPLE_ABF;
    diag_inv_kernel<B><<<rb ? nbc : nb, SIM_THREADS, 0, s->stream>>>(s->gd, s->J, wc, s->lsc, abf, rb ? 1 : 0, s->dinv_d);
    SIM_LAUNCHED(s);
    if (rb) {
        ilu_black_kernel<B><<<nbc, SIM_THREADS, 0, s->stream>>>(s->gd, s->J, wc, s->lsc, abf, s->dinv_d);
        SIM_LAUNCHED(s);
    }
    if (sizeof(T) != sizeof(double)) {
        cast_kernel<T><<<SIM_RED_BLOCKS, SIM_THREADS, 0, s->stream>>>(s->dinv_d, (T *)s->dinv, (long)B * B * 2 * s->gd.H);
        SIM_LAUNCHED(s);
    }
    return SIM_OK;
}

sim_status cpr_setup(sim_t *s) {
    sim_status st;
    if (s->b == 2) st = sim_mixed(s) ? setup_bt<2, float>(s) : setup_bt<2, double>(s);
    else st = sim_mixed(s) ? setup_bt<3, float>(s) : setup_bt<3, double>(s);
    if (st != SIM_OK) return st;
    s->precond_ready = true;
    s->setup_gen++;
    return SIM_OK;
}

// blocks of a launch over the rows of level l (lanes per row on the ELL levels)
static int level_blocks(int n, int l, int threads) { return sim_blocks((long)n * (l > 0 ? ell_lanes(n) : 1), threads); }

// first level handled by the one-launch coarse cycle (nl: no fusion)
static int coarse_start(const sim_t *s) {
    const int nl = (int)s->lev.size();
    if (nl < 3) return nl;
    int l0 = nl - 1;
    while (l0 - 1 >= 1 && s->lev[l0 - 1].n <= coarse_rows(sim_mixed(s)) && nl - (l0 - 1) <= kCoarseMaxLevels) l0--;
    return (nl - l0 >= 3) ? l0 : nl;   // worth a launch only when it replaces several
}

// the arrays the cluster launch of the coarse levels reads (none without it)
template <typename T>
static L2Prefetch coarse_prefetch(const sim_t *s) {
    L2Prefetch pf{};
    const int nl = (int)s->lev.size();
    const int lf = s->opt.fused_coarse ? coarse_start(s) : nl;
    auto add = [&](const void *p, size_t bytes) {
        if (p && bytes >= 16 && pf.count < kPrefetchMax) { pf.p[pf.count] = p; pf.bytes[pf.count] = bytes; pf.count++; }
    };
    for (int l = lf; l < nl; l++) {
        const AmgLevel &L = s->lev[l];
        const size_t ell = (size_t)L.width * L.n;
        if (l + 1 == nl) { add(L.coarse_inv, sizeof(double) * (size_t)L.n * L.n); break; }
        add(L.colA, sizeof(int) * ell);
        add(L.valT, sizeof(T) * ell);
        add(L.dinvT, sizeof(T) * L.n);
        add(L.mem, sizeof(int) * L.n);
    }
    return pf;
}

// a launch of `clusters` clusters of 16 CTAs, or of 8 where an
// occupancy query finds no room for 16 (a non-portable size); the query launches nothing
template <typename... KArgs>
static int coarse_ctas(void (*kernel)(KArgs...), int threads) {
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) {
        (void)cudaGetLastError();
        return 8;
    }
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = 16; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3(16); cfg.blockDim = dim3(threads);
    cfg.attrs = at; cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) != cudaSuccess) {
        (void)cudaGetLastError();
        return 8;
    }
    return n > 0 ? 16 : 8;
}
template <auto Kernel, typename... Args>
static cudaError_t launch_clusters(int clusters, int threads, cudaStream_t st, Args... args) {
    static PerDevice asked;                                    // per kernel: its attributes are its own
    const int ctas = asked.get(sim_device(), [&] { return coarse_ctas(Kernel, threads); });
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = ctas; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;     // as sim_launch
    at[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.gridDim = dim3(clusters * ctas); cfg.blockDim = dim3(threads); cfg.stream = st;
    cfg.attrs = at; cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, Kernel, args...);
}

template <typename T>
static CoarseLevel<T> coarse_level(const AmgLevel &L, int l) {
    CoarseLevel<T> d;
    d.n = L.n; d.width = L.width; d.diff = sizeof(T) == sizeof(float); d.st = l == 0; d.colA = L.colA; d.len = L.len; d.val = (const T *)L.valT;
    d.dinv = (const T *)L.dinvT;
    d.agg = L.agg; d.moff = L.moff; d.mem = L.mem;
    d.f = (T *)L.f; d.e = (T *)L.e; d.e2 = (T *)L.e2;
    return d;
}

// the one-launch application of a small grid
static bool small_grid(const sim_t *s) {
    return s->N <= kSmallCells && s->opt.fused_coarse && (int)s->lev.size() <= kCoarseMaxLevels;
}
template <typename T>
static SmallApply<T> small_apply(const sim_t *s) {
    SmallApply<T> S;
    S.cc.nlev = (int)s->lev.size(); S.cc.g = s->gd; S.cc.inv = (const double *)s->lev.back().coarse_inv;
    for (size_t l = 0; l < s->lev.size(); l++) S.cc.lv[l] = coarse_level<T>(s->lev[l], (int)l);
    S.full = s->opt.decouple == SIM_DECOUPLE_ABF;
    S.wT = (const T *)s->qiwT; S.lscT = S.full ? (const T *)s->lscT : nullptr; S.ahat = (const T *)s->ahat;
    S.dinv = sizeof(T) == sizeof(double) ? (const T *)s->dinv_d : (const T *)s->dinv;
    S.r2 = (T *)s->r2; S.zr = (T *)s->zr; S.x0 = (T *)s->x0; S.rhT = (T *)s->rhT; S.rpT = (T *)s->rpT; S.epacc = (T *)s->epacc;
    S.rb = s->opt.stage2 == SIM_STAGE2_ILU0_RB; S.fpf = s->opt.cpr_stages == 3; S.cycles = s->opt.amg_cycles;
    return S;
}

template <typename T>
static sim_status coarse_cycle(sim_t *s, int l0, const int *done) {
    const int nl = (int)s->lev.size();
    CoarseCycle<T> cc;
    cc.nlev = nl - l0; cc.g = s->gd;
    cc.inv = (const double *)s->lev[nl - 1].coarse_inv;
    for (int l = l0; l < nl; l++) {
        const AmgLevel &L = s->lev[l];
        CoarseLevel<T> &d = cc.lv[l - l0];
        d = coarse_level<T>(L, l);
    }
    if (!sim_cuda_ok(s, launch_clusters<coarse_cycle_kernel<T>>(1, kCoarseThreads, s->stream, cc, done), "coarse cycle")) return s->err;
    SIM_LAUNCHED(s);
    return SIM_OK;
}

// acc: add the result to acc instead of leaving it in e2 of level 0 (further cycles)
template <typename T>
static sim_status vcycle(sim_t *s, const int *done, T *acc = nullptr) {
    const int nl = (int)s->lev.size();
    const int lf = s->opt.fused_coarse ? coarse_start(s) : nl;
    // down: r = f - A e; f_{l+1} = P^T r; e_{l+1} = f_{l+1} / l1 (not on the coarsest)
    for (int l = 0; l + 1 < nl && l < lf; l++) {
        AmgLevel &L = s->lev[l], &C = s->lev[l + 1];
        const bool coarsest = (l + 1 == nl - 1);
        sim_launch(amg_resid_kernel<T>, level_blocks(L.n, l, s->tune_amg), s->tune_amg, s->stream, level_matT<T>(s, L, l), (const T *)L.f,
                                                                        (const T *)L.e, (T *)L.e2, done);
        SIM_LAUNCHED(s);
        sim_launch(amg_restrict_kernel<T>, sim_blocks(C.n, s->tune_amg), s->tune_amg, s->stream, (const T *)L.e2, L.moff, L.mem, C.n, (T *)C.f,
                                                                           coarsest ? nullptr : (T *)C.e,
                                                                           (const T *)C.dinvT, done);
        SIM_LAUNCHED(s);
    }
    if (lf < nl) {
        if (coarse_cycle<T>(s, lf, done) != SIM_OK) return s->err;
    } else {
        AmgLevel &Cn = s->lev[nl - 1];
        sim_launch(coarse_solve_kernel<T>, sim_blocks((long)Cn.n * 32), SIM_THREADS, s->stream, Cn.n, (const double *)Cn.coarse_inv,
                                                                                        (const T *)Cn.f, (T *)Cn.e, done);
        SIM_LAUNCHED(s);
    }
    // up: e_l += P e_{l+1}; e2_l = smooth(e_l); the corrected vector of level l is e2_l
    for (int l = (lf < nl ? lf : nl - 1) - 1; l >= 0; l--) {
        AmgLevel &L = s->lev[l], &C = s->lev[l + 1];
        const T *ec = (l + 1 == nl - 1) ? (const T *)C.e : (const T *)C.e2;
        sim_launch(amg_prolong_kernel<T>, sim_blocks(L.n, s->tune_amg), s->tune_amg, s->stream, L.n, L.agg, ec, (T *)L.e, done);
        SIM_LAUNCHED(s);
        const bool add = l == 0 && acc;
        sim_launch(amg_smooth_kernel<T>, level_blocks(L.n, l, s->tune_amg), s->tune_amg, s->stream, level_matT<T>(s, L, l), (const T *)L.f,
                                                                         (const T *)L.e, (const T *)L.dinvT,
                                                                         add ? acc : (T *)L.e2, done, add);
        SIM_LAUNCHED(s);
    }
    return SIM_OK;
}

template <int B, typename T, typename TZ>
static sim_status apply_btz(sim_t *s, const double *r, TZ *z, const int *done) {
    const int N = s->N;
    const int nb = sim_blocks(N);
    if (s->opt.precond != SIM_PRECOND_CPR) {
        sim_launch(simple_prec_kernel<B, TZ>, nb, SIM_THREADS, s->stream, s->gd, r, s->dinv_d, z,
                                                                   s->opt.precond == SIM_PRECOND_BJACOBI, done);
        SIM_LAUNCHED(s);
        return SIM_OK;
    }
    AmgLevel &L0 = s->lev[0];
    const int rb = s->opt.stage2 == SIM_STAGE2_ILU0_RB;
    const T *dinv = sizeof(T) == sizeof(double) ? (const T *)s->dinv_d : (const T *)s->dinv;
    const int full = s->opt.decouple == SIM_DECOUPLE_ABF;
    const T *lscT = full ? (const T *)s->lscT : nullptr;
    const bool fpf = s->opt.cpr_stages == 3;
    if (small_grid(s) && !s->learned_active) {
        if (!sim_cuda_ok(s, launch_clusters<small_apply_kernel<B, T, TZ>>(1, kSmallThreads, s->stream, small_apply<T>(s), r, z, done),
                         "CPR application"))
            return s->err;
        SIM_LAUNCHED(s);
        return SIM_OK;
    }
    if (fpf) {
        // CPR-FPF: stage F on L r first (x0), then stage P on the residual it leaves
        sim_launch(stage2_a_kernel<B, T>, sim_blocks(N, s->tune_stage), s->tune_stage, s->stream, s->gd, r, (const T *)s->qiwT, lscT, nullptr,
                                                                (const T *)s->ahat, dinv, nullptr, (T *)s->r2,
                                                                (T *)s->zr, rb, done);
        SIM_LAUNCHED(s);
        if (rb) {
            sim_launch(stage2_b_kernel<B, T, T>, colour_blocks(s, s->tune_stage), s->tune_stage, s->stream, s->gd, (const T *)s->ahat, dinv, (const T *)s->r2,
                                                                       (T *)s->zr, nullptr, nullptr, (T *)s->x0, done);
            SIM_LAUNCHED(s);
        }
        sim_launch(stage2_c_kernel<B, T, T>, rb ? colour_blocks(s, s->tune_stage) : sim_blocks(N, s->tune_stage), s->tune_stage, s->stream, s->gd, (const T *)s->ahat, dinv, (const T *)s->zr,
                                                                   nullptr, nullptr, (T *)s->x0, rb, done);
        SIM_LAUNCHED(s);
        sim_launch(fpf_resid_kernel<B, T>, nb, SIM_THREADS, s->stream, s->gd, r, (const T *)s->qiwT, lscT, (const T *)s->ahat,
                                                                 (const T *)s->x0, (const T *)L0.dinvT, (T *)s->rhT,
                                                                 (T *)L0.f, (T *)L0.e, coarse_prefetch<T>(s), done);
        SIM_LAUNCHED(s);
    } else {
        sim_launch(restrict_p_kernel<B, T>, nb, SIM_THREADS, s->stream, N, r, (const T *)s->qiwT, full, (const T *)L0.dinvT,
                                                                  (T *)L0.f, (T *)L0.e, coarse_prefetch<T>(s), done);
        SIM_LAUNCHED(s);
    }
    const T *ep;
    if (s->lev.size() == 1) {
        sim_launch(coarse_solve_kernel<T>, sim_blocks((long)L0.n * 32), SIM_THREADS, s->stream, L0.n, (const double *)L0.coarse_inv,
                                                                                        (const T *)L0.f, (T *)L0.e2, done);
        SIM_LAUNCHED(s);
    } else if (vcycle<T>(s, done) != SIM_OK) {
        return s->err;
    }
    ep = (const T *)L0.e2;
    if (s->opt.amg_cycles > 1 && s->lev.size() > 1) {
        // further cycles on the pressure residual left by the previous ones
        const bool keep = s->opt.amg_cycles > 2 || (s->learned_active && s->net);   // someone reads rpT
        for (int c = 1; c < s->opt.amg_cycles; c++) {
            const bool first = c == 1;
            sim_launch(cycle_next_kernel<T>, sim_blocks(N, 128), 128, s->stream,
                level_matT<T>(s, L0, 0), (const T *)(first ? L0.f : s->rpT), (const T *)(first ? L0.e2 : s->epacc),
                (const T *)L0.dinvT, (T *)L0.f, (T *)L0.e, first && keep ? (T *)s->rpT : nullptr,
                first ? (T *)s->epacc : nullptr, done);
            SIM_LAUNCHED(s);
            if (vcycle<T>(s, done, (T *)s->epacc) != SIM_OK) return s->err;
        }
        ep = (const T *)s->epacc;
    }
    if (s->learned_active && s->net) {
        // extra stage: the network's correction of the pressure residual left by stage P
        const T *rp = (s->opt.amg_cycles > 1 && s->lev.size() > 1) ? (const T *)s->rpT : (const T *)L0.f;
        sim_launch(amg_resid_kernel<T>, sim_blocks(N, 128), 128, s->stream, level_matT<T>(s, L0, 0), rp, ep, (T *)s->lres, done);
        SIM_LAUNCHED(s);
        rms_kernel<T><<<SIM_RED_BLOCKS, SIM_THREADS, 0, s->stream>>>(N, (const T *)s->lres, s->red, s->ticket, s->lrms, done);
        SIM_LAUNCHED(s);
        learned_in_kernel<T><<<sim_blocks(N), SIM_THREADS, 0, s->stream>>>(N, (const T *)s->lres, s->lrms, s->lfeat, s->lx, done);
        SIM_LAUNCHED(s);
        const int64_t l0 = net_launches(s->net);
        if (net_infer(s->net, s->lx, s->ly, s->stream, done) != SIM_OK) return sim_fail(s, SIM_ECUDA, "learned stage inference");
        s->launches += net_launches(s->net) - l0;
        // minimal-residual scaling of the correction: never increases ||r'||_2
        learned_apply_kernel<T><<<sim_blocks(N, 128), 128, 0, s->stream>>>(level_matT<T>(s, L0, 0), s->ly, s->lrms,
                                                                          (T *)s->lep, done);
        SIM_LAUNCHED(s);
        mr_step_kernel<T><<<SIM_RED_BLOCKS, SIM_THREADS, 0, s->stream>>>(N, (const T *)s->lep, (const T *)s->lres, s->red,
                                                                        s->ticket, s->lrms, done);
        SIM_LAUNCHED(s);
        learned_out_kernel<T><<<sim_blocks(N), SIM_THREADS, 0, s->stream>>>(N, ep, s->ly, s->lrms, (T *)s->lep, done);
        SIM_LAUNCHED(s);
        ep = (const T *)s->lep;
    }
    const T *addv = fpf ? (const T *)s->x0 : nullptr;
    sim_launch(stage2_a_kernel<B, T>, sim_blocks(N, s->tune_stage), s->tune_stage, s->stream, s->gd, fpf ? nullptr : r, (const T *)s->qiwT, lscT,
                                                            (const T *)s->rhT, (const T *)s->ahat, dinv, ep, (T *)s->r2,
                                                            (T *)s->zr, rb, done);
    SIM_LAUNCHED(s);
    if (rb) {
        sim_launch(stage2_b_kernel<B, T, TZ>, colour_blocks(s, s->tune_stage), s->tune_stage, s->stream, s->gd, (const T *)s->ahat, dinv, (const T *)s->r2,
                                                                    (T *)s->zr, ep, addv, z, done);
        SIM_LAUNCHED(s);
    }
    sim_launch(stage2_c_kernel<B, T, TZ>, rb ? colour_blocks(s, s->tune_stage) : sim_blocks(N, s->tune_stage), s->tune_stage, s->stream, s->gd, (const T *)s->ahat, dinv, (const T *)s->zr, ep, addv,
                                                                z, rb, done);
    SIM_LAUNCHED(s);
    return SIM_OK;
}

sim_status cpr_apply(sim_t *s, const double *r, void *z, const int *done) {
    if (!s->precond_ready) { if (cpr_setup(s) != SIM_OK) return s->err; }
    if (s->b == 2)
        return sim_mixed(s) ? apply_btz<2, float, float>(s, r, (float *)z, done) : apply_btz<2, double, double>(s, r, (double *)z, done);
    return sim_mixed(s) ? apply_btz<3, float, float>(s, r, (float *)z, done) : apply_btz<3, double, double>(s, r, (double *)z, done);
}

// ===========================================================================
// CPR application batched over the members of an ensemble
//
// One launch per stage covers every member: the restriction, each V-cycle
// level's residual / restriction / prolongation / smoothing (a member takes
// part in the launches of the levels it has), the coarse end (one 16-CTA
// cluster per member for its fused coarse levels, or the dense product of its
// coarsest level) and the three stage-F sweeps.  Block b of a launch takes
// work[b] = (member, block of the member's rows), reads the member's operands
// from a device table and runs the single-system row arithmetic, so every
// member's result equals that of its own application.  A member whose restart
// cycle is done (its FGMRES control word) returns at once.
// ===========================================================================
namespace {
constexpr int kBatchLevels = 16;
constexpr int kBatchAmgThreads = 128;

template <typename T>
struct BLevel {
    Mat<T> A;                   // the level's matrix (apply precision)
    const T *dinv;              // 1 / l1 row sums
    const int *agg, *moff, *mem;
    T *f, *e, *e2;
    int n;
};

template <typename T>
struct CMember {
    GridDesc g;
    long n;                     // b N
    const double *V;            // input of application j: V + j n (FP64)
    T *Z;                       // output: Z + j n
    const T *wT, *lscT, *ahat, *dinv;
    T *r2, *zr;
    int full, rb, nl, lf;
    const double *inv;          // dense inverse of the coarsest level
    const CoarseCycle<T> *cc;   // the fused coarse levels (device copy) or null
    const int *done;
    BLevel<T> lv[kBatchLevels];
};

template <typename T>
__device__ __forceinline__ const CMember<T> &cmember(const CMember<T> *M, const int2 *work, int *vb) {
    const int2 wk = work[blockIdx.x];
    *vb = wk.y;
    return M[wk.x];
}

template <int B, typename T>
__global__ void b_restrict_p_kernel(const CMember<T> *M, const int2 *work, int j) {
    int vb;
    const CMember<T> &m = cmember(M, work, &vb);
    if (skip(m.done)) return;
    const int i = vb * blockDim.x + threadIdx.x;
    if (i >= m.g.N) return;
    const BLevel<T> &L0 = m.lv[0];
    restrict_p_row<B, T>(m.g.N, m.V + (size_t)j * m.n, m.wT, m.full, L0.dinv, L0.f, L0.e, i);
}

// down the V-cycle at level l: e2 = f - A e (mode 0, rows of l) or the
// restriction of e2 to level l + 1 (mode 1, rows of l + 1)
template <typename T>
__global__ void b_amg_down_kernel(const CMember<T> *M, const int2 *work, int l, int mode) {
    int vb;
    const CMember<T> &m = cmember(M, work, &vb);
    if (skip(m.done)) return;
    const int i = vb * blockDim.x + threadIdx.x;
    const BLevel<T> &L = m.lv[l];
    if (mode == 0) {
        amg_resid_row<T>(L.A, L.f, L.e, L.e2, i);
    } else {
        const BLevel<T> &C = m.lv[l + 1];
        if (i < C.n) amg_restrict_row<T>(L.e2, L.moff, L.mem, C.f, l + 1 == m.nl - 1 ? nullptr : C.e, C.dinv, i);
    }
}

// up the V-cycle at level l: e += P e_c (mode 0), then e2 = e + (f - A e) / l1 (mode 1)
template <typename T>
__global__ void b_amg_up_kernel(const CMember<T> *M, const int2 *work, int l, int mode) {
    int vb;
    const CMember<T> &m = cmember(M, work, &vb);
    if (skip(m.done)) return;
    const int i = vb * blockDim.x + threadIdx.x;
    const BLevel<T> &L = m.lv[l];
    if (mode == 0) {
        if (i >= L.n) return;
        const BLevel<T> &C = m.lv[l + 1];
        const T *ec = (l + 1 == m.nl - 1) ? C.e : C.e2;
        L.e[i] += ec[L.agg[i]];
    } else {
        amg_smooth_row<T>(L.A, L.f, L.e, L.dinv, L.e2, i);
    }
}

// coarsest level without the fused cycle: e = Inv f, one warp per row (a
// one-level hierarchy writes e2 of level 0, the stage-P correction)
template <typename T>
__global__ void b_coarse_solve_kernel(const CMember<T> *M, const int2 *work) {
    int vb;
    const CMember<T> &m = cmember(M, work, &vb);
    if (skip(m.done)) return;
    const BLevel<T> &C = m.lv[m.nl - 1];
    const int warp = (vb * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (warp >= C.n) return;
    double s = 0.0;
    for (int q = lane; q < C.n; q += 32) s += m.inv[(long)warp * C.n + q] * (double)C.f[q];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if (lane == 0) (m.nl == 1 ? C.e2 : C.e)[warp] = (T)s;
}

// the fused coarse levels: cluster c runs member members[c]
template <typename T>
__global__ void __launch_bounds__(kCoarseThreads, 1) b_coarse_cycle_kernel(const CMember<T> *M, const int *members) {
    const int nb = (int)cg::this_cluster().num_blocks();
    const CMember<T> &m = M[members[blockIdx.x / nb]];
    if (skip(m.done)) return;          // uniform over the cluster (one member)
    coarse_cycle_body<T>(*m.cc, (int)(blockIdx.x % nb), nb);
}

// whole applications of small members: cluster c runs tab[c]
template <typename T>
struct SmallMember {
    SmallApply<T> S;
    const double *V;            // input of application j: V + j n (FP64)
    T *Z;                       // output: Z + j n
    long n;
    const int *done;
};
template <int B, typename T>
__global__ void __launch_bounds__(kSmallThreads, 1) b_small_apply_kernel(const SmallMember<T> *tab, int j) {
    const int nb = (int)cg::this_cluster().num_blocks();
    const SmallMember<T> &m = tab[blockIdx.x / nb];
    if (skip(m.done)) return;          // uniform over the cluster (one member)
    small_apply_body<B, T, T>(m.S, m.V + (size_t)j * m.n, m.Z + (size_t)j * m.n, (int)(blockIdx.x % nb), nb);
}

// stage F on the residual of stage P: sweep 0 (all cells), 1 (black), 2 (red,
// or all cells for block Jacobi)
template <int B, typename T>
__global__ void b_stage2_kernel(const CMember<T> *M, const int2 *work, int j, int sweep) {
    int vb;
    const CMember<T> &m = cmember(M, work, &vb);
    if (skip(m.done)) return;
    const long t = vb * (long)blockDim.x + threadIdx.x;
    const T *ep = m.lv[0].e2;
    T *out = m.Z + (size_t)j * m.n;
    if (sweep == 0) {
        if (t >= m.g.N) return;
        stage2_a_row<B, T>(m.g, m.V + (size_t)j * m.n, m.wT, m.lscT, nullptr, m.ahat, m.dinv, ep, m.r2, m.zr, m.rb, (int)t);
    } else if (sweep == 1) {
        const int i = colour_cell(m.g, t, 1);
        if (i >= 0) stage2_b_row<B, T, T>(m.g, m.ahat, m.dinv, m.r2, m.zr, ep, nullptr, out, i);
    } else {
        const int i = m.rb ? colour_cell(m.g, t, 0) : (t < m.g.N ? (int)t : -1);
        if (i >= 0) stage2_c_row<B, T, T>(m.g, m.ahat, m.dinv, m.zr, ep, nullptr, out, m.rb, i);
    }
}
}  // namespace

struct CprBatch {
    int nm = 0, b = 0, mixed = 0, rb = 0;
    void *dmem = nullptr;  size_t mem_cap = 0;    // CMember<T>[nm]
    void *dcc = nullptr;   size_t cc_cap = 0;     // CoarseCycle<T>[ncl]
    int2 *dwork = nullptr; size_t work_cap = 0;
    int *dcl = nullptr;    size_t cl_cap = 0;     // members with fused coarse levels
    void *dsmall = nullptr; size_t small_cap = 0; // SmallMember<T>[nsmall]
    int ncl = 0, nsmall = 0;
    struct List { long off = 0; int count = 0; };
    List cell256, cell64, stage1, stage2, cs;
    std::vector<List> down_r, down_c, up, up_s;
};

static cudaError_t grow(void **p, size_t *cap, size_t bytes) {
    if (bytes <= *cap) return cudaSuccess;
    if (*p) cudaFree(*p);
    *p = nullptr; *cap = 0;
    const cudaError_t e = cudaMalloc(p, bytes);
    if (e == cudaSuccess) *cap = bytes;
    return e;
}

// the members' current hierarchies are batchable: the same options, block
// size and precision, two-stage CPR with one V-cycle, no learned stage, no
// rate-controlled wells, at most kBatchLevels levels
bool cpr_batchable(sim_t *const *ms, int nm) {
    if (nm < 1) return false;
    const sim_options &o = ms[0]->opt;
    for (int k = 0; k < nm; k++) {
        const sim_t *s = ms[k];
        const sim_options &p = s->opt;
        if (s->b != ms[0]->b || sim_mixed(s) != sim_mixed(ms[0]) || p.precond != SIM_PRECOND_CPR ||
            p.stage2 != o.stage2 || p.decouple != o.decouple || p.cpr_stages != 2 || p.amg_cycles != 1 ||
            p.krylov != SIM_KRYLOV_FGMRES || p.gmres_m != o.gmres_m || p.orth != o.orth || s->learned_on || s->nrate)
            return false;
    }
    return true;
}

template <typename T>
static cudaError_t batch_build_t(CprBatch *cb, sim_t *const *ms, int nm, cudaStream_t st) {
    std::vector<CMember<T>> hm(nm);
    std::vector<CoarseCycle<T>> hcc;
    std::vector<int> hcl;
    std::vector<int2> work;
    std::vector<SmallMember<T>> hsm;
    // up to eight small members take an application in one launch, a cluster each (as
    // many as are resident at once); more of them fill the GPU as rows of the others do
    int nsmall = 0;
    for (int k = 0; k < nm; k++) nsmall += small_grid(ms[k]) ? 1 : 0;
    std::vector<char> small(nm, 0);
    for (int k = 0; k < nm; k++) small[k] = nsmall <= 8 && small_grid(ms[k]);
    cb->down_r.clear(); cb->down_c.clear(); cb->up.clear(); cb->up_s.clear();
    auto add_list = [&](CprBatch::List &L, auto blocks_of) {
        L.off = (long)work.size();
        for (int k = 0; k < nm; k++) {
            const int nb = small[k] ? 0 : blocks_of(k);
            for (int q = 0; q < nb; q++) work.push_back(make_int2(k, q));
        }
        L.count = (int)((long)work.size() - L.off);
    };
    int maxdown = 0, maxup = 0;
    for (int k = 0; k < nm; k++) {
        sim_t *s = ms[k];
        CMember<T> &m = hm[k];
        memset(&m, 0, sizeof(m));
        const int nl = (int)s->lev.size();
        if (nl < 1 || nl > kBatchLevels || !s->precond_ready) return cudaErrorInvalidValue;
        m.g = s->gd; m.n = (long)s->N * s->b;
        m.V = s->V; m.Z = (T *)s->Z;
        m.wT = (const T *)s->qiwT;
        m.full = s->opt.decouple == SIM_DECOUPLE_ABF;
        m.lscT = m.full ? (const T *)s->lscT : nullptr;
        m.ahat = (const T *)s->ahat;
        m.dinv = sizeof(T) == sizeof(double) ? (const T *)s->dinv_d : (const T *)s->dinv;
        m.r2 = (T *)s->r2; m.zr = (T *)s->zr;
        m.rb = s->opt.stage2 == SIM_STAGE2_ILU0_RB;
        m.nl = nl;
        m.lf = (s->opt.fused_coarse && nl > 1) ? coarse_start(s) : nl;
        m.inv = (const double *)s->lev[nl - 1].coarse_inv;
        m.done = &s->ctl->done;
        for (int l = 0; l < nl; l++) {
            AmgLevel &L = s->lev[l];
            BLevel<T> &d = m.lv[l];
            d.A = level_matT<T>(s, L, l);
            d.dinv = (const T *)L.dinvT; d.agg = L.agg; d.moff = L.moff; d.mem = L.mem;
            d.f = (T *)L.f; d.e = (T *)L.e; d.e2 = (T *)L.e2; d.n = L.n;
        }
        if (small[k]) {
            hsm.push_back(SmallMember<T>{small_apply<T>(s), s->V, (T *)s->Z, m.n, m.done});
            continue;
        }
        if (m.lf < nl) {
            CoarseCycle<T> cc;
            cc.nlev = nl - m.lf; cc.g = s->gd;
            cc.inv = m.inv;
            for (int l = m.lf; l < nl; l++) {
                const AmgLevel &L = s->lev[l];
                CoarseLevel<T> &d = cc.lv[l - m.lf];
                d = coarse_level<T>(L, l);
            }
            hcc.push_back(cc);
            hcl.push_back(k);
        }
        const int down = nl > 1 ? std::min(nl - 1, m.lf) : 0;
        const int top = nl > 1 ? (m.lf < nl ? m.lf : nl - 1) : 0;
        maxdown = std::max(maxdown, down);
        maxup = std::max(maxup, top);
    }
    auto down_of = [&](int k) { const CMember<T> &m = hm[k]; return m.nl > 1 ? std::min(m.nl - 1, m.lf) : 0; };
    auto top_of = [&](int k) { const CMember<T> &m = hm[k]; return m.nl > 1 ? (m.lf < m.nl ? m.lf : m.nl - 1) : 0; };
    add_list(cb->cell256, [&](int k) { return sim_blocks(hm[k].g.N, SIM_THREADS); });
    add_list(cb->cell64, [&](int k) { return sim_blocks(hm[k].g.N, kStageThreads); });
    add_list(cb->stage1, [&](int k) { return hm[k].rb ? colour_blocks(ms[k], kStageThreads) : 0; });
    add_list(cb->stage2, [&](int k) { return hm[k].rb ? colour_blocks(ms[k], kStageThreads) : sim_blocks(hm[k].g.N, kStageThreads); });
    add_list(cb->cs, [&](int k) { const CMember<T> &m = hm[k];
                                  return (m.nl == 1 || m.lf == m.nl) ? sim_blocks((long)m.lv[m.nl - 1].n * 32, SIM_THREADS) : 0; });
    cb->down_r.resize(maxdown); cb->down_c.resize(maxdown); cb->up.resize(maxup); cb->up_s.resize(maxup);
    for (int l = 0; l < maxdown; l++) {
        add_list(cb->down_r[l], [&](int k) { return l < down_of(k) ? level_blocks(hm[k].lv[l].n, l, kBatchAmgThreads) : 0; });
        add_list(cb->down_c[l], [&](int k) { return l < down_of(k) ? sim_blocks(hm[k].lv[l + 1].n, kBatchAmgThreads) : 0; });
    }
    for (int l = 0; l < maxup; l++) {
        add_list(cb->up[l], [&](int k) { return l < top_of(k) ? sim_blocks(hm[k].lv[l].n, kBatchAmgThreads) : 0; });
        add_list(cb->up_s[l], [&](int k) { return l < top_of(k) ? level_blocks(hm[k].lv[l].n, l, kBatchAmgThreads) : 0; });
    }
    cudaError_t e;
    if ((e = grow(&cb->dmem, &cb->mem_cap, sizeof(CMember<T>) * nm)) != cudaSuccess) return e;
    if ((e = grow((void **)&cb->dwork, &cb->work_cap, sizeof(int2) * std::max<size_t>(1, work.size()))) != cudaSuccess) return e;
    if (!hcc.empty()) {
        if ((e = grow(&cb->dcc, &cb->cc_cap, sizeof(CoarseCycle<T>) * hcc.size())) != cudaSuccess) return e;
        if ((e = grow((void **)&cb->dcl, &cb->cl_cap, sizeof(int) * hcl.size())) != cudaSuccess) return e;
        for (size_t c = 0; c < hcc.size(); c++) hm[hcl[c]].cc = (const CoarseCycle<T> *)cb->dcc + c;
        if ((e = cudaMemcpyAsync(cb->dcc, hcc.data(), sizeof(CoarseCycle<T>) * hcc.size(), cudaMemcpyHostToDevice, st)) != cudaSuccess) return e;
        if ((e = cudaMemcpyAsync(cb->dcl, hcl.data(), sizeof(int) * hcl.size(), cudaMemcpyHostToDevice, st)) != cudaSuccess) return e;
    }
    cb->ncl = (int)hcl.size();
    if (!hsm.empty()) {
        if ((e = grow(&cb->dsmall, &cb->small_cap, sizeof(SmallMember<T>) * hsm.size())) != cudaSuccess) return e;
        if ((e = cudaMemcpyAsync(cb->dsmall, hsm.data(), sizeof(SmallMember<T>) * hsm.size(), cudaMemcpyHostToDevice, st)) != cudaSuccess) return e;
    }
    cb->nsmall = (int)hsm.size();
    if ((e = cudaMemcpyAsync(cb->dmem, hm.data(), sizeof(CMember<T>) * nm, cudaMemcpyHostToDevice, st)) != cudaSuccess) return e;
    if (!work.empty() && (e = cudaMemcpyAsync(cb->dwork, work.data(), sizeof(int2) * work.size(), cudaMemcpyHostToDevice, st)) != cudaSuccess) return e;
    // the host tables must outlive the asynchronous copies
    if ((e = cudaStreamSynchronize(st)) != cudaSuccess) return e;
    cb->nm = nm; cb->b = ms[0]->b; cb->mixed = sim_mixed(ms[0]); cb->rb = hm[0].rb;
    return cudaSuccess;
}

CprBatch *cpr_batch_new() { return new CprBatch(); }

void cpr_batch_free(CprBatch *cb) {
    if (!cb) return;
    if (cb->dmem) cudaFree(cb->dmem);
    if (cb->dcc) cudaFree(cb->dcc);
    if (cb->dwork) cudaFree(cb->dwork);
    if (cb->dcl) cudaFree(cb->dcl);
    if (cb->dsmall) cudaFree(cb->dsmall);
    delete cb;
}

cudaError_t cpr_batch_build(CprBatch *cb, sim_t *const *ms, int nm, cudaStream_t st) {
    return sim_mixed(ms[0]) ? batch_build_t<float>(cb, ms, nm, st) : batch_build_t<double>(cb, ms, nm, st);
}

template <int B, typename T>
static int batch_apply_t(const CprBatch *cb, cudaStream_t st, int j) {
    const CMember<T> *M = (const CMember<T> *)cb->dmem;
    const int2 *W = cb->dwork;
    int launches = 0;
    auto go = [&](const CprBatch::List &L, int threads, auto launch) {
        if (L.count > 0) { launch(L.count, threads, W + L.off); launches++; }
    };
    if (cb->nsmall > 0) {
        if (launch_clusters<b_small_apply_kernel<B, T>>(cb->nsmall, kSmallThreads, st, (const SmallMember<T> *)cb->dsmall, j) != cudaSuccess)
            return -1;
        launches++;
    }
    go(cb->cell256, SIM_THREADS, [&](int n, int t, const int2 *w) { sim_launch(b_restrict_p_kernel<B, T>, n, t, st, M, w, j); });
    for (size_t l = 0; l < cb->down_r.size(); l++) {
        go(cb->down_r[l], kBatchAmgThreads, [&](int n, int t, const int2 *w) { sim_launch(b_amg_down_kernel<T>, n, t, st, M, w, (int)l, 0); });
        go(cb->down_c[l], kBatchAmgThreads, [&](int n, int t, const int2 *w) { sim_launch(b_amg_down_kernel<T>, n, t, st, M, w, (int)l, 1); });
    }
    if (cb->ncl > 0) {
        if (launch_clusters<b_coarse_cycle_kernel<T>>(cb->ncl, kCoarseThreads, st, M, (const int *)cb->dcl) != cudaSuccess) return -1;
        launches++;
    }
    go(cb->cs, SIM_THREADS, [&](int n, int t, const int2 *w) { sim_launch(b_coarse_solve_kernel<T>, n, t, st, M, w); });
    for (int l = (int)cb->up.size() - 1; l >= 0; l--) {
        go(cb->up[l], kBatchAmgThreads, [&](int n, int t, const int2 *w) { sim_launch(b_amg_up_kernel<T>, n, t, st, M, w, l, 0); });
        go(cb->up_s[l], kBatchAmgThreads, [&](int n, int t, const int2 *w) { sim_launch(b_amg_up_kernel<T>, n, t, st, M, w, l, 1); });
    }
    go(cb->cell64, kStageThreads, [&](int n, int t, const int2 *w) { sim_launch(b_stage2_kernel<B, T>, n, t, st, M, w, j, 0); });
    go(cb->stage1, kStageThreads, [&](int n, int t, const int2 *w) { sim_launch(b_stage2_kernel<B, T>, n, t, st, M, w, j, 1); });
    go(cb->stage2, kStageThreads, [&](int n, int t, const int2 *w) { sim_launch(b_stage2_kernel<B, T>, n, t, st, M, w, j, 2); });
    return launches;
}

// one batched CPR application (input V_j, output Z_j of every member);
// returns the number of kernels launched, or -1 on a launch error
int cpr_batch_apply(const CprBatch *cb, cudaStream_t st, int j) {
    int n;
    if (cb->b == 2) n = cb->mixed ? batch_apply_t<2, float>(cb, st, j) : batch_apply_t<2, double>(cb, st, j);
    else n = cb->mixed ? batch_apply_t<3, float>(cb, st, j) : batch_apply_t<3, double>(cb, st, j);
    return cudaGetLastError() == cudaSuccess ? n : -1;
}

sim_status cpr_copy_level_ell(sim_t *s, int level, int *col, double *val) {
    if (level < 1 || level >= (int)s->lev.size()) return sim_fail(s, SIM_EINVAL, "level out of range");
    const AmgLevel &L = s->lev[level];
    SIM_CK(s, cudaMemcpyAsync(col, L.col, sizeof(int) * (size_t)L.width * L.n, cudaMemcpyDeviceToHost, s->stream));
    SIM_CK(s, cudaMemcpyAsync(val, L.val, sizeof(double) * (size_t)L.width * L.n, cudaMemcpyDeviceToHost, s->stream));
    SIM_CK(s, cudaStreamSynchronize(s->stream));
    return SIM_OK;
}

// Training pairs for the learned stage.  For Krylov vector v_j: f = (L v_j)_p,
// one stage-P V-cycle e_p, the residual it leaves r' = f - A_p e_p (the input
// of the learned stage in apply_btz), and as target the error that residual
// corresponds to, A_p^-1 r', approximated by kRefine V-cycles of iterative
// refinement.  Input r' / rms(r') with the log-transmissibility features;
// target normalised by its own RMS (the stage is scaled by minimal residual).
constexpr int kRefine = 8;

template <typename T>
static sim_status learned_pairs_t(sim_t *s, int k, float *x, float *y) {
    const int N = s->N;
    AmgLevel &L0 = s->lev[0];
    const int full = s->opt.decouple == SIM_DECOUPLE_ABF;
    const Mat<T> A0 = level_matT<T>(s, L0, 0);
    auto cycle = [&](void) -> sim_status {
        if (s->lev.size() == 1) {
            sim_launch(coarse_solve_kernel<T>, sim_blocks((long)L0.n * 32), SIM_THREADS, s->stream,
                L0.n, (const double *)L0.coarse_inv, (const T *)L0.f, (T *)L0.e2, nullptr);
            SIM_LAUNCHED(s);
            return SIM_OK;
        }
        return vcycle<T>(s, nullptr);
    };
    for (int j = 0; j < k; j++) {
        const double *v = s->V + (size_t)j * N * s->b;
        if (s->b == 2) sim_launch(restrict_p_kernel<2, T>, sim_blocks(N), SIM_THREADS, s->stream, N, v, (const T *)s->qiwT, full, (const T *)L0.dinvT, (T *)L0.f, (T *)L0.e, L2Prefetch{}, nullptr);
        else sim_launch(restrict_p_kernel<3, T>, sim_blocks(N), SIM_THREADS, s->stream, N, v, (const T *)s->qiwT, full, (const T *)L0.dinvT, (T *)L0.f, (T *)L0.e, L2Prefetch{}, nullptr);
        SIM_LAUNCHED(s);
        if (cycle() != SIM_OK) return s->err;
        // r' = f - A_p e_p into rpT; the first refinement cycle starts from it
        sim_launch(amg_resid_kernel<T>, sim_blocks(N, 128), 128, s->stream, A0, (const T *)L0.f, (const T *)L0.e2, (T *)s->rpT,
                                                                     nullptr);
        SIM_LAUNCHED(s);
        sim_launch(copy_add_kernel<T>, sim_blocks(N), SIM_THREADS, s->stream, N, (const T *)s->rpT, (T *)s->lres, 0, nullptr);
        SIM_LAUNCHED(s);
        SIM_CK(s, cudaMemsetAsync(s->epacc, 0, sizeof(T) * (size_t)N, s->stream));
        for (int c = 0; c < kRefine; c++) {
            sim_launch(cycle_next_kernel<T>, sim_blocks(N, 128), 128, s->stream, A0, (const T *)s->rpT, (const T *)s->epacc,
                                                                           (const T *)L0.dinvT, (T *)L0.f, (T *)L0.e, nullptr,
                                                                           nullptr, nullptr);
            SIM_LAUNCHED(s);
            if (cycle() != SIM_OK) return s->err;
            sim_launch(copy_add_kernel<T>, sim_blocks(N), SIM_THREADS, s->stream, N, (const T *)L0.e2, (T *)s->epacc, 1, nullptr);
            SIM_LAUNCHED(s);
        }
        rms_kernel<T><<<SIM_RED_BLOCKS, SIM_THREADS, 0, s->stream>>>(N, (const T *)s->lres, s->red, s->ticket, s->lrms, nullptr);
        SIM_LAUNCHED(s);
        rms_kernel<T><<<SIM_RED_BLOCKS, SIM_THREADS, 0, s->stream>>>(N, (const T *)s->epacc, s->red, s->ticket, s->lrms + 1,
                                                                    nullptr);
        SIM_LAUNCHED(s);
        pair_kernel<T><<<sim_blocks(N), SIM_THREADS, 0, s->stream>>>(N, (const T *)s->lres, (const T *)s->epacc, s->lrms,
                                                                    s->lfeat, x + (size_t)j * N * 4, y + (size_t)j * N);
        SIM_LAUNCHED(s);
    }
    return SIM_OK;
}

sim_status cpr_learned_pairs(sim_t *s, int k, float *x, float *y) {
    if (s->opt.precond != SIM_PRECOND_CPR || !s->precond_ready || s->lev.empty())
        return sim_fail(s, SIM_EINVAL, "training pairs need a CPR preconditioner set up by a solve");
    return sim_mixed(s) ? learned_pairs_t<float>(s, k, x, y) : learned_pairs_t<double>(s, k, x, y);
}

sim_status cpr_learned_features(sim_t *s) {
    const int N = s->N;
    logt_kernel<<<sim_blocks(N), SIM_THREADS, 0, s->stream>>>(s->gd, s->T, s->lfeat);
    SIM_LAUNCHED(s);
    std::vector<float> h((size_t)N * 3);
    SIM_CK(s, cudaMemcpyAsync(h.data(), s->lfeat, sizeof(float) * 3 * (size_t)N, cudaMemcpyDeviceToHost, s->stream));
    SIM_CK(s, cudaStreamSynchronize(s->stream));
    double m[3] = {0, 0, 0}, q[3] = {0, 0, 0};
    for (int i = 0; i < N; i++)
        for (int c = 0; c < 3; c++) { const double v = h[(size_t)i * 3 + c]; m[c] += v; q[c] += v * v; }
    float mf[3], sf[3];
    for (int c = 0; c < 3; c++) {
        const double mu = m[c] / N, var = q[c] / N - mu * mu;
        mf[c] = (float)mu; sf[c] = (float)(var > 1e-12 ? std::sqrt(var) : 0.0);
    }
    standardize_kernel<<<sim_blocks(N), SIM_THREADS, 0, s->stream>>>(N, s->lfeat, mf[0], mf[1], mf[2], sf[0], sf[1], sf[2]);
    SIM_LAUNCHED(s);
    return SIM_OK;
}
