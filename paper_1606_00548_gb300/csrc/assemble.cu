// Residual and Jacobian assembly on the device (FP64), Newton update, norms.
//
// Discretisation (paper Sec. 2.4): backward Euler (Eq. 10), two-point
// cell-centred fluxes with transmissibility K kr rho A / (mu dd) (Eq. 11),
// phase potentials from Eq. (4) with zero capillary pressure, wells by the
// sink/source rate of Eq. (6) under BHP control (Eq. 7) with the Peaceman
// index.  Readings of the open points: depth z positive down with
// Phi = p - rho g z; harmonic face transmissibility; single-point upstream
// weighting per phase (tie -> lower-index cell); arithmetic-mean face density;
// water injectors inject at the cell's total mobility.
//
// Layout: x, R [c][N]; J [d][r][c][N]; per-cell flux properties
// [q][1+b][N] with q = phase densities then (phase, component) mobilities.
// One thread per cell writes only its own rows, so no atomics are needed;
// each face flux is evaluated by both of its cells in the same canonical
// (L, R) orientation, so the two contributions cancel exactly.

#include "sim_internal.cuh"

namespace {

// ---------------------------------------------------------------------------
// per-cell properties, Eq. (3)-(5) ingredients, with their exact derivatives.
// GB300's FP64 pipe takes 2 lanes per clock and SM, so the chain rule is written
// out for the unknowns a quantity depends on (a dual number of every quantity
// multiplies and adds the zeros too), divisions are kept to one reciprocal per
// denominator, and the tables carry their slopes.  524k black-oil cells: 498 -> 210 us.
//
// Unknown order p, s (Sw), x (Sg of a saturated cell, pb of an undersaturated one).
// Only derivatives that can be non-zero are stored, in this order per cell:
//   b = 2: rho_w (v, p) rho_o (v, p) | mob_w (v, p, s) mob_o (v, p, s)
//   b = 3: rho_w (v, p) rho_o (v, p, x) rho_g (v, p) | mob_w (v, p, s)
//          mob_o, mob_og (v, p, s, x) mob_g (v, p, x)
// where mob_q is the (phase, component) pair's mobility times its density:
// b = 2: (w,w) (o,o);  b = 3: (w,w) (o,o) (o,g) (g,g)
// ---------------------------------------------------------------------------
template <int B> struct Layout {
    static constexpr int NPAIR = (B == 2) ? 2 : 4;
    static constexpr int NP = (B == 2) ? 10 : 21;                // stored values per cell
    __host__ __device__ static constexpr int pair_phase(int q) { return B == 2 ? q : (q == 0 ? 0 : (q <= 2 ? 1 : 2)); }
    __host__ __device__ static constexpr int pair_comp(int q) { return B == 2 ? q : (q == 0 ? 0 : (q == 1 ? 1 : 2)); }
    // place of phase a's density and of its derivative by unknown k (-1: zero)
    __host__ __device__ static constexpr int rho(int a) { return B == 2 ? 2 * a : (a == 0 ? 0 : (a == 1 ? 2 : 5)); }
    __host__ __device__ static constexpr int rho_d(int a, int k) {
        return k == 0 ? rho(a) + 1 : (B == 3 && a == 1 && k == 2 ? rho(a) + 2 : -1);
    }
    // the same of pair q's mobility
    __host__ __device__ static constexpr int mob(int q) { return B == 2 ? 4 + 3 * q : (q == 0 ? 7 : (q == 1 ? 10 : (q == 2 ? 14 : 18))); }
    __host__ __device__ static constexpr int mob_d(int q, int k) {
        if (k == 0) return mob(q) + 1;
        if (B == 2 || q == 0) return k == 1 ? mob(q) + 2 : -1;
        if (q == 3) return k == 2 ? mob(q) + 2 : -1;
        return mob(q) + 1 + k;
    }
};

template <int B>
struct Props {
    double acc[B], accd[B][B];     // accumulations and their derivatives
    double q[Layout<B>::NP];       // densities and mobilities as stored
    double lamt, lamtd[B];         // total mobility (water injectors)
};

// Corey curve of a normalised saturation, clipped to [0, 1], and its slope
__device__ __forceinline__ void corey(double s, double n, double &v, double &d) {
    if (s <= 0.0) { v = 0.0; d = 0.0; }
    else if (s >= 1.0) { v = 1.0; d = 0.0; }
    else if (n == 2.0) { v = s * s; d = 2.0 * s; }
    else { v = pow(s, n); d = n * pow(s, n - 1.0); }
}

// interval of the PVT table for abscissa x (piecewise linear, extrapolated)
__device__ __forceinline__ const double *pvt_at(const FluidConst &f, double x) {
    const double *t = f.pvt;
    for (int k = 1; k <= f.npvt - 2 && x >= __ldg(t + SIM_PVT_ROW); k++) t += SIM_PVT_ROW;
    return t;
}
// value at x of column c of interval row t (columns: value, slope); slope in d
__device__ __forceinline__ double pvt_val(const double *t, int c, double x, double &d) {
    d = __ldg(t + 2 + 2 * c);
    return (x - __ldg(t)) * d + __ldg(t + 1 + 2 * c);
}

template <int B>
__device__ __forceinline__ void cell_props(const FluidConst &f, double poro, double vol, double p, double sw, double x3,
                                           int ph, Props<B> &o) {
    const double pv0 = poro * vol;
    const double pv = ((p - f.p_ref) * f.c_rock + 1.0) * poro * vol, pvp = f.c_rock * pv0;
    if constexpr (B == 2) {
        const double rw = exp((p - f.p_ref) * f.c_w) * f.rho_w_ref, rwp = rw * f.c_w;
        const double ro = exp((p - f.p_ref) * f.c_o) * f.rho_o_ref, rop = ro * f.c_o;
        const double ds = f.i_mob;                       // 1 / (1 - swc - sor)
        const double se = (sw - f.swc) * ds, so = 1.0 - sw;
        double kw, kwd, ko, kod;
        corey(se, f.nw, kw, kwd);
        corey(1.0 - se, f.now, ko, kod);
        kw *= f.i_muw; kwd *= ds * f.i_muw; ko *= f.i_muo; kod *= -ds * f.i_muo;
        o.acc[0] = pv * (rw * sw);
        o.accd[0][0] = (pvp * rw + pv * rwp) * sw; o.accd[0][1] = pv * rw;
        o.acc[1] = pv * (ro * so);
        o.accd[1][0] = (pvp * ro + pv * rop) * so; o.accd[1][1] = -(pv * ro);
        o.q[0] = rw; o.q[1] = rwp; o.q[2] = ro; o.q[3] = rop;
        o.q[4] = rw * kw; o.q[5] = rwp * kw; o.q[6] = rw * kwd;
        o.q[7] = ro * ko; o.q[8] = rop * ko; o.q[9] = ro * kod;
        o.lamt = kw + ko; o.lamtd[0] = 0.0; o.lamtd[1] = kwd + kod;
    } else {
        const bool sat = ph != 0;
        const double *tp = pvt_at(f, p);
        double bgd, mgd;
        const double bg = pvt_val(tp, 3, p, bgd), mug = pvt_val(tp, 4, p, mgd);
        // Bo, Rs, mu_o and their derivatives by p and x (x: pb of an undersaturated cell)
        double bo, bop, box, rs, rsp, rsx, mo, mop, mox;
        const double sg = sat ? x3 : 0.0, gx = sat ? 1.0 : 0.0;   // Sg and dSg/dx
        if (sat) {
            bo = pvt_val(tp, 0, p, bop); rs = pvt_val(tp, 1, p, rsp); mo = pvt_val(tp, 2, p, mop);
            box = rsx = mox = 0.0;
        } else {
            const double *tb = pvt_at(f, x3);
            const double du = p - x3, fb = 1.0 - du * f.bo_c_us, fm = du * f.muo_c_us + 1.0;
            double b0d, m0d;
            const double b0 = pvt_val(tb, 0, x3, b0d), m0 = pvt_val(tb, 2, x3, m0d);
            rs = pvt_val(tb, 1, x3, rsx); rsp = 0.0;
            bo = b0 * fb; bop = -(b0 * f.bo_c_us); box = b0d * fb - bop;
            mo = m0 * fm; mop = m0 * f.muo_c_us; mox = m0d * fm - mop;
        }
        const double bw = (p - f.bw_pref) * f.bw_c + 1.0;
        const double ib = 1.0 / bo, ibp = -(bop * ib) * ib, ibx = -(box * ib) * ib;
        const double ig = 1.0 / bg, igp = -(bgd * ig) * ig;
        const double im = 1.0 / mo, ih = 1.0 / mug;
        const double so = (1.0 - sw) - sg;
        double kw, kwd, ko, kod, kg, kgd, kr, krd;                // Corey curves and slopes
        corey((sw - f.swc) * f.i_mob, f.nw, kw, kwd);
        corey(((1.0 - f.sor) - sw) * f.i_mob, f.now, ko, kod);
        corey((sg - f.sgc) * f.i_mobg, f.ng, kg, kgd);
        corey(((1.0 - f.swc - f.sorg) - sg) * f.i_mobog, f.nog, kr, krd);
        kwd *= f.i_mob; kod *= -f.i_mob; kgd *= gx * f.i_mobg; krd *= -(gx * f.i_mobog);
        // Stone II with krow(Swc) = 1
        const double a1 = ko + kw, a2 = kr + kg;
        double kro = a1 * a2 - (kw + kg), kros = (kod + kwd) * a2 - kwd, krox = a1 * (krd + kgd) - kgd;
        if (kro < 0.0) kro = kros = krox = 0.0;
        // accumulations
        const double pw = pv * f.rho_ws, po = pv * f.rho_os, pg = pv * f.rho_gs;
        o.acc[0] = bw * sw * pw;
        o.accd[0][0] = (pvp * bw + pv * f.bw_c) * sw * f.rho_ws; o.accd[0][1] = bw * pw; o.accd[0][2] = 0.0;
        const double m1 = ib * so, m1p = ibp * so, m1x = ibx * so - ib * gx;
        o.acc[1] = m1 * po;
        o.accd[1][0] = (pvp * m1 + pv * m1p) * f.rho_os; o.accd[1][1] = -(ib * po); o.accd[1][2] = m1x * po;
        const double rb = rs * ib, rbp = rsp * ib + rs * ibp, rbx = rsx * ib + rs * ibx;
        const double m2 = rb * so + ig * sg, m2p = rbp * so + igp * sg, m2x = rbx * so + (ig - rb) * gx;
        o.acc[2] = m2 * pg;
        o.accd[2][0] = (pvp * m2 + pv * m2p) * f.rho_gs; o.accd[2][1] = -(rb * pg); o.accd[2][2] = m2x * pg;
        // densities
        const double rw = bw * f.rho_ws, rwp = f.bw_c * f.rho_ws, rg = ig * f.rho_gs, rgp = igp * f.rho_gs;
        const double ro_ = ib * f.rho_os, rop_ = ibp * f.rho_os, rox_ = ibx * f.rho_os;       // oil component in oil
        const double rog = rb * f.rho_gs, rogp = rbp * f.rho_gs, rogx = rbx * f.rho_gs;       // dissolved gas
        o.q[0] = rw; o.q[1] = rwp;
        o.q[2] = ro_ + rog; o.q[3] = rop_ + rogp; o.q[4] = rox_ + rogx;
        o.q[5] = rg; o.q[6] = rgp;
        // mobilities
        const double lw = kw * f.i_muw, lws = kwd * f.i_muw;
        const double lo = kro * im, lop = -(lo * mop) * im, los = kros * im, lox = (krox - lo * mox) * im;
        const double lg = kg * ih, lgp = -(lg * mgd) * ih, lgx = kgd * ih;
        o.q[7] = rw * lw; o.q[8] = rwp * lw; o.q[9] = rw * lws;
        o.q[10] = ro_ * lo; o.q[11] = rop_ * lo + ro_ * lop; o.q[12] = ro_ * los; o.q[13] = rox_ * lo + ro_ * lox;
        o.q[14] = rog * lo; o.q[15] = rogp * lo + rog * lop; o.q[16] = rog * los; o.q[17] = rogx * lo + rog * lox;
        o.q[18] = rg * lg; o.q[19] = rgp * lg + rg * lgp; o.q[20] = rg * lgx;
        o.lamt = (lw + lo) + lg;
        o.lamtd[0] = lop + lgp; o.lamtd[1] = lws + los; o.lamtd[2] = lox + lgx;
    }
}

__device__ __forceinline__ void cell_xyz(const GridDesc &g, int i, int &ix, int &iy, int &iz) {
    ix = i % g.nx;
    int t = i / g.nx;
    iy = t % g.ny;
    iz = t / g.ny;
}
__device__ __forceinline__ int nbr_of(const GridDesc &g, int i, int ix, int iy, int iz, int d) {
    switch (d) {
    case 1: return ix > 0 ? i - 1 : -1;
    case 2: return ix < g.nx - 1 ? i + 1 : -1;
    case 3: return iy > 0 ? i - g.nx : -1;
    case 4: return iy < g.ny - 1 ? i + g.nx : -1;
    case 5: return iz > 0 ? i - g.nx * g.ny : -1;
    case 6: return iz < g.nz - 1 ? i + g.nx * g.ny : -1;
    }
    return i;
}

// ---------------------------------------------------------------------------
// geometry: transmissibilities (Eq. 11, harmonic) and Peaceman well indices
// ---------------------------------------------------------------------------
__global__ void geometry_kernel(GridDesc g, const double *__restrict__ kx, const double *__restrict__ ky,
                                const double *__restrict__ kz, double *__restrict__ T) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= g.N) return;
    int ix, iy, iz;
    cell_xyz(g, i, ix, iy, iz);
    double tx = 0.0, ty = 0.0, tz = 0.0;
    if (ix < g.nx - 1) tx = SIM_DARCY * 2.0 * g.dy * g.dz / (g.dx / kx[i] + g.dx / kx[i + 1]);
    if (iy < g.ny - 1) ty = SIM_DARCY * 2.0 * g.dx * g.dz / (g.dy / ky[i] + g.dy / ky[i + g.nx]);
    if (iz < g.nz - 1) tz = SIM_DARCY * 2.0 * g.dx * g.dy / (g.dz / kz[i] + g.dz / kz[i + g.nx * g.ny]);
    T[i] = tx;
    T[g.N + i] = ty;
    T[2 * g.N + i] = tz;
}

__global__ void peaceman_kernel(GridDesc g, int nperf, const int *__restrict__ cell, const double *__restrict__ kx,
                                const double *__restrict__ ky, const double *__restrict__ rw,
                                const double *__restrict__ skin, double *__restrict__ wi) {
    int q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= nperf) return;
    int c = cell[q];
    double a = kx[c], b = ky[c];
    double ro = 0.28 * sqrt(sqrt(b / a) * g.dx * g.dx + sqrt(a / b) * g.dy * g.dy) / (pow(b / a, 0.25) + pow(a / b, 0.25));
    wi[q] = 2.0 * M_PI * SIM_DARCY * sqrt(a * b) * g.dz / (log(ro / rw[q]) + skin[q]);
}

// ---------------------------------------------------------------------------
// accumulation only (mass at the start of a step, component totals)
// ---------------------------------------------------------------------------
template <int B>
__global__ void accumulation_kernel(FluidConst f, GridDesc g, const double *__restrict__ x, const int8_t *__restrict__ ph,
                                    const double *__restrict__ poro, double *__restrict__ acc) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= g.N) return;
    Props<B> P;
    cell_props<B>(f, poro[i], g.dx * g.dy * g.dz, x[i], x[g.N + i], B == 3 ? x[2 * g.N + i] : 0.0, B == 3 ? ph[i] : 1, P);
#pragma unroll
    for (int c = 0; c < B; c++) acc[c * (long)g.N + i] = P.acc[c];
}

// ---------------------------------------------------------------------------
// assembly pass 1: properties, accumulation rows of R and of the centre block
// ---------------------------------------------------------------------------
template <int B>
__global__ void __launch_bounds__(SIM_THREADS) props_kernel(FluidConst f, GridDesc g, const double *__restrict__ x,
                                                            const int8_t *__restrict__ ph, const double *__restrict__ poro,
                                                            const double *__restrict__ mold, double inv_dt,
                                                            double *__restrict__ props, double *__restrict__ R,
                                                            double *__restrict__ J) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= g.N) return;
    const long N = g.N;
    Props<B> P;
    cell_props<B>(f, poro[i], g.dx * g.dy * g.dz, x[i], x[N + i], B == 3 ? x[2 * N + i] : 0.0, B == 3 ? ph[i] : 1, P);
#pragma unroll
    for (int t = 0; t < Layout<B>::NP; t++) props[t * N + i] = P.q[t];
#pragma unroll
    for (int c = 0; c < B; c++) {
        R[c * N + i] = (P.acc[c] - mold[c * N + i]) * inv_dt;
#pragma unroll
        for (int k = 0; k < B; k++) J[(c * B + k) * N + i] = P.accd[c][k] * inv_dt;
    }
}

// ---------------------------------------------------------------------------
// assembly pass 2: upwinded Darcy fluxes through the six faces of each cell.
//
// Each face is evaluated by both of its cells, as the flow into this cell i from
// its neighbour j: F = T m_up dphi, dphi = (p_j - p_i) - rho_bar G, G = g (z_j - z_i).
// Seen from the other side every operand but dphi and F, which change sign, is the
// same, so the two contributions cancel exactly.  A tie (dphi = 0) takes the cell of
// lower index.
//
// Bound by the FP64 pipe: 33 operations for a face across which gravity does not
// act (G = 0: one potential difference for all phases, no density derivatives) and
// 55 for a vertical one, about 250 a cell; a form that carries the zero
// derivatives, both upstream candidates and gravity on every face takes 840.
// Which cell's derivatives the upstream mobility adds to is chosen by selecting
// the accumulator (integer moves), not by multiplying with zeros.
// 524k cells, black oil: 1105 -> 260 us (the operations at the pipe's rate: 216 us).
// ---------------------------------------------------------------------------
template <int B, bool GRAV>
__device__ __forceinline__ void face_flux(const double (&own)[Layout<B>::NP], const double (&nb)[Layout<B>::NP], double Tf,
                                          double dp, double G, bool lower, double (&Ri)[B], double (&Jc)[B * B],
                                          double (&Jd)[B * B]) {
    using L = Layout<B>;
    const double hG = 0.5 * G;
#pragma unroll
    for (int a = 0; a < B; a++) {
        const double dphi = GRAV ? dp - (own[L::rho(a)] + nb[L::rho(a)]) * hG : dp;
        const bool use_nb = lower ? dphi > 0.0 : dphi >= 0.0;     // lower: this cell has the lower index
        const double t = Tf * dphi;
#pragma unroll
        for (int q = 0; q < L::NPAIR; q++) {
            if (L::pair_phase(q) != a) continue;
            const int c = L::pair_comp(q);
            const double gm = Tf * (use_nb ? nb[L::mob(q)] : own[L::mob(q)]);
            Ri[c] -= gm * dphi;
            Jc[c * B] += gm;
            Jd[c * B] -= gm;
            if (GRAV) {
                const double gh = gm * hG;
#pragma unroll
                for (int k = 0; k < B; k++) {
                    const int r = L::rho_d(a, k);
                    if (r < 0) continue;
                    Jc[c * B + k] += gh * own[r];
                    Jd[c * B + k] += gh * nb[r];
                }
            }
#pragma unroll
            for (int k = 0; k < B; k++) {
                const int m = L::mob_d(q, k);
                if (m < 0) continue;
                const double v = (use_nb ? Jd[c * B + k] : Jc[c * B + k]) - t * (use_nb ? nb[m] : own[m]);
                Jc[c * B + k] = use_nb ? Jc[c * B + k] : v;
                Jd[c * B + k] = use_nb ? v : Jd[c * B + k];
            }
        }
    }
}

template <int B>
__global__ void __launch_bounds__(128, 3) flux_kernel(GridDesc g, const double *__restrict__ x,
                                                      const double *__restrict__ props, const double *__restrict__ T,
                                                      double *__restrict__ R, double *__restrict__ J) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= g.N) return;
    const long N = g.N;
    constexpr int NP = Layout<B>::NP;
    int ix, iy, iz;
    cell_xyz(g, i, ix, iy, iz);
    double Ri[B], Jc[B * B];
#pragma unroll
    for (int c = 0; c < B; c++) Ri[c] = R[c * N + i];
#pragma unroll
    for (int t = 0; t < B * B; t++) Jc[t] = J[t * N + i];
    double own[NP];
#pragma unroll
    for (int t = 0; t < NP; t++) own[t] = props[t * N + i];
    const double p_i = x[i];
    const double depth_i = g.top + (iz + 0.5) * g.dz;
#pragma unroll 1
    for (int oi = 0; oi < 6; oi++) {
        const int d = oi == 0 ? 5 : oi == 1 ? 3 : oi == 2 ? 1 : oi == 3 ? 2 : oi == 4 ? 4 : 6;
        const int j = nbr_of(g, i, ix, iy, iz, d);
        double Jd[B * B];
#pragma unroll
        for (int t = 0; t < B * B; t++) Jd[t] = 0.0;
        if (j >= 0) {
            const bool lower = (d & 1) == 0;          // + direction: this cell has the lower index
            const double Tf = T[(long)((d - 1) >> 1) * N + (lower ? i : j)];
            double nb[NP];
#pragma unroll
            for (int t = 0; t < NP; t++) nb[t] = props[t * N + j];
            const double dp = x[j] - p_i;
            if (d >= 5) {
                const double depth_j = g.top + ((lower ? iz + 1 : iz - 1) + 0.5) * g.dz;
                face_flux<B, true>(own, nb, Tf, dp, SIM_GRAV * (depth_j - depth_i) / 1e5, lower, Ri, Jc, Jd);
            } else {
                face_flux<B, false>(own, nb, Tf, dp, 0.0, lower, Ri, Jc, Jd);
            }
        }
#pragma unroll
        for (int t = 0; t < B * B; t++) J[(long)(d * B * B + t) * N + i] = Jd[t];
    }
#pragma unroll
    for (int c = 0; c < B; c++) R[c * N + i] = Ri[c];
#pragma unroll
    for (int t = 0; t < B * B; t++) J[t * N + i] = Jc[t];
}

// ---------------------------------------------------------------------------
// assembly pass 3: well terms (Eq. 6) at the perforated cells, one thread per
// perforation (distinct cells, checked at creation) over as many SMs as there are
// warps of them: one block for all of them is bound by its SM's FP64 pipe (160
// perforations 84 us, 2,500 perforations 435 us; now 22 us and 6 us for the sums).
// ---------------------------------------------------------------------------
// Border blocks of Eq. (16) per perforation q: apw[c][q] = dR_c/dp_h and,
// for the well's controlled component cc, awp[k][q] = dq_cc/dx_k; the
// perforation's component rates and its controlled rate go to qperf[0..3][q].
template <int B>
__global__ void __launch_bounds__(32) perf_kernel(FluidConst f, GridDesc g, const double *__restrict__ x,
                                                  const int8_t *__restrict__ ph, const double *__restrict__ poro, int nperf,
                                                  const int *__restrict__ cell, const int *__restrict__ type,
                                                  const double *__restrict__ wi, const double *__restrict__ zh,
                                                  const int *__restrict__ pwell, const int *__restrict__ wctrl,
                                                  const double *__restrict__ wp, double *__restrict__ R,
                                                  double *__restrict__ J, double *__restrict__ apw,
                                                  double *__restrict__ awp, double *__restrict__ qperf) {
    using L = Layout<B>;
    const int q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= nperf) return;
    const long N = g.N;
    const int i = cell[q];
    const int iz = i / (g.nx * g.ny);
    const int w = pwell[q];
    const int ctrl = wctrl[w];
    const int cc = ctrl == 1 ? 0 : (ctrl == 2 ? 1 : -1);    // controlled component (water 0, oil 1)
    Props<B> P;
    const double p = x[i];
    cell_props<B>(f, poro[i], g.dx * g.dy * g.dz, p, x[N + i], B == 3 ? x[2 * N + i] : 0.0, B == 3 ? ph[i] : 1, P);
    const double dh = SIM_GRAV * (zh[q] - (g.top + (iz + 0.5) * g.dz)) / 1e5;
    const double W = wi[q];
    const double bhp = wp[w];
    double a_pw[3] = {0.0, 0.0, 0.0}, a_wp[3] = {0.0, 0.0, 0.0}, qc4[4] = {0.0, 0.0, 0.0, 0.0};
    const double Dw = bhp - p - P.q[0] * dh;         // head of a water-filled injector
    const bool inj = type[q] == SIM_WELL_WATER_INJECTOR;
    if (inj && (Dw >= 0.0 || ctrl)) {
        // water at the cell's total mobility; a rate-controlled injector keeps
        // this form for a negative head too (its solution injects, and the
        // form keeps dR_w/dp_h from vanishing on the Newton path)
        const double rw = P.q[0], rwp = P.q[1], lam = rw * P.lamt;
        const double qw = W * lam * Dw;
        R[i] -= qw;
        qc4[0] = qw;
        a_pw[0] -= W * lam;
#pragma unroll
        for (int k = 0; k < B; k++) {
            const double lamd = rw * P.lamtd[k] + (k == 0 ? rwp * P.lamt : 0.0);
            const double dD = k == 0 ? -1.0 - rwp * dh : 0.0;
            const double dq = W * (lamd * Dw + lam * dD);
            J[k * N + i] -= dq;
            if (cc == 0) a_wp[k] += dq;
        }
        if (cc == 0) qc4[3] = qw;
    } else {
        // producer (Eq. 6 per phase), or a BHP-controlled injector in
        // backflow: the cell's phases leave at their own mobilities, driven
        // for the injector by its water head (continuous at Dw = 0)
#pragma unroll
        for (int a = 0; a < B; a++) {
            const double Dp = inj ? Dw : bhp - p - P.q[L::rho(a)] * dh;
#pragma unroll
            for (int pq = 0; pq < L::NPAIR; pq++) {
                if (L::pair_phase(pq) != a) continue;
                const int c = L::pair_comp(pq);
                const double m = P.q[L::mob(pq)];
                const double qc = W * m * Dp;
                R[c * N + i] -= qc;
                qc4[c] += qc;
                a_pw[c] -= W * m;
#pragma unroll
                for (int k = 0; k < B; k++) {
                    const int r0 = L::rho_d(0, k), ra = L::rho_d(a, k), mk = L::mob_d(pq, k);
                    const double rd = inj ? (r0 >= 0 ? P.q[r0] : 0.0) : (ra >= 0 ? P.q[ra] : 0.0);
                    const double dD = (k == 0 ? -1.0 : 0.0) - rd * dh;
                    const double dq = W * ((mk >= 0 ? P.q[mk] : 0.0) * Dp + m * dD);
                    J[(long)(c * B + k) * N + i] -= dq;
                    if (c == cc) a_wp[k] += dq;
                }
                if (c == cc) qc4[3] = qc;
            }
        }
    }
#pragma unroll
    for (int c = 0; c < 3; c++) {
        apw[(long)c * nperf + q] = a_pw[c];
        awp[(long)c * nperf + q] = a_wp[c];
    }
#pragma unroll
    for (int c = 0; c < 4; c++) qperf[(long)c * nperf + q] = qc4[c];
}

// Well equations: one warp per well sums its perforations (lanes stride over them,
// then a fixed shuffle tree) into R_w, A_ww and the well's rates; one block, whose
// first warp then sums the rates over the wells and takes the largest relative
// residual of the rate controls (a rate that is no number is in its cell's residual too,
// where the CNV maximum finds it).
constexpr int kWellThreads = 512;
__global__ void __launch_bounds__(kWellThreads) well_sum_kernel(int nperf, const int *__restrict__ woff, int nwells,
                                                                const int *__restrict__ wctrl,
                                                                const double *__restrict__ wrate,
                                                                const double *__restrict__ wbhp_c,
                                                                const double *__restrict__ wp,
                                                                const double *__restrict__ apw,
                                                                const double *__restrict__ qperf, double *__restrict__ rw,
                                                                double *__restrict__ aww, double *qwell,
                                                                double *__restrict__ wcnv, double *__restrict__ qtot) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    for (int w = wid; w < nwells; w += kWellThreads / 32) {
        const int ctrl = wctrl[w], cc = ctrl == 1 ? 0 : 1;
        double v[5] = {0.0, 0.0, 0.0, 0.0, 0.0};     // component rates, controlled rate, dR_w/dp_h
        for (int q = woff[w] + lane; q < woff[w + 1]; q += 32) {
#pragma unroll
            for (int c = 0; c < 4; c++) v[c] += qperf[(long)c * nperf + q];
            if (ctrl) v[4] -= apw[(long)cc * nperf + q];
        }
#pragma unroll
        for (int c = 0; c < 5; c++)
            for (int o = 16; o > 0; o >>= 1) v[c] += __shfl_down_sync(0xffffffffu, v[c], o);
        if (lane == 0) {
            rw[w] = ctrl ? v[3] - wrate[w] : wp[w] - wbhp_c[w];
            aww[w] = ctrl ? v[4] : 1.0;
            for (int c = 0; c < 3; c++) qwell[(long)c * nwells + w] = v[c];
        }
    }
    __syncthreads();
    if (wid != 0) return;
    double t[3] = {0.0, 0.0, 0.0}, m = 0.0;
    for (int w = lane; w < nwells; w += 32) {
#pragma unroll
        for (int c = 0; c < 3; c++) t[c] += qwell[(long)c * nwells + w];
        if (wctrl[w]) {
            const double sc = fabs(wrate[w]) > 1.0 ? fabs(wrate[w]) : 1.0;
            const double v = fabs(rw[w]) / sc;
            if (!(v <= m)) m = v;
        }
    }
    for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
        for (int c = 0; c < 3; c++) t[c] += __shfl_down_sync(0xffffffffu, t[c], o);
        const double u = __shfl_down_sync(0xffffffffu, m, o);
        if (!(u <= m)) m = u;
    }
    if (lane == 0) {
        for (int c = 0; c < 3; c++) qtot[c] = t[c];
        *wcnv = m;
    }
}

// b += A_pw A_ww^-1 R_w at the perforations of rate-controlled wells
// (the right-hand side of the system with the well unknowns eliminated)
__global__ void well_rhs_kernel(long N, int b, int nperf, const int *__restrict__ cell, const int *__restrict__ pwell,
                                const int *__restrict__ wctrl, const double *__restrict__ apw,
                                const double *__restrict__ rw, const double *__restrict__ aww, double *__restrict__ rhs) {
    const int q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= nperf) return;
    const int w = pwell[q];
    if (!wctrl[w]) return;
    const double u = rw[w] / aww[w];
    const int i = cell[q];
    for (int c = 0; c < b; c++) rhs[c * N + i] += apw[(long)c * nperf + q] * u;
}

// dp_h = (-R_w - A_wp dx) / A_ww, limited to chop_dp; one warp per well
__global__ void well_update_kernel(long N, int b, int nperf, int nwells, const int *__restrict__ cell,
                                   const int *__restrict__ woff, const int *__restrict__ wctrl,
                                   const double *__restrict__ awp, const double *__restrict__ rw,
                                   const double *__restrict__ aww, const double *__restrict__ dx, double chop_dp,
                                   double *__restrict__ wp) {
    const int w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (w >= nwells || !wctrl[w]) return;
    double t = 0.0;
    for (int q = woff[w] + lane; q < woff[w + 1]; q += 32) {
        const int i = cell[q];
        for (int k = 0; k < b; k++) t += awp[(long)k * nperf + q] * dx[k * N + i];
    }
    for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
    if (lane == 0) {
        double d = (-rw[w] - t) / aww[w];
        if (fabs(d) > chop_dp) d = d > 0 ? chop_dp : -chop_dp;
        wp[w] += d;
    }
}

// y -= A_pw A_ww^-1 A_wp x at the rate-controlled wells' perforations; one warp per well
template <typename X>
__global__ void well_op_kernel(long N, int b, int nperf, int nwells, const int *__restrict__ cell,
                               const int *__restrict__ woff, const int *__restrict__ wctrl,
                               const double *__restrict__ apw, const double *__restrict__ awp,
                               const double *__restrict__ aww, const X *__restrict__ x, double *__restrict__ y,
                               const int *done) {
    if (done && *(volatile const int *)done) return;
    const int w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (w >= nwells || !wctrl[w]) return;
    double t = 0.0;
    for (int q = woff[w] + lane; q < woff[w + 1]; q += 32) {
        const int i = cell[q];
        for (int k = 0; k < b; k++) t += awp[(long)k * nperf + q] * (double)x[k * N + i];
    }
    for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
    const double u = __shfl_sync(0xffffffffu, t, 0) / aww[w];
    for (int q = woff[w] + lane; q < woff[w + 1]; q += 32) {
        const int i = cell[q];
        for (int c = 0; c < b; c++) y[c * N + i] -= apw[(long)c * nperf + q] * u;
    }
}

// ---------------------------------------------------------------------------
// reductions: CNV max, component mass, non-finite count (deterministic:
// fixed grid, per-block partials reduced in block order by the last block)
// ---------------------------------------------------------------------------
__device__ __forceinline__ double nanmax(double a, double b) { return (b > a || b != b) ? b : a; }

template <int OP>   // 0 sum, 1 max (NaN-propagating)
__device__ __forceinline__ double block_reduce(double v) {
    __shared__ double sh[32];
    for (int o = 16; o > 0; o >>= 1) {
        double t = __shfl_down_sync(0xffffffffu, v, o);
        v = OP == 0 ? v + t : nanmax(v, t);
    }
    int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    __syncthreads();
    if (lane == 0) sh[wid] = v;
    __syncthreads();
    if (wid == 0) {
        v = (lane < (int)(blockDim.x >> 5)) ? sh[lane] : (OP == 0 ? 0.0 : 0.0);
        for (int o = 16; o > 0; o >>= 1) {
            double t = __shfl_down_sync(0xffffffffu, v, o);
            v = OP == 0 ? v + t : nanmax(v, t);
        }
    }
    return v;   // valid in thread 0
}

// last block of the grid folds the per-block partials [nv][gridDim] into out[nv]
template <int OP>
__device__ void finish_grid(double *partials, int nv, unsigned int *ticket, double *out) {
    __shared__ bool last;
    __threadfence();
    if (threadIdx.x == 0) {
        unsigned int t = atomicAdd(ticket, 1u);
        last = (t == gridDim.x - 1);
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    // one warp per value, lanes stride over the partials, fixed shuffle tree
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    for (int v = wid; v < nv; v += nw) {
        double acc = 0.0;
        for (int k = lane; k < (int)gridDim.x; k += 32) {
            const double p = __ldcg(partials + (long)v * gridDim.x + k);
            acc = OP == 0 ? acc + p : nanmax(acc, p);
        }
        for (int o = 16; o > 0; o >>= 1) {
            const double t = __shfl_down_sync(0xffffffffu, acc, o);
            acc = OP == 0 ? acc + t : nanmax(acc, t);
        }
        if (lane == 0) out[v] = acc;
    }
    if (threadIdx.x == 0) *ticket = 0u;
}

// the larger of two non-negative values or NaNs by their bits (a NaN's exceed every
// number's, so it propagates), without the FP64 pipe
__device__ __forceinline__ long long absbits(double v) { return __double_as_longlong(v) & 0x7fffffffffffffffLL; }

// largest |R_c| dt / (pv rho_c) of the cells of this thread: one division a cell
// (524k black-oil cells: 47 -> 30 us)
template <int B>
__device__ __forceinline__ double cnv_max(const GridDesc &g, const double *__restrict__ R, const double *__restrict__ poro,
                                          double dt, double r0, double r1, double r2) {
    const long N = g.N;
    const double vol = g.dx * g.dy * g.dz;
    const double k[3] = {dt / (vol * r0), dt / (vol * r1), dt / (vol * r2)};
    long long m = 0;
    for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < N; i += (long)gridDim.x * blockDim.x) {
        long long c0 = 0;
#pragma unroll
        for (int c = 0; c < B; c++) c0 = max(c0, absbits(R[c * N + i] * k[c]));
        m = max(m, absbits(__longlong_as_double(c0) / poro[i]));
    }
    return __longlong_as_double(m);
}

template <int B>
__global__ void cnv_kernel(GridDesc g, const double *__restrict__ R, const double *__restrict__ poro, double dt, double r0,
                           double r1, double r2, double *partials, unsigned int *ticket, double *out) {
    const double m = block_reduce<1>(cnv_max<B>(g, R, poro, dt, r0, r1, r2));
    if (threadIdx.x == 0) partials[blockIdx.x] = m;
    finish_grid<1>(partials, 1, ticket, out);
}

template <int B>
__global__ void mass_kernel(FluidConst f, GridDesc g, const double *__restrict__ x, const int8_t *__restrict__ ph,
                            const double *__restrict__ poro, double *partials, unsigned int *ticket, double *out) {
    const long N = g.N;
    double m[B];
#pragma unroll
    for (int c = 0; c < B; c++) m[c] = 0.0;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < N; i += gridDim.x * blockDim.x) {
        Props<B> P;
        cell_props<B>(f, poro[i], g.dx * g.dy * g.dz, x[i], x[N + i], B == 3 ? x[2 * N + i] : 0.0, B == 3 ? ph[i] : 1, P);
#pragma unroll
        for (int c = 0; c < B; c++) m[c] += P.acc[c];
    }
#pragma unroll
    for (int c = 0; c < B; c++) {
        double t = block_reduce<0>(m[c]);
        if (threadIdx.x == 0) partials[c * gridDim.x + blockIdx.x] = t;
    }
    finish_grid<0>(partials, B, ticket, out);
}

__global__ void nonfinite_kernel(const double *__restrict__ v, long n, double *partials, unsigned int *ticket, double *out) {
    double c = 0.0;
    for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x)
        if (!isfinite(v[i])) c += 1.0;
    c = block_reduce<0>(c);
    if (threadIdx.x == 0) partials[blockIdx.x] = c;
    finish_grid<0>(partials, 1, ticket, out);
}

// ---------------------------------------------------------------------------
// Newton update: Appleyard chop, saturation clamp, black-oil variable switch
// ---------------------------------------------------------------------------
template <int B>
__global__ void update_kernel(int N, double chop_ds, double chop_dp, const double *__restrict__ dx, double *__restrict__ x,
                              int8_t *__restrict__ ph) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N) return;
    double d[B], xi[B];
#pragma unroll
    for (int c = 0; c < B; c++) { d[c] = dx[c * N + i]; xi[c] = x[c * N + i]; }
    int sat = B == 3 ? ph[i] : 1;
    double ds = fabs(d[1]), dp = fabs(d[0]);
    if (B == 3) {
        if (sat) { if (fabs(d[2]) > ds) ds = fabs(d[2]); }
        else { if (fabs(d[2]) > dp) dp = fabs(d[2]); }
    }
    double fct = 1.0;
    if (ds > chop_ds) fct = chop_ds / ds;
    if (dp > chop_dp && chop_dp / dp < fct) fct = chop_dp / dp;
#pragma unroll
    for (int c = 0; c < B; c++) xi[c] += fct * d[c];
    if (xi[1] < 0.0) xi[1] = 0.0;
    if (xi[1] > 1.0) xi[1] = 1.0;
    if (B == 3) {
        if (sat && xi[2] < 0.0) { sat = 0; xi[2] = xi[0]; }
        else if (!sat && xi[2] > xi[0]) { sat = 1; xi[2] = 0.0; }
        if (!sat && xi[1] > 1.0 - 1e-6) { sat = 1; xi[2] = 0.0; }
        if (sat && xi[2] > 1.0 - xi[1]) xi[2] = 1.0 - xi[1];
        ph[i] = (int8_t)sat;
    }
#pragma unroll
    for (int c = 0; c < B; c++) x[c * N + i] = xi[c];
}

}  // namespace

// ===========================================================================
// host launchers
// ===========================================================================
static double *poro_of(sim_t *s) { return s->poro; }

// grid of the state's reductions: up to three blocks per SM
static int state_blocks(long n) { const int b = sim_blocks(n); return b < SIM_RED_BLOCKS ? b : SIM_RED_BLOCKS; }

sim_status k_geometry(sim_t *s, const double *kx, const double *ky, const double *kz, const double *poro,
                      const int *wcell, const int *wtype, const int *pwell, const double *wzh, const double *wrw,
                      const double *wskin) {
    const int N = s->N;
    double *dk = (double *)sim_alloc(s, sizeof(double) * 3 * (size_t)N);
    if (!dk) return s->err;
    SIM_CK(s, cudaMemcpyAsync(dk, kx, sizeof(double) * N, cudaMemcpyHostToDevice, s->stream));
    SIM_CK(s, cudaMemcpyAsync(dk + N, ky, sizeof(double) * N, cudaMemcpyHostToDevice, s->stream));
    SIM_CK(s, cudaMemcpyAsync(dk + 2 * (size_t)N, kz, sizeof(double) * N, cudaMemcpyHostToDevice, s->stream));
    SIM_CK(s, cudaMemcpyAsync(s->poro, poro, sizeof(double) * N, cudaMemcpyHostToDevice, s->stream));
    geometry_kernel<<<sim_blocks(N), SIM_THREADS, 0, s->stream>>>(s->gd, dk, dk + N, dk + 2 * (size_t)N, s->T);
    SIM_LAUNCHED(s);
    const int np = s->nperf;
    if (np > 0) {
        double *tmp = (double *)sim_alloc(s, sizeof(double) * 2 * (size_t)np);
        if (!tmp) return s->err;
        SIM_CK(s, cudaMemcpyAsync(s->perf_cell, wcell, sizeof(int) * np, cudaMemcpyHostToDevice, s->stream));
        SIM_CK(s, cudaMemcpyAsync(s->perf_type, wtype, sizeof(int) * np, cudaMemcpyHostToDevice, s->stream));
        SIM_CK(s, cudaMemcpyAsync(s->perf_well, pwell, sizeof(int) * np, cudaMemcpyHostToDevice, s->stream));
        SIM_CK(s, cudaMemcpyAsync(s->perf_zh, wzh, sizeof(double) * np, cudaMemcpyHostToDevice, s->stream));
        SIM_CK(s, cudaMemcpyAsync(tmp, wrw, sizeof(double) * np, cudaMemcpyHostToDevice, s->stream));
        SIM_CK(s, cudaMemcpyAsync(tmp + np, wskin, sizeof(double) * np, cudaMemcpyHostToDevice, s->stream));
        peaceman_kernel<<<sim_blocks(np), SIM_THREADS, 0, s->stream>>>(s->gd, np, s->perf_cell, dk, dk + N, tmp, tmp + np,
                                                                       s->perf_wi);
        SIM_LAUNCHED(s);
        SIM_CK(s, cudaStreamSynchronize(s->stream));
        sim_free(s, tmp);
    }
    SIM_CK(s, cudaStreamSynchronize(s->stream));
    sim_free(s, dk);
    return SIM_OK;
}

sim_status k_accumulation(sim_t *s, const double *x, const int8_t *ph, double *acc) {
    if (s->b == 2)
        accumulation_kernel<2><<<sim_blocks(s->N), SIM_THREADS, 0, s->stream>>>(s->fc, s->gd, x, ph, poro_of(s), acc);
    else
        accumulation_kernel<3><<<sim_blocks(s->N), SIM_THREADS, 0, s->stream>>>(s->fc, s->gd, x, ph, poro_of(s), acc);
    SIM_LAUNCHED(s);
    return SIM_OK;
}

template <int B>
static sim_status assemble_b(sim_t *s, double dt) {
    const int N = s->N;
    props_kernel<B><<<sim_blocks(N), SIM_THREADS, 0, s->stream>>>(s->fc, s->gd, s->x, s->ph, poro_of(s), s->mold,
                                                                  1.0 / dt, s->props, s->R, s->J);
    SIM_LAUNCHED(s);
    flux_kernel<B><<<sim_blocks(N, 128), 128, 0, s->stream>>>(s->gd, s->x, s->props, s->T, s->R, s->J);
    SIM_LAUNCHED(s);
    if (s->nwells > 0) {
        perf_kernel<B><<<sim_blocks(s->nperf, 32), 32, 0, s->stream>>>(s->fc, s->gd, s->x, s->ph, poro_of(s), s->nperf,
                                                                     s->perf_cell, s->perf_type, s->perf_wi, s->perf_zh,
                                                                     s->perf_well, s->wctrl, s->wp, s->R, s->J, s->apw,
                                                                     s->awp, s->qperf);
        SIM_LAUNCHED(s);
        well_sum_kernel<<<1, kWellThreads, 0, s->stream>>>(s->nperf, s->woff, s->nwells, s->wctrl, s->wrate, s->wbhp_c,
                                                           s->wp, s->apw, s->qperf, s->rw, s->aww, s->qwell, s->wcnv,
                                                           s->qtot);
        SIM_LAUNCHED(s);
    } else {
        SIM_CK(s, cudaMemsetAsync(s->qtot, 0, sizeof(double) * 3, s->stream));
        SIM_CK(s, cudaMemsetAsync(s->wcnv, 0, sizeof(double), s->stream));
    }
    return SIM_OK;
}

sim_status k_assemble(sim_t *s, double dt) {
    s->precond_ready = false;
    return s->b == 2 ? assemble_b<2>(s, dt) : assemble_b<3>(s, dt);
}

sim_status k_well_rhs(sim_t *s, double *rhs) {
    if (s->nrate == 0) return SIM_OK;
    well_rhs_kernel<<<sim_blocks(s->nperf), SIM_THREADS, 0, s->stream>>>(s->N, s->b, s->nperf, s->perf_cell, s->perf_well,
                                                                         s->wctrl, s->apw, s->rw, s->aww, rhs);
    SIM_LAUNCHED(s);
    return SIM_OK;
}

sim_status k_well_update(sim_t *s, const double *dx) {
    if (s->nrate == 0) return SIM_OK;
    well_update_kernel<<<sim_blocks((long)s->nwells * 32), SIM_THREADS, 0, s->stream>>>(
        s->N, s->b, s->nperf, s->nwells, s->perf_cell, s->woff, s->wctrl, s->awp, s->rw, s->aww, dx, s->opt.chop_dp, s->wp);
    SIM_LAUNCHED(s);
    return SIM_OK;
}

template <typename X>
sim_status k_well_op(sim_t *s, const X *x, double *y, const int *done) {
    if (s->nrate == 0) return SIM_OK;
    well_op_kernel<X><<<sim_blocks((long)s->nwells * 32), SIM_THREADS, 0, s->stream>>>(
        s->N, s->b, s->nperf, s->nwells, s->perf_cell, s->woff, s->wctrl, s->apw, s->awp, s->aww, x, y, done);
    SIM_LAUNCHED(s);
    return SIM_OK;
}
template sim_status k_well_op<double>(sim_t *, const double *, double *, const int *);
template sim_status k_well_op<float>(sim_t *, const float *, double *, const int *);

sim_status k_cnv(sim_t *s, double dt, double *cnv_host, double *well_cnv_host) {
    const double *rho = s->fc.cnv_rho;
    if (s->b == 2)
        cnv_kernel<2><<<state_blocks(s->N), SIM_THREADS, 0, s->stream>>>(s->gd, s->R, poro_of(s), dt, rho[0], rho[1], rho[2],
                                                                         s->red, s->ticket, s->scal);
    else
        cnv_kernel<3><<<state_blocks(s->N), SIM_THREADS, 0, s->stream>>>(s->gd, s->R, poro_of(s), dt, rho[0], rho[1], rho[2],
                                                                         s->red, s->ticket, s->scal);
    SIM_LAUNCHED(s);
    SIM_CK(s, cudaMemcpyAsync(s->h_pinned, s->scal, sizeof(double), cudaMemcpyDeviceToHost, s->stream));
    if (well_cnv_host) SIM_CK(s, cudaMemcpyAsync(s->h_pinned + 1, s->wcnv, sizeof(double), cudaMemcpyDeviceToHost, s->stream));
    SIM_CK(s, cudaStreamSynchronize(s->stream));
    *cnv_host = s->h_pinned[0];
    if (well_cnv_host) *well_cnv_host = s->h_pinned[1];
    return SIM_OK;
}

sim_status k_component_mass(sim_t *s, double *m3) {
    if (s->b == 2)
        mass_kernel<2><<<state_blocks(s->N), SIM_THREADS, 0, s->stream>>>(s->fc, s->gd, s->x, s->ph, poro_of(s), s->red, s->ticket, s->scal);
    else
        mass_kernel<3><<<state_blocks(s->N), SIM_THREADS, 0, s->stream>>>(s->fc, s->gd, s->x, s->ph, poro_of(s), s->red, s->ticket, s->scal);
    SIM_LAUNCHED(s);
    SIM_CK(s, cudaMemcpyAsync(s->h_pinned, s->scal, sizeof(double) * 3, cudaMemcpyDeviceToHost, s->stream));
    SIM_CK(s, cudaStreamSynchronize(s->stream));
    for (int c = 0; c < 3; c++) m3[c] = c < s->b ? s->h_pinned[c] : 0.0;
    return SIM_OK;
}

sim_status k_newton_update(sim_t *s, const double *dx) {
    if (s->b == 2)
        update_kernel<2><<<sim_blocks(s->N), SIM_THREADS, 0, s->stream>>>(s->N, s->opt.chop_ds, s->opt.chop_dp, dx, s->x, s->ph);
    else
        update_kernel<3><<<sim_blocks(s->N), SIM_THREADS, 0, s->stream>>>(s->N, s->opt.chop_ds, s->opt.chop_dp, dx, s->x, s->ph);
    SIM_LAUNCHED(s);
    return SIM_OK;
}

sim_status k_finite(sim_t *s, const double *v, long n, int *ok) {
    nonfinite_kernel<<<state_blocks(n), SIM_THREADS, 0, s->stream>>>(v, n, s->red, s->ticket, s->scal);
    SIM_LAUNCHED(s);
    SIM_CK(s, cudaMemcpyAsync(s->h_pinned, s->scal, sizeof(double), cudaMemcpyDeviceToHost, s->stream));
    SIM_CK(s, cudaStreamSynchronize(s->stream));
    *ok = s->h_pinned[0] == 0.0;
    return SIM_OK;
}

// ===========================================================================
// CNV without device allocation (sim_cnv_noalloc)
//
// Scratch: the per-block partial maxima and the last-block ticket live in a
// file-scope device array of NOALLOC_SCRATCH = SIM_RED_BLOCKS + 1 doubles
// (456 partials and one ticket word: 457 doubles, 3,656 bytes), held by every
// GPU that loads the library until the process exits.  Host code never uses
// the array's name as a pointer (on the host it is only a stand-in): every
// call looks the device address up with cudaGetSymbolAddress, with the
// caller's device current, so no address outlives a device reset.
// ===========================================================================
namespace {
constexpr int NOALLOC_SCRATCH = SIM_RED_BLOCKS + 1;   // partials + ticket word
static __device__ __align__(256) double g_cnv_scratch[NOALLOC_SCRATCH];

template <int B>
__global__ void cnv_noalloc_kernel(GridDesc g, const double *__restrict__ R, const double *__restrict__ poro, double dt,
                                   double r0, double r1, double r2, double *scratch, double *out) {
    const double m = block_reduce<1>(cnv_max<B>(g, R, poro, dt, r0, r1, r2));
    if (threadIdx.x == 0) scratch[blockIdx.x] = m;
    finish_grid<1>(scratch, 1, (unsigned int *)(scratch + SIM_RED_BLOCKS), out);
}
}  // namespace

extern "C" sim_status sim_cnv_noalloc(int32_t nx, int32_t ny, int32_t nz, double dx, double dy, double dz, int32_t b,
                                      const double *R_dev, const double *poro_dev, const double *cnv_rho, double dt,
                                      double *cnv_dev, void *cuda_stream) {
    if (!R_dev || !poro_dev || !cnv_rho || !cnv_dev) return sim_fail(nullptr, SIM_EINVAL, "sim_cnv_noalloc: NULL pointer");
    if (nx < 1 || ny < 1 || nz < 1 || !(dx > 0 && dy > 0 && dz > 0) || !(dt > 0) || (b != 2 && b != 3))
        return sim_fail(nullptr, SIM_EINVAL, "sim_cnv_noalloc: bad grid, block size or dt");
    for (int c = 0; c < b; c++)
        if (!(cnv_rho[c] > 0)) return sim_fail(nullptr, SIM_EINVAL, "sim_cnv_noalloc: cnv_rho must be positive");
    const long long N = (long long)nx * ny * nz;
    if (N * b > 0x7fffffffLL)
        return sim_fail(nullptr, SIM_ELIMIT, "sim_cnv_noalloc: N*b must stay below 2^31 (32-bit indexing)");
    int dev = 0;   // the caller's current device: the one whose copy of the array is used
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return sim_fail(nullptr, SIM_ECUDA, std::string("sim_cnv_noalloc: ") + cudaGetErrorString(e));
    // the array's device address on that device (a lookup, no allocation)
    double *scratch = nullptr;
    e = cudaGetSymbolAddress((void **)&scratch, g_cnv_scratch);
    if (e != cudaSuccess || !scratch)
        return sim_fail(nullptr, SIM_ECUDA, std::string("sim_cnv_noalloc: cudaGetSymbolAddress: ") + cudaGetErrorString(e));
    cudaStream_t st = (cudaStream_t)cuda_stream;
    // the ticket must start at zero; the partials are overwritten before use
    e = cudaMemsetAsync(scratch + SIM_RED_BLOCKS, 0, sizeof(double), st);
    if (e != cudaSuccess) return sim_fail(nullptr, SIM_ECUDA, std::string("sim_cnv_noalloc: ") + cudaGetErrorString(e));
    GridDesc g;
    g.nx = nx; g.ny = ny; g.nz = nz; g.N = (int)N; g.dx = dx; g.dy = dy; g.dz = dz; g.top = 0.0; g.H = 0;
    const double r2 = b == 3 ? cnv_rho[2] : 1.0;
    if (b == 2)
        cnv_noalloc_kernel<2><<<SIM_RED_BLOCKS, SIM_THREADS, 0, st>>>(g, R_dev, poro_dev, dt, cnv_rho[0], cnv_rho[1], r2,
                                                                     scratch, cnv_dev);
    else
        cnv_noalloc_kernel<3><<<SIM_RED_BLOCKS, SIM_THREADS, 0, st>>>(g, R_dev, poro_dev, dt, cnv_rho[0], cnv_rho[1], r2,
                                                                     scratch, cnv_dev);
    e = cudaGetLastError();
    if (e != cudaSuccess) return sim_fail(nullptr, SIM_ECUDA, std::string("sim_cnv_noalloc: ") + cudaGetErrorString(e));
    return SIM_OK;
}
