// Hand-written adjoint (vector-Jacobian product) of the semi-discrete
// operator dU/dt = -sum_d (F_{j+1/2} - F_{j-1/2}) / dx_d.
//
// For a cotangent w (one value per cell and variable) the face flux F_f of
// direction d receives the cotangent phi_f = (w_{j+1} - w_j) / dx_d (w = 0
// outside the domain), and gU = sum_f (dF_f / dU_stencil)^T phi_f.  Every
// face recomputes its forward quantities (Roe state, detector, LLF speeds,
// projections, reconstructions: nothing is stored by the forward pass) and
// then runs the reverse of each step:
//   back-projection (Eq. reconstruction2)  -> the face steps of vjp_weno_line
//   reconstruction (Eq. eq6, eq11, eq18, eq8-r) -> recon_adj
//   splitting and projection (Eq. flxuspliting, eqchara) -> proj_all_adj
//   regularization parameter (Eq. eq27-29) and detector (Eq. eq28)
//   Roe average (Sec. 2.4 step (1)) -> roe_adj
//   cell primitives and physical flux -> cell_adj
// The hybrid flag and the cell that attains each LLF maximum are held at
// their forward values (first index on ties): the operator is piecewise
// smooth and this is the derivative of the active piece.
//
// Accumulation is deterministic: a tile of SEG cells recomputes the SEG + 5
// faces that touch its cells, writes each face's contribution to its six
// stencil cells in shared memory, and gathers them per cell in face order.
// A linear-upwind face stores two bar vectors, of the central-flux sum and
// of the detector difference, and the gather applies their fixed stencil
// weights; a WENO face stores U and F bars for each of its six cells.  Every
// face adds Roe-field bars for its two neighbours and one bar per LLF speed
// for the cell attaining it.
//
// Each direction runs in two passes over the same tiles.  Pass 0 (k_vjp)
// takes the linear-upwind faces, writes (or adds) the gradient, and lists
// each tile that has a WENO face among the faces it recomputes, with a mask
// of its lines.  Pass 1 (k_vjp_weno) takes the WENO faces of the listed lines
// and adds their contributions.  The WENO reverse of a face holds 6 x nvar
// projections and their bars; pass 1 spreads it over the lanes as the forward
// sweep does, and keeping it out of pass 0 lets the common linear-upwind
// tiles run with far fewer registers and more resident warps.
// Contributions to ghost cells go to a per-line buffer that a second kernel
// maps back through the boundary conditions.
#pragma once

#include "weno_kernels.cuh"

namespace wis {

// q sgn(x): q with x's sign applied, zero where x is zero; for double on the
// integer pipes (the FP64 pipe bounds the adjoint), the same value as the
// product for finite q (a zero result may differ in its sign only)
__device__ __forceinline__ double times_sign(double q, double x)
{
    const long long xb = __double_as_longlong(x);
    const long long r = __double_as_longlong(q) ^ (xb & (long long)0x8000000000000000ULL);
    return (xb & 0x7fffffffffffffffLL) == 0 ? 0.0 : __longlong_as_double(r);
}
__device__ __forceinline__ float times_sign(float q, float x)
{
    return x > 0.0f ? q : (x < 0.0f ? -q : 0.0f);
}

// record bars of one cell (NQ entries, same layout as CellLayout) -> dU;
// isq = 1/sqrt(rho), ic = 1/c, the pressure p and the sound speed c as
// cell_prims computed them for the forward record
template <typename T, int DIM, int DIR>
__device__ __forceinline__ void cell_adj(const T* U, T gamma, T isq, T ic, T p, T c, const T* qb, T* Ub)
{
    using CL = CellLayout<DIM>;
    constexpr int NV = DIM + 2;
    const T gm1 = gamma - T(1);
    const T rho = U[0];
    const T irho = isq * isq;
    T m2 = T(0);
#pragma unroll
    for (int k = 0; k < DIM; ++k) m2 = fmaT(U[1 + k], U[1 + k], m2);
    const T E = U[DIM + 1];
    const T un = U[1 + DIR] * irho;
    const T Ep = E + p;

#pragma unroll
    for (int v = 0; v < NV; ++v) Ub[v] = qb[CL::U + v];
    T unb = T(0), cb = T(0), isqb = T(0), Epb = T(0), pb = T(0), irhob = T(0), m2b = T(0);
    // |un - c|, |un|, |un + c|: the bars take the signs of their arguments
    const T lm = times_sign(qb[CL::LM], un - c), lp = times_sign(qb[CL::LP], un + c);
    unb += lm; cb -= lm;
    unb += times_sign(qb[CL::L0], un);
    unb += lp; cb += lp;
    Ub[0] += qb[CL::SQ] * isq; isqb += qb[CL::SQ] * rho;
    Epb += qb[CL::SH] * isq; isqb += qb[CL::SH] * Ep;
#pragma unroll
    for (int k = 0; k < DIM; ++k) { Ub[1 + k] += qb[CL::SU + k] * isq; isqb += qb[CL::SU + k] * U[1 + k]; }
    Epb += qb[CL::F + DIM + 1] * un; unb += qb[CL::F + DIM + 1] * Ep;
#pragma unroll
    for (int k = 0; k < DIM; ++k) { Ub[1 + k] += qb[CL::F + 1 + k] * un; unb += qb[CL::F + 1 + k] * U[1 + k]; }
    pb += qb[CL::F + 1 + DIR];
    Ub[1 + DIR] += qb[CL::F + 0];
    Ub[DIM + 1] += Epb; pb += Epb;
    Ub[1 + DIR] += unb * irho; irhob += unb * U[1 + DIR];
    // c = sqrt(gamma p irho): dc = gamma (irho dp + p dirho) / (2 c)
    const T cg = halve(cb) * ic * gamma;
    pb = fmaT(cg, irho, pb); irhob = fmaT(cg, p, irhob);
    // p = gm1 (E - irho m2 / 2)
    const T pg = pb * gm1, hpg = halve(pg);
    Ub[DIM + 1] += pg; irhob = fmaT(-hpg, m2, irhob); m2b = -hpg * irho;
    // m2 = |m|^2, irho = isq^2, isq = rho^-1/2
    const T m2b2 = m2b + m2b;
#pragma unroll
    for (int k = 0; k < DIM; ++k) Ub[1 + k] = fmaT(U[1 + k], m2b2, Ub[1 + k]);
    isqb = fmaT(isq + isq, irhob, isqb);
    Ub[0] = fmaT(isqb, -halve(isq) * irho, Ub[0]);
}

template <typename T, int DIM> struct RoeBar {
    T u[DIM];
    T c, ic, H, b1, hq2, rt;
};

template <typename T, int DIM>
__device__ __forceinline__ void zero(RoeBar<T, DIM>& b)
{
#pragma unroll
    for (int k = 0; k < DIM; ++k) b.u[k] = T(0);
    b.c = b.ic = b.H = b.b1 = b.hq2 = b.rt = T(0);
}

// adjoint of w = L x (proj_all): accumulates xb and rb
template <typename T, int DIM, int DIR>
__device__ __forceinline__ void proj_all_adj(const Roe<T, DIM>& r, const T* x, const T* wb, T* xb,
                                             RoeBar<T, DIM>& rb)
{
    constexpr int LAST = DIM + 1;
    T dot = r.u[0] * x[1];
#pragma unroll
    for (int k = 1; k < DIM; ++k) dot = fmaT(r.u[k], x[1 + k], dot);
    const T y = fmaT(r.hq2, x[0], x[DIM + 1]) - dot;
    const T z = fmaT(r.u[DIR], x[0], -x[1 + DIR]);
    const T t1b = halve(wb[0] + wb[LAST]) - wb[1];
    const T ab = halve(wb[0] - wb[LAST]);
    int s = 2;
#pragma unroll
    for (int t = 0; t < DIM; ++t) {
        if (t == DIR) continue;
        xb[1 + t] += wb[s];
        xb[0] -= wb[s] * r.u[t];
        rb.u[t] -= wb[s] * x[0];
        ++s;
    }
    xb[0] += wb[1];
    const T zb = ab * r.ic;
    rb.ic += ab * z;
    rb.u[DIR] += zb * x[0];
    xb[0] += zb * r.u[DIR];
    xb[1 + DIR] -= zb;
    rb.b1 += t1b * y;
    const T yb = t1b * r.b1;
    rb.hq2 += yb * x[0];
    xb[0] += yb * r.hq2;
    xb[DIM + 1] += yb;
#pragma unroll
    for (int k = 0; k < DIM; ++k) { rb.u[k] -= yb * x[1 + k]; xb[1 + k] -= yb * r.u[k]; }
}

// adjoint of the Roe average; gab/gbb: bars of the Roe fields of cells j and
// j+1, relative to CL::SU (sqrt(rho) u at 0 .. DIM-1, sqrt(rho) H at DIM,
// sqrt(rho) at DIM + 1)
template <typename T, int DIM, typename GA, typename GB>
__device__ __forceinline__ void roe_adj(GA get_a, GB get_b, T gamma, const Roe<T, DIM>& r, RoeBar<T, DIM> rb,
                                        T* gab, T* gbb)
{
    using CL = CellLayout<DIM>;
    const T gm1 = gamma - T(1);
    const T sa = get_a(CL::SQ), sb = get_b(CL::SQ);
    const T inv = Ar<T>::rcp_f(sa + sb);   // as in roe_state
    // b1 = gm1 ic^2; c = c2 ic (= sqrt c2); ic = c2^-1/2; c2 = gm1 (H - hq2)
    rb.ic = fmaT(rb.b1 * gm1, r.ic + r.ic, rb.ic);
    const T ic3 = r.ic * r.ic * r.ic;
    const T c2b = halve(fmaT(rb.c, r.ic, -rb.ic * ic3));
    rb.H += c2b * gm1;
    rb.hq2 -= c2b * gm1;
    T invb = T(0);
#pragma unroll
    for (int k = 0; k < DIM; ++k) {
        const T ub = rb.u[k] + r.u[k] * rb.hq2;
        gab[k] += ub * inv;
        gbb[k] += ub * inv;
        invb += ub * (get_a(CL::SU + k) + get_b(CL::SU + k));
    }
    gab[DIM] += rb.H * inv;
    gbb[DIM] += rb.H * inv;
    invb += rb.H * (get_a(CL::SH) + get_b(CL::SH));
    const T sb_ = -invb * inv * inv;
    gab[DIM + 1] += sb_ + rb.rt * sb;
    gbb[DIM + 1] += sb_ + rb.rt * sa;
}

// 1 / x of a positive normal number: refined in double, rounded in float
__device__ __forceinline__ double inv_pos(double x) { return rcp_newton(x); }
__device__ __forceinline__ float inv_pos(float x) { return 1.0f / x; }

// adjoint of the reconstruction: fb -> bars of a..e (set) and of lam; returns
// the reconstructed value
template <typename T>
__device__ __forceinline__ T recon_adj(T a, T b, T c, T d, T e, T lam, T eps, T fb, T* xb, T& lamb)
{
    const T q0 = T(0.5) * (c + d);
    const T q1 = fmaT(T(1.5), c, T(-0.5) * b);
    const T q2 = fmaT(T(1.0 / 3.0), c, fmaT(T(5.0 / 6.0), d, T(-1.0 / 6.0) * e));
    const T q3 = fmaT(T(1.0 / 3.0), a, fmaT(T(-7.0 / 6.0), b, T(11.0 / 6.0) * c));
    const T b0 = (d - c) * (d - c), b1 = (c - b) * (c - b);
    const T t2 = fmaT(T(-2), d, c) + e, s2 = fmaT(T(-4), d, T(3) * c) + e;
    const T be2 = fmaT(T(13.0 / 12.0), t2 * t2, T(0.25) * (s2 * s2));
    const T t3 = fmaT(T(-2), b, a) + c, s3 = fmaT(T(-4), b, a) + T(3) * c;
    const T be3 = fmaT(T(13.0 / 12.0), t3 * t3, T(0.25) * (s3 * s3));
    const T tt = fmaT(T(-4), b + d, a + e) + T(6) * c, st = fmaT(T(2), b - d, e - a);
    const T tau = fmaT(T(13.0 / 12.0), tt * tt, T(0.25) * (st * st));
    const T te = fmaT(T(-2), c, b + d);
    const T E = (te * te) * T(1.0 / 45.0);
    const T dk[4] = {T(0.4), T(0.2), T(0.3), T(0.1)};
    const T beta[4] = {b0, b1, be2, be3};
    const T lt = lam * tau;
    T iD[4], al[4];
    T S = T(0);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        iD[k] = inv_pos(fmaT(lam, beta[k], (k < 2 ? E : T(0)) + eps));
        al[k] = dk[k] * (T(1) + lt * iD[k]);
        S += al[k];
    }
    const T iS = inv_pos(S);
    const T q[4] = {q0, q1, q2, q3};
    T fh = T(0);
#pragma unroll
    for (int k = 0; k < 4; ++k) fh = fmaT(al[k] * iS, q[k], fh);
    // reverse
    T qb[4], ltb = T(0), betab[4], Eb = T(0);
    lamb = T(0);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        qb[k] = fb * al[k] * iS;
        const T alb = (q[k] - fh) * fb * iS;
        const T r = alb * dk[k] * iD[k];
        ltb += r;
        const T Db = -r * (lt * iD[k]);
        lamb += Db * beta[k];
        betab[k] = Db * lam;
        if (k < 2) Eb += Db;
    }
    lamb += ltb * tau;
    const T taub = ltb * lam;
    T ab = T(0), bb = T(0), cb = T(0), db = T(0), eb = T(0);
    // beta_0, beta_1
    db += T(2) * (d - c) * betab[0]; cb -= T(2) * (d - c) * betab[0];
    cb += T(2) * (c - b) * betab[1]; bb -= T(2) * (c - b) * betab[1];
    // beta_2
    T tb = betab[2] * T(13.0 / 6.0) * t2, sb = betab[2] * T(0.5) * s2;
    cb += tb + T(3) * sb; db += T(-2) * tb - T(4) * sb; eb += tb + sb;
    // beta_3
    tb = betab[3] * T(13.0 / 6.0) * t3; sb = betab[3] * T(0.5) * s3;
    ab += tb + sb; bb += T(-2) * tb - T(4) * sb; cb += tb + T(3) * sb;
    // tau_5
    tb = taub * T(13.0 / 6.0) * tt; sb = taub * T(0.5) * st;
    ab += tb - sb; eb += tb + sb; bb += T(-4) * tb + T(2) * sb; db += T(-4) * tb - T(2) * sb; cb += T(6) * tb;
    // E
    tb = Eb * T(2.0 / 45.0) * te;
    bb += tb; cb -= T(2) * tb; db += tb;
    // candidate fluxes
    ab += qb[3] * T(1.0 / 3.0);
    bb += T(-0.5) * qb[1] + T(-7.0 / 6.0) * qb[3];
    cb += T(0.5) * qb[0] + T(1.5) * qb[1] + T(1.0 / 3.0) * qb[2] + T(11.0 / 6.0) * qb[3];
    db += T(0.5) * qb[0] + T(5.0 / 6.0) * qb[2];
    eb += T(-1.0 / 6.0) * qb[2];
    xb[0] = ab; xb[1] = bb; xb[2] = cb; xb[3] = db; xb[4] = eb;
    return fh;
}

struct VjpArgs {
    const void* U;      // state, interior only (the caller's array)
    const void* W;      // cotangent, interior only
    void* G;            // gradient, interior only (written / accumulated)
    void* ghost;        // [line][6][NV] gradients of ghost cells
    int* n_weno_tiles;  // tiles of this direction with a WENO face (zero before pass 0)
    int2* weno_tiles;   // their linear indices and the mask of their lines with one, in no
                        // particular order (pass 0 appends)
    int tiles[3];       // tile grid of this direction (set by the launcher)
    int accumulate;     // 0: G = ..., 1: G += ... (pass 0; pass 1 always adds)
    int n[3];
    long long sy, sz, sv, off0;
    double inv_dx, eps_h, gamma, eps, c_lambda;
    double slim;   // 60 sqrt(eps_h), as in the forward sweep
    double lam_k;  // c_lambda / 3600
    int fx;        // FP64: the six-point sums of linear faces in 64-bit integers, as in the
                   // forward sweep (use_fx)
    // the same pre-rounded for float kernels: a conversion or a division per
    // thread would run on the slow FP64 pipe (38% of the cycles of the float
    // x pass)
    float inv_dx_f, gamma_f, eps_f, slim_f, lam_k_f;
    int hybrid;
    // boundary conditions of this direction, for the ghost cells computed
    // while staging (the fields stage_cell reads: bc_lo, bc_hi, bc_state,
    // fix_line, tm = null)
    SweepArgs bc;
    // cell primitives (cell_prims, PrimLayout records at STRIDE g): P read
    // (an earlier direction stored them), Pout computed and stored for the
    // tile's own cells, both null: computed and kept to the tile (FP64 only)
    const void* P;
    void* Pout;
};

// A tile is LINES grid lines x SEG cells along the sweep, one thread per
// face.  Lines along x take one line of 59 cells.  For y and z lines in FP32
// a tile takes 8 x-adjacent lines of 27 cells, so that the strided loads of
// one line position cover a 32-byte sector; in FP64 the arithmetic bounds
// those sweeps and one line per tile keeps 4 CTAs per SM resident.
template <typename T, int DIM, int DIR> struct VjpTile {
    static constexpr int LINES = (DIR != 0 && sizeof(T) == 4) ? 8 : 1;
    static constexpr int SEG = LINES == 1 ? 59 : 27;
    static constexpr int NT = LINES * (SEG + 5);
};

template <typename T, int DIM, int DIR>
struct VjpSmem {
    static constexpr int LINES = VjpTile<T, DIM, DIR>::LINES;
    static constexpr int SEG = VjpTile<T, DIM, DIR>::SEG;
    static constexpr int NF = SEG + 5;          // faces c0-2 .. c0+SEG+2 per line
    static constexpr int NC = SEG + 10;         // cells c0-5 .. c0+SEG+4 per line
    static constexpr int LNF = LINES * NF, LNC = LINES * NC;
    static constexpr int NQ = CellLayout<DIM>::NQ;
    static constexpr int NV = DIM + 2;
    // per face: the two bar vectors of a linear-upwind face (NUF entries),
    // Roe-field bars of cells 2 and 3 (the face's neighbours), the three LLF
    // speed bars, and (as one int) the stencil slots of the cells attaining
    // the speeds and whether the pass takes the face
    // per cell after the record: 1/sqrt(rho), 1/c and, in FP64, p and c
    // (in FP32 the per-cell reverse recomputes those two: two more staged
    // rows cost the shared-memory-bound float tiles more than they save)
    static constexpr int NX = sizeof(T) == 8 ? 4 : 2;
    static constexpr int NUF = 2 * NV;
    static constexpr int NRB = DIM + 2;
    static constexpr int NFB = NUF + 2 * NRB + 3;
    static constexpr size_t bytes =
        sizeof(T) * ((size_t)(NQ + NX) * LNC + (size_t)NV * LNC + (size_t)LNF * NFB) + sizeof(int) * (size_t)LNF;
};

// One tile of one direction of the VJP: tile (bx, by, bz) = LINES grid lines
// x SEG cells; shared arrays hold position p of line l at p * LINES + l.
// Returns (to every thread) the mask of its lines that have a WENO face.
template <typename T, int DIM, int DIR>
__device__ __forceinline__ unsigned int vjp_tile(const VjpArgs& a, int bx, int by, int bz, unsigned char* smem_raw)
{
    using CL = CellLayout<DIM>;
    using SM = VjpSmem<T, DIM, DIR>;
    constexpr int NV = DIM + 2, NQ = CL::NQ, SEG = SM::SEG, NF = SM::NF;
    constexpr int LINES = SM::LINES, LNF = SM::LNF, LNC = SM::LNC;
    constexpr int NT = VjpTile<T, DIM, DIR>::NT;
    constexpr int NUF = SM::NUF, NRB = SM::NRB;
    T* cq = reinterpret_cast<T*>(smem_raw);   // [NQ + NX][NC][LINES] records, 1/sqrt(rho), 1/c (, p, c)
    T* wq = cq + (NQ + SM::NX) * LNC;         // [NV][NC][LINES] cotangent
    T* UF = wq + NV * LNC;                    // [NF][LINES][NUF] bars of dU and of the central-flux sum
    T* RB = UF + LNF * NUF;                  // [NF][LINES][2][NRB] Roe-field bars of cells 2 and 3
    T* SP = RB + LNF * 2 * NRB;               // [NF][LINES][3] LLF speed bars
    int* SL = reinterpret_cast<int*>(SP + LNF * 3);   // [NF][LINES] slots attaining the speeds, face taken
    constexpr int SKIP = 1 << 12;   // the face belongs to the other pass

    const int nd = a.n[DIR];
    const int c0 = bx * SEG;
    // line coordinates: the two indices other than DIR; the lines of a
    // multi-line tile are consecutive in x
    int ix0 = 0, j = 0, k = 0;
    if (DIR == 0) { j = by; k = bz; }
    else if (DIR == 1) { ix0 = by * LINES; k = bz; }
    else { ix0 = by * LINES; j = bz; }
    const int nlx = DIR == 0 ? 1 : (a.n[0] - ix0 < LINES ? a.n[0] - ix0 : LINES);   // lines present
    const long long sd = DIR == 0 ? 1LL : (DIR == 1 ? a.sy : a.sz);
    const long long base0 = a.off0 + (long long)ix0 + (long long)j * a.sy + (long long)k * a.sz;
    const T* Ug = reinterpret_cast<const T*>(a.U);
    const T* Wg = reinterpret_cast<const T*>(a.W);
    const T gamma = pick<T>(a.gamma, a.gamma_f);

    __shared__ unsigned int weno_lines;
    if (threadIdx.x == 0) weno_lines = 0u;

    // stage cells c0-5 .. c0+SEG+4 that exist (-3 .. nd+2); ghost cells come
    // from the boundary conditions, and the cotangent is zero on them
    for (int idx = threadIdx.x; idx < LNC; idx += NT) {
        const int p = idx / LINES, l = idx - (idx / LINES) * LINES;
        const int cell = c0 - 5 + p;
        if (l < nlx && cell >= -3 && cell <= nd + 2) {
            // in-plane index of the line for the boundary conditions: the row
            // for x sweeps, the column for y and z sweeps
            const int line = DIR == 0 ? j : ix0 + l;
            using PL = PrimLayout<DIM>;
            T U[NV], q[NQ], inv[2], P[PL::NP], W[NV];
            const bool inside = cell >= 0 && cell < nd;
            const long long g = base0 + l + (long long)cell * sd;
#pragma unroll
            for (int v = 0; v < NV; ++v) W[v] = inside ? Wg[g + v * a.sv] : T(0);
            if constexpr (sizeof(T) == 8) {
                long long gs = 0;
                bool flip = false;
                const int fixed = cell_source<DIR>(a.bc, base0 + l, line, cell, nd, gs, flip);
                if (fixed >= 0) {
#pragma unroll
                    for (int v = 0; v < NV; ++v) U[v] = a.bc.bc_state[fixed][v];
                    cell_prims<T, DIM>(U, gamma, gamma - T(1), P, inv);
                } else {
#pragma unroll
                    for (int v = 0; v < NV; ++v) U[v] = Ug[gs + v * a.sv];
                    if (a.P != nullptr) {
                        // 1/sqrt(rho) = sqrt(rho) / rho and 1/c from the
                        // stored record (within an ulp or two of the staged
                        // values)
                        load_prims<DIM>(reinterpret_cast<const T*>(a.P), gs, P);
                        inv[0] = P[PL::SQ] * P[PL::IRHO];
                        inv[1] = Ar<T>::rcp_f(P[PL::C]);
                    } else {
                        cell_prims<T, DIM>(U, gamma, gamma - T(1), P, inv);
                        if (a.Pout != nullptr && cell >= c0 && cell < c0 + SEG && cell < nd)
                            store_prims<DIM>(reinterpret_cast<T*>(a.Pout), gs, P);
                    }
                    if (flip) {
                        U[1 + DIR] = -U[1 + DIR];
                        P[PL::SU + DIR] = -P[PL::SU + DIR];
                    }
                }
            } else {
                // float: no stored primitives (the float tiles were measured
                // slower with the source lookup above)
                stage_cell<T, DIM, DIR>(a.bc, Ug, base0 + l, line, cell, nd, U);
                cell_prims<T, DIM>(U, gamma, gamma - T(1), P, inv);
            }
#pragma unroll
            for (int v = 0; v < NV; ++v) wq[v * LNC + idx] = W[v];
            cell_record<T, DIM, DIR>(U, P, q);
#pragma unroll
            for (int kk = 0; kk < NQ; ++kk) cq[kk * LNC + idx] = q[kk];
            cq[NQ * LNC + idx] = inv[0];
            cq[(NQ + 1) * LNC + idx] = inv[1];
            if constexpr (SM::NX == 4) {
                cq[(NQ + 2) * LNC + idx] = P[PrimLayout<DIM>::P];
                cq[(NQ + 3) * LNC + idx] = P[PrimLayout<DIM>::C];
            }
        } else {
#pragma unroll
            for (int v = 0; v < NV; ++v) wq[v * LNC + idx] = T(0);
        }
    }
    __syncthreads();

    // ---- per face: forward recompute and reverse -------------------------
    const T slim = pick<T>(a.slim, a.slim_f), inv_dx = pick<T>(a.inv_dx, a.inv_dx_f);
    // Float: the gradient of earlier directions is loaded before the faces,
    // for the first cell that this thread gathers
    constexpr bool EARLY = sizeof(T) == 4;
    T eg[NV];
    if constexpr (EARLY) {
        const int p = threadIdx.x / LINES, l = threadIdx.x - (threadIdx.x / LINES) * LINES;
        const int cell = c0 - 3 + p;
        const bool read = a.accumulate && l < nlx && cell >= c0 && cell < c0 + SEG && cell < nd;
        const T* Gr = reinterpret_cast<const T*>(a.G) + base0 + l + (long long)cell * sd;
#pragma unroll
        for (int v = 0; v < NV; ++v) eg[v] = read ? Gr[v * a.sv] : T(0);
    }

    for (int ff = threadIdx.x; ff < LNF; ff += NT) {
        const int f = ff / LINES, l = ff - (ff / LINES) * LINES;
        const int face = c0 - 2 + f;            // face i' between cells i'-1 and i'
        if (l >= nlx || face < 0 || face > nd) continue;
        // stencil cell j-2 = face-3 sits at position f of line l
        auto rec = [&](int m, int kk) -> T { return cq[kk * LNC + (f + m) * LINES + l]; };
        // the bars of the detector difference (U slots) and of the
        // central-flux sum (F slots)
        T* UFf = UF + (size_t)ff * NUF;
        T* RBf = RB + (size_t)ff * 2 * NRB;    // Roe-field bars of cells 2 and 3
        // cotangent of the face flux: (w_{right} - w_{left}) / dx
        T phi[NV];
#pragma unroll
        for (int v = 0; v < NV; ++v)
            phi[v] = (wq[v * LNC + (f + 3) * LINES + l] - wq[v * LNC + (f + 2) * LINES + l]) * inv_dx;

        auto ga = [&](int kk) -> T { return rec(2, kk); };
        auto gb = [&](int kk) -> T { return rec(3, kk); };
        const Roe<T, DIM> r = roe_state<T, DIM>(ga, gb, gamma - T(1));
        RoeBar<T, DIM> rb;
        zero(rb);
        T dU[NV];
#pragma unroll
        for (int v = 0; v < NV; ++v) {
            const int kk = CL::U + v;
            if (sizeof(T) == 8 && a.fx) {
                const double x[6] = {rec(0, kk), rec(1, kk), rec(2, kk), rec(3, kk), rec(4, kk), rec(5, kk)};
                dU[v] = T(fx_detector(x));
            } else {
                dU[v] = fmaT(T(10), rec(2, kk) - rec(3, kk),
                             fmaT(T(5), rec(4, kk) - rec(1, kk), rec(0, kk) - rec(5, kk)));
            }
        }
        T w[NV];
        proj_all<T, DIM, DIR>(r, dU, w);
        const T lim = slim * r.rt;
        bool smooth = a.hybrid != 0;
#pragma unroll
        for (int s = 0; s < NV; ++s) smooth = smooth && abs_lt(w[s], lim);
        if (!smooth) {   // pass 1 takes this face
            atomicOr(&weno_lines, 1u << l);
            SL[ff] = SKIP;
            continue;
        }
        // LLF speeds and the cells attaining them
        T am = rec(0, CL::LM), a0 = rec(0, CL::L0), ap = rec(0, CL::LP);
        int im = 0, i0 = 0, ip = 0;
#pragma unroll
        for (int m = 1; m < 6; ++m) {
            // the speeds are non-negative: compared on their bit patterns
            // (integer pipes), first index on ties as before
            const T xm = rec(m, CL::LM), x0 = rec(m, CL::L0), xp = rec(m, CL::LP);
            if (lt_nn(am, xm)) { am = xm; im = m; }
            if (lt_nn(a0, x0)) { a0 = x0; i0 = m; }
            if (lt_nn(ap, xp)) { ap = xp; ip = m; }
        }
        T alb_m = T(0), alb_0 = T(0), alb_p = T(0);
        T wb[NV], dUb[NV];
#pragma unroll
        for (int s = 0; s < NV; ++s) { wb[s] = T(0); dUb[s] = T(0); }
        {
            // F = [central(F) + a0 dU + k0 R^{u-c} + k3 R^{u+c}] / 60 with
            // k0 = (am - a0) w_0, k3 = (ap - a0) w_last, the form the forward
            // sweep evaluates (ups_dissipation_add); the gather applies the
            // central weights to the bar Fb of the sum
            T Fb[NV];
#pragma unroll
            for (int v = 0; v < NV; ++v) {
                Fb[v] = phi[v] * T(1.0 / 60.0);
                UFf[CL::F + v] = Fb[v];
            }
            constexpr int LAST = NV - 1;
            const T k0 = (am - a0) * w[0], k3 = (ap - a0) * w[LAST];
            const T sum = k0 + k3, dd = k3 - k0;
            const T unc = r.u[DIR] * r.c;
            // out[0] += s; out[1 + k] += u_k s (+ c dd along DIR); out[E] += H s + u_n c dd
            T sb = fmaT(r.H, Fb[LAST], Fb[0]);
#pragma unroll
            for (int k = 0; k < DIM; ++k) {
                sb = fmaT(r.u[k], Fb[1 + k], sb);
                rb.u[k] = fmaT(sum, Fb[1 + k], rb.u[k]);
            }
            const T ddb = fmaT(r.c, Fb[1 + DIR], unc * Fb[LAST]);
            rb.H = fmaT(sum, Fb[LAST], rb.H);
            const T uncb = dd * Fb[LAST];
            rb.u[DIR] = fmaT(uncb, r.c, rb.u[DIR]);
            rb.c = fmaT(uncb, r.u[DIR], fmaT(dd, Fb[1 + DIR], rb.c));
            const T k0b = sb - ddb, k3b = sb + ddb;
            alb_m = k0b * w[0];
            alb_p = k3b * w[LAST];
            wb[0] = k0b * (am - a0);
            wb[LAST] = k3b * (ap - a0);
            // a0 dU: the entropy and shear fields' speed
            T dot = T(0);
#pragma unroll
            for (int v = 0; v < NV; ++v) {
                dot = fmaT(Fb[v], dU[v], dot);
                dUb[v] = a0 * Fb[v];
            }
            alb_0 = dot - alb_m - alb_p;
        }
        // detector: w = L dU, dU = (U0 - U5) + 5 (U4 - U1) + 10 (U2 - U3)
        proj_all_adj<T, DIM, DIR>(r, dU, wb, dUb, rb);
#pragma unroll
        for (int v = 0; v < NV; ++v) UFf[CL::U + v] = dUb[v];
        SP[ff * 3 + 0] = alb_m;
        SP[ff * 3 + 1] = alb_0;
        SP[ff * 3 + 2] = alb_p;
        SL[ff] = im | (i0 << 4) | (ip << 8);
#pragma unroll
        for (int kk = 0; kk < 2 * NRB; ++kk) RBf[kk] = T(0);
        roe_adj<T, DIM>(ga, gb, gamma, r, rb, RBf, RBf + NRB);
    }
    __syncthreads();
    const unsigned int any_weno = weno_lines;

    // ---- gather per cell: faces i' in [i-2, i+3], stencil slot m = i - i' + 3
    T* Gg = reinterpret_cast<T*>(a.G);
    T* ghost = reinterpret_cast<T*>(a.ghost);
    const bool first = c0 == 0, last = c0 + SEG >= nd;
    for (int idx = threadIdx.x; idx < LINES * (SEG + 6); idx += NT) {
        const int p = idx / LINES, l = idx - (idx / LINES) * LINES;
        const int cell = c0 - 3 + p;   // owned cells c0..c0+SEG-1 and boundary ghosts
        const bool owned = cell >= c0 && cell < c0 + SEG && cell < nd;
        const bool gl = first && cell < 0 && cell >= -3;
        const bool gr = last && cell >= nd && cell <= nd + 2;
        if (l >= nlx || (!owned && !gl && !gr)) continue;
        T qb[NQ];
#pragma unroll
        for (int kk = 0; kk < NQ; ++kk) qb[kk] = T(0);
        // FP64: the face (index into the face arrays) that gives
        // this cell its stencil slot m, -1 where none does
        int fslot[6] = {-1, -1, -1, -1, -1, -1};
        // central-flux and detector weights of stencil slot m (FP32)
        constexpr T cf[6] = {T(1), T(-8), T(37), T(37), T(-8), T(1)};
        constexpr T cd[6] = {T(1), T(-5), T(10), T(-10), T(5), T(-1)};
#pragma unroll
        for (int m = 5; m >= 0; --m) {
            const int fi = cell - m + 3;   // faces in increasing order
            if (fi < 0 || fi > nd) continue;
            const int f = fi - (c0 - 2);
            if (f < 0 || f >= NF) continue;
            const int ff = f * LINES + l;
            const int sl = SL[ff];
            if (sl & SKIP) continue;
            // the entries this cell receives from face fi, in the record
            // layout; the others are zero for it
            if constexpr (sizeof(T) == 8) {
                fslot[m] = ff;
            } else {
                const T* uf = UF + (size_t)ff * NUF;
#pragma unroll
                for (int v = 0; v < NV; ++v) {
                    qb[CL::U + v] = fmaT(cd[m], uf[CL::U + v], qb[CL::U + v]);
                    qb[CL::F + v] = fmaT(cf[m], uf[CL::F + v], qb[CL::F + v]);
                }
            }
            if (m == 2 || m == 3) {
                const T* rbp = RB + ((size_t)ff * 2 + (m - 2)) * NRB;
#pragma unroll
                for (int kk = 0; kk < NRB; ++kk) qb[CL::SU + kk] += rbp[kk];
            }
            if ((sl & 15) == m) qb[CL::LM] += SP[ff * 3 + 0];
            if (((sl >> 4) & 15) == m) qb[CL::L0] += SP[ff * 3 + 1];
            if (((sl >> 8) & 15) == m) qb[CL::LP] += SP[ff * 3 + 2];
        }
        if constexpr (sizeof(T) == 8) {
            // stencil weights of slot m: detector (1, -5, 10, -10, 5, -1)
            // on the U slots, central flux (1, -8, 37, 37, -8, 1) on the F
            // slots, applied as sums and differences of the symmetric pairs
            // (10 FP64 operations per variable instead of 12, none with a.fx;
            // 121x97x113: passes 0 of the three directions 3.53 -> 3.13 ms; in FP32 the
            // six loads held at once cost the 256-thread tiles a CTA per SM,
            // so FP32 keeps one multiply-add per slot)
#pragma unroll
            for (int v = 0; v < NV; ++v) {
                T bu[6], bf[6];
#pragma unroll
                for (int m = 0; m < 6; ++m) {
                    const T* uf = UF + (size_t)(fslot[m] < 0 ? 0 : fslot[m]) * NUF;
                    bu[m] = fslot[m] < 0 ? T(0) : uf[CL::U + v];
                    bf[m] = fslot[m] < 0 ? T(0) : uf[CL::F + v];
                }
                if (a.fx) {
                    qb[CL::U + v] = T(fx_detector(reinterpret_cast<const double*>(bu)));
                    qb[CL::F + v] = T(fx_central_flux(reinterpret_cast<const double*>(bf)));
                } else {
                    qb[CL::U + v] = fmaT(T(10), bu[2] - bu[3], fmaT(T(5), bu[4] - bu[1], bu[0] - bu[5]));
                    qb[CL::F + v] = fmaT(T(37), bf[2] + bf[3], fmaT(T(-8), bf[1] + bf[4], bf[0] + bf[5]));
                }
            }
        }
        const int pc = cell - (c0 - 5);
        T U[NV], Ub[NV];
#pragma unroll
        for (int v = 0; v < NV; ++v) U[v] = cq[(CL::U + v) * LNC + pc * LINES + l];
        const int ci = pc * LINES + l;
        const T isq = cq[NQ * LNC + ci], ic = cq[(NQ + 1) * LNC + ci];
        T pc_p, pc_c;
        if constexpr (SM::NX == 4) {
            pc_p = cq[(NQ + 2) * LNC + ci];
            pc_c = cq[(NQ + 3) * LNC + ci];
        } else {
            // p and c as cell_prims forms them
            const T irho = isq * isq;
            T m2 = T(0);
#pragma unroll
            for (int k = 0; k < DIM; ++k) m2 = fmaT(U[1 + k], U[1 + k], m2);
            pc_p = (gamma - T(1)) * fmaT(T(-0.5) * irho, m2, U[DIM + 1]);
            pc_c = gamma * pc_p * irho * ic;
        }
        cell_adj<T, DIM, DIR>(U, gamma, isq, ic, pc_p, pc_c, qb, Ub);
        if (owned) {
            const long long g = base0 + l + (long long)cell * sd;
#pragma unroll
            for (int v = 0; v < NV; ++v) {
                if (!a.accumulate) Gg[g + v * a.sv] = Ub[v];
                else if (EARLY && idx == (int)threadIdx.x) Gg[g + v * a.sv] = eg[v] + Ub[v];
                else Gg[g + v * a.sv] += Ub[v];
            }
        } else {
            const long long i = ix0 + l;
            const long long line = DIR == 0 ? ((long long)k * a.n[1] + j)
                                            : (DIR == 1 ? ((long long)k * a.n[0] + i) : ((long long)j * a.n[0] + i));
            const int slot = gl ? (-cell - 1) : (3 + cell - nd);   // 0..2 left (-1,-2,-3), 3..5 right
#pragma unroll
            for (int v = 0; v < NV; ++v) {
                ghost[(line * 6 + slot) * NV + v] = Ub[v];
            }
        }
    }
    return any_weno;
}

// Pass 0: one CTA per tile; a tile with a WENO face appends itself to the
// list.
template <typename T, int DIM, int DIR>
__global__ void __launch_bounds__(VjpTile<T, DIM, DIR>::NT) k_vjp(VjpArgs a)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const unsigned int lines = vjp_tile<T, DIM, DIR>(a, blockIdx.x, blockIdx.y, blockIdx.z, smem_raw);
    if (lines != 0u && threadIdx.x == 0)
        a.weno_tiles[atomicAdd(a.n_weno_tiles, 1)] =
            make_int2(blockIdx.x + a.tiles[0] * (blockIdx.y + a.tiles[1] * blockIdx.z), (int)lines);
}

// Shared memory of pass 1: one line of a tile.
template <typename T, int DIM, int DIR>
struct VjpWenoSmem {
    static constexpr int SEG = VjpTile<T, DIM, DIR>::SEG;
    static constexpr int NF = SEG + 5, NC = SEG + 10;
    static constexpr int NV = DIM + 2, NQ = CellLayout<DIM>::NQ, NX = 4;   // record, then 1/sqrt(rho), 1/c, p, c
    static constexpr int QC = 12, QB = 24;    // WENO faces per chunk, per batch
    static constexpr int NUF = 2 * NV, NRB = DIM + 2;
    // face data: Roe state, detector difference and its projection, flux
    // cotangent and its projection, splitting speeds
    static constexpr int U = 0, C = DIM, IC = DIM + 1, H = DIM + 2, B1 = DIM + 3, HQ2 = DIM + 4, RT = DIM + 5,
                         IRT2 = DIM + 6, DU = DIM + 7, W = DU + NV, PHI = W + NV, WCB = PHI + NV, AL = WCB + NV,
                         NFD = AL + 3;
    // sums over a face: bars of u, 1/c, b1, |u|^2/2 and of the three speeds,
    // then the bars of lambda^s and the reconstructed values of the fields
    static constexpr int NPB = DIM + 6, NFS = NPB + 2 * NV;
    static constexpr size_t cells = (size_t)NC * (NQ + NX + NV);
    static constexpr size_t faces = (size_t)NF * NFD + (size_t)QB * (6 * NUF + NFS + NV + 2 * NRB + 3);
    static constexpr size_t chunk = (size_t)QC * (NV * 2 * 6 + NV * 2 * 2 + 6 * NPB);
    static constexpr size_t bytes = sizeof(T) * (cells + faces + chunk) + sizeof(int) * 2 * (size_t)NF;
};
constexpr int kVjpWenoThreads = 128;

// The WENO faces of one line of a tile: line l of tile (bx, by, bz).
//
// A face's reverse is about 3500 FP64 instructions.  With one thread per face
// (255 registers and spills) a tile's dozen WENO faces filled a dozen lanes
// of two warps; here one lane takes a (face, cell) of the projections and
// their adjoints and a (face, field, sign) of the reconstruction's, in chunks
// of QC queued faces, and one lane per face the rest.  The faces go in
// batches of QB, each gathered into the bars that a thread keeps for its cell,
// so that three CTAs fit an SM (two with room for all 64 faces: 2.91 ms); few
// lines have more than one batch.  Ragged 121x97x113 box
// in FP64 with a slab across z: pass 1 of the z direction 11.76 -> 2.31 ms.
template <typename T, int DIM, int DIR>
__device__ __forceinline__ void vjp_weno_line(const VjpArgs& a, int bx, int by, int bz, int l, unsigned char* smem_raw)
{
    using CL = CellLayout<DIM>;
    using PL = PrimLayout<DIM>;
    using SM = VjpWenoSmem<T, DIM, DIR>;
    constexpr int NV = SM::NV, NQ = SM::NQ, NX = SM::NX, SEG = SM::SEG, NF = SM::NF, NC = SM::NC;
    constexpr int QC = SM::QC, QB = SM::QB, NUF = SM::NUF, NRB = SM::NRB, NFD = SM::NFD, NFS = SM::NFS, NPB = SM::NPB;
    constexpr int NT = kVjpWenoThreads, LINES = VjpTile<T, DIM, DIR>::LINES, LAST = NV - 1;
    T* cq = reinterpret_cast<T*>(smem_raw);   // [NQ + NX][NC]
    T* wq = cq + (NQ + NX) * NC;              // [NV][NC] cotangent
    T* FD = wq + NV * NC;                     // [NF][NFD]
    T* UF = FD + NF * NFD;                    // [QB][6][NUF] projections of U and F, then their bars
    T* FS = UF + QB * 6 * NUF;                // [QB][NFS]
    T* DB = FS + QB * NFS;                    // [QB][NV] bars of the detector difference
    T* RB = DB + QB * NV;                     // [QB][2][NRB] Roe-field bars of cells 2 and 3
    T* SP = RB + QB * 2 * NRB;                // [QB][3] speed bars
    T* XB = SP + QB * 3;                      // [QC][NV][2][6] bars of f+-
    T* LF = XB + QC * NV * 2 * 6;             // [QC][NV][2][2] bar of lambda^s, reconstructed value
    T* PB = LF + QC * NV * 2 * 2;             // [QC][6][NPB] per-cell parts of the face sums
    int* SL = reinterpret_cast<int*>(PB + QC * 6 * NPB);   // [NF] slots attaining the speeds
    int* queue = SL + NF;
    __shared__ int wcount[NT / 32];
    constexpr int SKIP = 1 << 12;             // no WENO face; otherwise its place in the queue from bit 13 on
    static_assert(NF <= NT, "one face per thread");

    const int nd = a.n[DIR], c0 = bx * SEG;
    int ix = 0, j = 0, k = 0;
    if (DIR == 0) { j = by; k = bz; }
    else if (DIR == 1) { ix = by * LINES + l; k = bz; }
    else { ix = by * LINES + l; j = bz; }
    const long long sd = DIR == 0 ? 1LL : (DIR == 1 ? a.sy : a.sz);
    const long long base = a.off0 + (long long)ix + (long long)j * a.sy + (long long)k * a.sz;
    const int line = DIR == 0 ? j : ix;   // in-plane index for the boundary conditions
    const T* Ug = reinterpret_cast<const T*>(a.U);
    const T* Wg = reinterpret_cast<const T*>(a.W);
    const T gamma = pick<T>(a.gamma, a.gamma_f), gm1 = gamma - T(1);

    // ---- cells c0 - 5 .. c0 + SEG + 4 that exist
    for (int p = threadIdx.x; p < NC; p += NT) {
        const int cell = c0 - 5 + p;
        const bool inside = cell >= 0 && cell < nd;
#pragma unroll
        for (int v = 0; v < NV; ++v) wq[v * NC + p] = inside ? Wg[base + (long long)cell * sd + v * a.sv] : T(0);
        if (cell >= -3 && cell <= nd + 2) {
            T U[NV], q[NQ], inv[2], P[PL::NP];
            stage_cell<T, DIM, DIR>(a.bc, Ug, base, line, cell, nd, U);
            cell_prims<T, DIM>(U, gamma, gm1, P, inv);
            cell_record<T, DIM, DIR>(U, P, q);
#pragma unroll
            for (int kk = 0; kk < NQ; ++kk) cq[kk * NC + p] = q[kk];
            cq[NQ * NC + p] = inv[0];
            cq[(NQ + 1) * NC + p] = inv[1];
            cq[(NQ + 2) * NC + p] = P[PL::P];
            cq[(NQ + 3) * NC + p] = P[PL::C];
        }
    }
    __syncthreads();

    // ---- WENO faces: the forward quantities of the whole face
    const T lam_k = pick<T>(a.lam_k, a.lam_k_f), eps = pick<T>(a.eps, a.eps_f);
    const T inv_dx = pick<T>(a.inv_dx, a.inv_dx_f), slim = pick<T>(a.slim, a.slim_f);
    const int myf = threadIdx.x;
    int slots = SKIP;
    auto face_data = [&](int f) {
        const int face = c0 - 2 + f;
        if (f >= NF || face < 0 || face > nd) return;
        auto rec = [&](int m, int kk) -> T { return cq[kk * NC + f + m]; };
        auto ga = [&](int kk) -> T { return rec(2, kk); };
        auto gb = [&](int kk) -> T { return rec(3, kk); };
        const Roe<T, DIM> r = roe_state<T, DIM>(ga, gb, gm1);
        T dU[NV], w[NV];
#pragma unroll
        for (int v = 0; v < NV; ++v) {
            const int kk = CL::U + v;
            dU[v] = fmaT(T(10), rec(2, kk) - rec(3, kk), fmaT(T(5), rec(4, kk) - rec(1, kk), rec(0, kk) - rec(5, kk)));
        }
        proj_all<T, DIM, DIR>(r, dU, w);
        const T lim = slim * r.rt;
        bool smooth = a.hybrid != 0;
        if (sizeof(T) == 8 && a.fx) {
            // the flag is pass 0's; the weights keep the FP64 form of the
            // detector (their derivative amplifies its rounding where a
            // field's own data are smooth)
            T dx[NV], wx[NV];
#pragma unroll
            for (int v = 0; v < NV; ++v) {
                const int kk = CL::U + v;
                const double x[6] = {rec(0, kk), rec(1, kk), rec(2, kk), rec(3, kk), rec(4, kk), rec(5, kk)};
                dx[v] = T(fx_detector(x));
            }
            proj_all<T, DIM, DIR>(r, dx, wx);
#pragma unroll
            for (int s = 0; s < NV; ++s) smooth = smooth && abs_lt(wx[s], lim);
        } else {
#pragma unroll
            for (int s = 0; s < NV; ++s) smooth = smooth && abs_lt(w[s], lim);
        }
        if (smooth) return;   // pass 0 took this face
        T am = rec(0, CL::LM), a0 = rec(0, CL::L0), ap = rec(0, CL::LP);
        int im = 0, i0 = 0, ip = 0;
#pragma unroll
        for (int m = 1; m < 6; ++m) {
            const T xm = rec(m, CL::LM), x0 = rec(m, CL::L0), xp = rec(m, CL::LP);
            if (lt_nn(am, xm)) { am = xm; im = m; }
            if (lt_nn(a0, x0)) { a0 = x0; i0 = m; }
            if (lt_nn(ap, xp)) { ap = xp; ip = m; }
        }
        slots = im | (i0 << 4) | (ip << 8);
        T* fd = FD + f * NFD;
#pragma unroll
        for (int kk = 0; kk < DIM; ++kk) fd[SM::U + kk] = r.u[kk];
        fd[SM::C] = r.c; fd[SM::IC] = r.ic; fd[SM::H] = r.H; fd[SM::B1] = r.b1; fd[SM::HQ2] = r.hq2; fd[SM::RT] = r.rt;
        fd[SM::IRT2] = T(1) / (r.rt * r.rt);
        fd[SM::AL] = am; fd[SM::AL + 1] = a0; fd[SM::AL + 2] = ap;
        // cotangent of the face flux, (w_right - w_left) / dx, and R^T of it
        T phi[NV];
#pragma unroll
        for (int v = 0; v < NV; ++v) {
            phi[v] = (wq[v * NC + f + 3] - wq[v * NC + f + 2]) * inv_dx;
            fd[SM::PHI + v] = phi[v];
            fd[SM::DU + v] = dU[v];
            fd[SM::W + v] = w[v];
        }
        T sumb = phi[0];
#pragma unroll
        for (int kk = 0; kk < DIM; ++kk) sumb = fmaT(phi[1 + kk], r.u[kk], sumb);
        const T difb = fmaT(phi[LAST], r.u[DIR], phi[1 + DIR]) * r.c, eh = fmaT(phi[LAST], r.H, sumb);
        fd[SM::WCB] = eh - difb;
        fd[SM::WCB + 1] = fmaT(phi[LAST], r.hq2, sumb);
        int s = 2;
#pragma unroll
        for (int kk = 0; kk < DIM; ++kk) {
            if (kk == DIR) continue;
            fd[SM::WCB + s] = fmaT(phi[LAST], r.u[kk], phi[1 + kk]);
            ++s;
        }
        fd[SM::WCB + LAST] = eh + difb;
    };
    face_data(myf);
    // the queue in face order
    const unsigned int mine = __ballot_sync(0xffffffffu, slots != SKIP);
    if ((threadIdx.x & 31) == 0) wcount[threadIdx.x >> 5] = __popc(mine);
    __syncthreads();
    int nq = 0, pos = __popc(mine & ((1u << (threadIdx.x & 31)) - 1u));
#pragma unroll
    for (int w = 0; w < NT / 32; ++w) {
        if (w < (int)(threadIdx.x >> 5)) pos += wcount[w];
        nq += wcount[w];
    }
    if (slots != SKIP) queue[pos] = myf;
    if (myf < NF) SL[myf] = slots == SKIP ? SKIP : slots | (pos << 13);
    __syncthreads();

    auto load_roe = [&](const T* fd, Roe<T, DIM>& r) {
#pragma unroll
        for (int kk = 0; kk < DIM; ++kk) r.u[kk] = fd[SM::U + kk];
        r.c = fd[SM::C]; r.ic = fd[SM::IC]; r.H = fd[SM::H]; r.b1 = fd[SM::B1]; r.hq2 = fd[SM::HQ2]; r.rt = fd[SM::RT];
    };
    // the cell whose bars this thread gathers
    static_assert(SEG + 6 <= NT, "one cell per thread");
    const bool first = c0 == 0, last = c0 + SEG >= nd;
    const int cell = c0 - 3 + (int)threadIdx.x;
    const bool owned = cell >= c0 && cell < c0 + SEG && cell < nd;
    const bool gl = first && cell < 0 && cell >= -3;
    const bool gr = last && cell >= nd && cell <= nd + 2;
    const bool gathers = (int)threadIdx.x < SEG + 6 && (owned || gl || gr);
    bool touched = false;
    T qb[NQ];
#pragma unroll
    for (int kk = 0; kk < NQ; ++kk) qb[kk] = T(0);
    for (int b0 = 0; b0 < nq; b0 += QB) {
        const int qn = nq - b0 < QB ? nq : b0 + QB;
        for (int q0 = b0; q0 < qn; q0 += QC) {
            const int qc = qn - q0 < QC ? qn - q0 : QC;
            // projections of U_m and F_m (Eq. eqchara)
            for (int it = threadIdx.x; it < qc * 6; it += NT) {
                const int f = queue[q0 + it / 6], m = it % 6, e = q0 - b0 + it / 6;
                Roe<T, DIM> r;
                load_roe(FD + f * NFD, r);
                T xu[NV], xf[NV], vv[NV], gg[NV];
#pragma unroll
                for (int v = 0; v < NV; ++v) { xu[v] = cq[(CL::U + v) * NC + f + m]; xf[v] = cq[(CL::F + v) * NC + f + m]; }
                proj_all<T, DIM, DIR>(r, xu, vv);
                proj_all<T, DIM, DIR>(r, xf, gg);
                T* uf = UF + (e * 6 + m) * NUF;
#pragma unroll
                for (int s = 0; s < NV; ++s) { uf[s] = vv[s]; uf[NV + s] = gg[s]; }
            }
            __syncthreads();
            // reconstructions and their reverse; the minus part on the mirrored
            // stencil m = 5 .. 1
            for (int it = threadIdx.x; it < qc * NV * 2; it += NT) {
                const int q = it / (2 * NV), rem = it - q * 2 * NV, s = rem >> 1, sg = rem & 1;
                const int f = queue[q0 + q];
                const T* fd = FD + f * NFD;
                const T al = fd[SM::AL + (s == 0 ? 0 : (s == LAST ? 2 : 1))];
                const T ws = fd[SM::W + s], lam = lam_k * (ws * ws) * fd[SM::IRT2];
                const T ha = sg ? T(-0.5) * al : T(0.5) * al;
                T x[5], xb[5], lb;
#pragma unroll
                for (int i = 0; i < 5; ++i) {
                    const T* uf = UF + ((q0 - b0 + q) * 6 + (sg ? 5 - i : i)) * NUF + s;
                    x[i] = fmaT(ha, uf[0], T(0.5) * uf[NV]);
                }
                const T val = recon_adj<T>(x[0], x[1], x[2], x[3], x[4], lam, eps, fd[SM::WCB + s], xb, lb);
                T* o = XB + ((q * NV + s) * 2 + sg) * 6;
#pragma unroll
                for (int i = 0; i < 5; ++i) o[sg ? 5 - i : i] = xb[i];
                o[sg ? 0 : 5] = T(0);
                LF[((q * NV + s) * 2 + sg) * 2] = lb;
                LF[((q * NV + s) * 2 + sg) * 2 + 1] = val;
            }
            __syncthreads();
            // splitting and projections in reverse, per stencil cell
            for (int it = threadIdx.x; it < qc * 6; it += NT) {
                const int q = it / 6, m = it - q * 6, f = queue[q0 + q];
                const T* fd = FD + f * NFD;
                Roe<T, DIM> r;
                load_roe(fd, r);
                T* uf = UF + ((q0 - b0 + q) * 6 + m) * NUF;
                T vb[NV], gb[NV], alb[3] = {T(0), T(0), T(0)};
#pragma unroll
                for (int s = 0; s < NV; ++s) {
                    const T fp = XB[((q * NV + s) * 2) * 6 + m], fm = XB[((q * NV + s) * 2 + 1) * 6 + m];
                    const int as = s == 0 ? 0 : (s == LAST ? 2 : 1);
                    const T d = T(0.5) * (fp - fm);
                    gb[s] = T(0.5) * (fp + fm);
                    vb[s] = fd[SM::AL + as] * d;
                    alb[as] = fmaT(uf[s], d, alb[as]);
                }
                RoeBar<T, DIM> rb;
                zero(rb);
                T x[NV], xb[NV];
#pragma unroll
                for (int h = 0; h < 2; ++h) {
#pragma unroll
                    for (int v = 0; v < NV; ++v) { x[v] = cq[((h ? CL::F : CL::U) + v) * NC + f + m]; xb[v] = T(0); }
                    proj_all_adj<T, DIM, DIR>(r, x, h ? gb : vb, xb, rb);
#pragma unroll
                    for (int v = 0; v < NV; ++v) uf[h * NV + v] = xb[v];
                }
                T* o = PB + it * NPB;
#pragma unroll
                for (int kk = 0; kk < DIM; ++kk) o[kk] = rb.u[kk];
                o[DIM] = rb.ic; o[DIM + 1] = rb.b1; o[DIM + 2] = rb.hq2;
#pragma unroll
                for (int i = 0; i < 3; ++i) o[DIM + 3 + i] = alb[i];
            }
            __syncthreads();
            // sums over the cells and over the signs
            for (int it = threadIdx.x; it < qc * NFS; it += NT) {
                const int q = it / NFS, c = it - q * NFS;
                T sum;
                if (c < NPB) {
                    const T* o = PB + q * 6 * NPB + c;
                    sum = o[0];
#pragma unroll
                    for (int m = 1; m < 6; ++m) sum += o[m * NPB];
                } else {
                    const int s = (c - NPB) % NV, w = (c - NPB) / NV;
                    const T* o = LF + (q * NV + s) * 4 + w;
                    sum = o[0] + o[2];
                }
                FS[(q0 - b0 + q) * NFS + c] = sum;
            }
        }
        __syncthreads();

        // ---- per face: weights' parameter, detector, back-projection and Roe average in reverse
        for (int e = threadIdx.x; e < qn - b0; e += NT) {
            const int f = queue[b0 + e];
            const T *fd = FD + f * NFD, *fs = FS + e * NFS, *lb = fs + NPB, *wch = lb + NV;
            Roe<T, DIM> r;
            load_roe(fd, r);
            RoeBar<T, DIM> rb;
            zero(rb);
            const T sum = wch[0] + wch[1] + wch[LAST], dif = wch[LAST] - wch[0], oE = fd[SM::PHI + LAST];
#pragma unroll
            for (int kk = 0; kk < DIM; ++kk) rb.u[kk] = fmaT(fd[SM::PHI + 1 + kk], sum, fs[kk]);
            rb.c = fmaT(oE, r.u[DIR], fd[SM::PHI + 1 + DIR]) * dif;
            rb.u[DIR] = fmaT(oE * r.c, dif, rb.u[DIR]);
            int s = 2;
#pragma unroll
            for (int kk = 0; kk < DIM; ++kk) {
                if (kk == DIR) continue;
                rb.u[kk] = fmaT(oE, wch[s], rb.u[kk]);
                ++s;
            }
            rb.H = oE * (wch[0] + wch[LAST]);
            rb.ic = fs[DIM];
            rb.b1 = fs[DIM + 1];
            rb.hq2 = fmaT(oE, wch[1], fs[DIM + 2]);
            // lam = c w^2 / (3600 rt^2)
            const T irt2 = fd[SM::IRT2], irt = irt2 * r.rt;
            T wb[NV], dUb[NV], dU[NV];
#pragma unroll
            for (int v = 0; v < NV; ++v) {
                const T w = fd[SM::W + v], lw = lam_k * w * irt2;
                wb[v] = lb[v] * (lw + lw);
                rb.rt = fmaT(lb[v], T(-2) * (lw * w) * irt, rb.rt);
                dU[v] = fd[SM::DU + v];
                dUb[v] = T(0);
            }
            proj_all_adj<T, DIM, DIR>(r, dU, wb, dUb, rb);
#pragma unroll
            for (int v = 0; v < NV; ++v) DB[e * NV + v] = dUb[v];
#pragma unroll
            for (int i = 0; i < 3; ++i) SP[e * 3 + i] = fs[DIM + 3 + i];
            T* RBf = RB + e * 2 * NRB;
            T ra[NRB], rbb[NRB];
#pragma unroll
            for (int kk = 0; kk < NRB; ++kk) ra[kk] = rbb[kk] = T(0);
            roe_adj<T, DIM>([&](int kk) -> T { return cq[kk * NC + f + 2]; }, [&](int kk) -> T { return cq[kk * NC + f + 3]; },
                            gamma, r, rb, ra, rbb);
#pragma unroll
            for (int kk = 0; kk < NRB; ++kk) { RBf[kk] = ra[kk]; RBf[NRB + kk] = rbb[kk]; }
        }
        __syncthreads();

        // ---- gather per cell, as in pass 0, faces in increasing order
        if (gathers) {
            constexpr T cd[6] = {T(1), T(-5), T(10), T(-10), T(5), T(-1)};
#pragma unroll
            for (int m = 5; m >= 0; --m) {
                const int f = cell - m + 3 - (c0 - 2);
                if (f < 0 || f >= NF) continue;
                const int sl = SL[f];
                const int e = (sl >> 13) - b0;
                if ((sl & SKIP) || e < 0 || e >= QB) continue;
                touched = true;
                const T* uf = UF + (e * 6 + m) * NUF;
#pragma unroll
                for (int v = 0; v < NV; ++v) {
                    qb[CL::U + v] += fmaT(cd[m], DB[e * NV + v], uf[v]);
                    qb[CL::F + v] += uf[NV + v];
                }
                if (m == 2 || m == 3) {
                    const T* rbp = RB + (e * 2 + (m - 2)) * NRB;
#pragma unroll
                    for (int kk = 0; kk < NRB; ++kk) qb[CL::SU + kk] += rbp[kk];
                }
                if ((sl & 15) == m) qb[CL::LM] += SP[e * 3 + 0];
                if (((sl >> 4) & 15) == m) qb[CL::L0] += SP[e * 3 + 1];
                if (((sl >> 8) & 15) == m) qb[CL::LP] += SP[e * 3 + 2];
            }
        }
        __syncthreads();   // the next batch reuses shared memory
    }
    T* Gg = reinterpret_cast<T*>(a.G);
    T* ghost = reinterpret_cast<T*>(a.ghost);
    if (touched) {
        const int pc = cell - (c0 - 5);
        T U[NV], Ub[NV];
#pragma unroll
        for (int v = 0; v < NV; ++v) U[v] = cq[(CL::U + v) * NC + pc];
        cell_adj<T, DIM, DIR>(U, gamma, cq[NQ * NC + pc], cq[(NQ + 1) * NC + pc], cq[(NQ + 2) * NC + pc],
                              cq[(NQ + 3) * NC + pc], qb, Ub);
        if (owned) {
            const long long g = base + (long long)cell * sd;
#pragma unroll
            for (int v = 0; v < NV; ++v) Gg[g + v * a.sv] += Ub[v];
        } else {
            const long long ln = DIR == 0 ? ((long long)k * a.n[1] + j)
                                          : (DIR == 1 ? ((long long)k * a.n[0] + ix) : ((long long)j * a.n[0] + ix));
            const int slot = gl ? (-cell - 1) : (3 + cell - nd);
#pragma unroll
            for (int v = 0; v < NV; ++v) ghost[(ln * 6 + slot) * NV + v] += Ub[v];
        }
    }
    __syncthreads();   // shared memory is reused by the next line
}

// Pass 1: a grid of resident CTAs takes the listed tiles in turn (each line
// writes only its own cells and ghost slots, so the order in which they are
// taken does not change the result).
template <typename T, int DIM, int DIR>
__global__ void __launch_bounds__(kVjpWenoThreads) k_vjp_weno(VjpArgs a)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    constexpr int LINES = VjpTile<T, DIM, DIR>::LINES;
    const long long n = (long long)*a.n_weno_tiles * LINES;
    for (long long it = blockIdx.x; it < n; it += gridDim.x) {
        const int2 t = a.weno_tiles[it / LINES];
        const int l = (int)(it % LINES);
        if (!((t.y >> l) & 1)) continue;
        const int bx = t.x % a.tiles[0], byz = t.x / a.tiles[0];
        vjp_weno_line<T, DIM, DIR>(a, bx, byz % a.tiles[1], byz / a.tiles[1], l, smem_raw);
    }
}

// ghost-cell gradients back to the interior cells they copy (the adjoint of
// the boundary conditions); fixed inflow states receive nothing
template <typename T, int DIM>
__global__ void k_ghost_adj(GhostArgs a, const void* ghost_, void* G_)
{
    constexpr int NV = DIM + 2;
    const int d = a.dir;
    const int nd = a.n[d];
    int e0, e1;
    if (d == 0) { e0 = a.n[1]; e1 = a.n[2]; }
    else if (d == 1) { e0 = a.n[0]; e1 = a.n[2]; }
    else { e0 = a.n[0]; e1 = a.n[1]; }
    const long long lines = (long long)e0 * e1;
    const long long sd = d == 0 ? 1LL : (d == 1 ? a.sy : a.sz);
    const T* ghost = reinterpret_cast<const T*>(ghost_);
    T* G = reinterpret_cast<T*>(G_);
    for (long long ln = blockIdx.x * (long long)blockDim.x + threadIdx.x; ln < lines;
         ln += (long long)gridDim.x * blockDim.x) {
        const int p0 = (int)(ln % e0), p1 = (int)(ln / e0);
        int i, j, k;
        if (d == 0) { i = 0; j = p0; k = p1; }
        else if (d == 1) { i = p0; j = 0; k = p1; }
        else { i = p0; j = p1; k = 0; }
        const long long base = a.off0 + (long long)i + (long long)j * a.sy + (long long)k * a.sz;
        for (int slot = 0; slot < 6; ++slot) {
            const int side = slot / 3, gl = slot % 3 + 1;
            int bc = side == 0 ? a.bc_lo : a.bc_hi;
            if (bc == BC_DMR_BOTTOM) {
                const double x = a.lo0 + (i + 0.5) * a.dx0;
                bc = x < 1.0 / 6.0 ? BC_INFLOW : BC_REFLECT;
            } else if (bc == BC_DMR_TOP || bc == BC_JET) {
                bc = BC_INFLOW;
            }
            if (bc == BC_INFLOW) continue;
            int src;
            if (bc == BC_TRANSMISSIVE) src = side == 0 ? 0 : nd - 1;
            else if (bc == BC_REFLECT) src = side == 0 ? gl - 1 : nd - gl;
            else src = side == 0 ? nd - gl : gl - 1;
            const long long g = base + (long long)src * sd;
#pragma unroll
            for (int v = 0; v < NV; ++v) {
                T val = ghost[(ln * 6 + slot) * NV + v];
                if (bc == BC_REFLECT && v == 1 + d) val = -val;
                G[g + v * a.sv] += val;
            }
        }
    }
}

}  // namespace wis
