// One tile of a 1D sweep that combines a Runge-Kutta stage: one thread per
// cell, face and output cell.
//
// The tile holds NT staged cells, their NT - 5 faces and the NT - 6 cells
// between them, so that no phase has a second, nearly empty round (with NT
// faces the five cells beyond NT cost a whole round of the per-cell
// arithmetic).  A persistent CTA chains such tiles along a line: the states of
// the next tile are loaded while this one is computed, and the base state of
// the stage is loaded before the faces, so that neither latency is exposed.
// The faces take the routines and the operand order of sweep_tile, and give
// the same bits.
#pragma once

#include "weno_kernels.cuh"

namespace wis {

template <typename T, int NT>
struct LineTile {
    static constexpr int FACES = NT - 5, SEG = NT - 6;
    static constexpr int NQ = CellLayout<1>::NQ, NV = 3, NR = FaceRec<T, 1>::NR;
    // one chunk of WENO faces gives every thread a stencil cell to project
    // and a reconstruction (both 6 per face)
    static constexpr int QC = NT / 6;
    static constexpr size_t bytes =
        sizeof(T) * ((size_t)(NQ + NV + NR) * NT + (size_t)QC * NV * 2 * 6 + (size_t)QC * NV * 2) + sizeof(int) * (size_t)NT;
};

// the state that thread threadIdx.x stages for the tile at cell c0
template <typename T>
__device__ __forceinline__ void line_load(const SweepArgs& a, int c0, T (&U)[3])
{
    const int along = c0 - 3 + (int)threadIdx.x, nd = a.n[0];
    if (along < nd + 3) {
        const T* Ug = reinterpret_cast<const T*>(a.U);
        if (along >= 0 && along < nd) {
            const T* p = Ug + a.off0 + along;
#pragma unroll
            for (int v = 0; v < 3; ++v) U[v] = p[v * a.sv];
        } else {
            stage_cell<T, 1, 0>(a, Ug, a.off0, 0, along, nd, U);
        }
    }
}

// Tile of the cells c0 .. c0 + SEG - 1.  U: this thread's state (line_load);
// replaced by that of the tile at cnext (none if negative).  wenos: this
// thread's count of owned WENO faces.  Returns whether a cell this thread
// wrote is not admissible.  Ends with a barrier.
template <typename T, int NT, bool EXACTDET, bool FX>
__device__ __forceinline__ bool line_tile(const SweepArgs& a, int c0, int cnext, T dt, T (&U)[3], unsigned char* smem_raw,
                                          TileCfl<T, 1>* cfl, unsigned int& wenos)
{
    using CL = CellLayout<1>;
    using FR = FaceRec<T, 1>;
    using LT = LineTile<T, NT>;
    constexpr int NQ = CL::NQ, NV = 3;
    T* cq = reinterpret_cast<T*>(smem_raw);   // [NQ][NT] cell records
    T* fh = cq + NQ * NT;                     // [NV][NT] face fluxes
    T* fr = fh + NV * NT;                     // [NR][NT] WENO face records
    T* fpm = fr + LT::NR * NT;                // [QC][NV][2][6]
    T* res = fpm + LT::QC * NV * 2 * 6;       // [QC][NV][2]
    int* queue = reinterpret_cast<int*>(res + LT::QC * NV * 2);
    __shared__ int qcount;

    const int nd = a.n[0], i = threadIdx.x;
    const T gamma = pick<T>(a.gamma, a.gamma_f), gm1 = gamma - T(1);
    if (i == 0) qcount = 0;
    if (c0 - 3 + i < nd + 3) {
        T q[NQ];
        cell_prepare<T, 1, 0>(U, gamma, gm1, q);
#pragma unroll
        for (int k = 0; k < NQ; ++k) cq[k * NT + i] = q[k];
    }
    __syncthreads();
    if (cnext >= 0) line_load(a, cnext, U);
    const bool out = i < LT::SEG && c0 + i < nd;
    const T rka = pick<T>(a.rk_a, a.rk_a_f), rkb = pick<T>(a.rk_b, a.rk_b_f);
    T un[NV] = {T(0), T(0), T(0)};
    if (out && rka != T(0)) {
        const T* p = reinterpret_cast<const T*>(a.Un) + a.off0 + c0 + i;
#pragma unroll
        for (int v = 0; v < NV; ++v) un[v] = p[v * a.sv];
    }

    bool weno = false;
    if (i < LT::FACES && c0 + i <= nd) {
        auto ga = [&](int k) -> T { return cq[k * NT + i + 2]; };
        auto gb = [&](int k) -> T { return cq[k * NT + i + 3]; };
        const Roe<T, 1> r = roe_state<T, 1>(ga, gb, gm1);
        // Eq. eq28 without the 1/60
        T dU[NV], w[NV];
#pragma unroll
        for (int v = 0; v < NV; ++v) {
            const T* u = cq + (CL::U + v) * NT + i;
            if (FX && a.fx) {
                const double x[6] = {u[0], u[1], u[2], u[3], u[4], u[5]};
                dU[v] = T(fx_detector(x));
            } else if (EXACTDET) dU[v] = -fifth_difference(u[0], u[1], u[2], u[3], u[4], u[5]);
            else dU[v] = fmaT(T(10), u[2] - u[3], fmaT(T(5), u[4] - u[1], u[0] - u[5]));
        }
        proj_all<T, 1, 0>(r, dU, w);
        const T lim = pick<T>(a.slim, a.slim_f) * r.rt;
        int fmask = 0;
#pragma unroll
        for (int s = 0; s < NV; ++s) fmask |= abs_lt(w[s], lim) ? (1 << s) : 0;
        const bool smooth = a.hybrid != 0 && fmask == (1 << NV) - 1;
        T am, a0, ap;
        if (a.split == SPLIT_LLF) {
            const T *lm = cq + CL::LM * NT + i, *l0 = cq + CL::L0 * NT + i, *lp = cq + CL::LP * NT + i;
            am = lm[0]; a0 = l0[0]; ap = lp[0];
#pragma unroll
            for (int m = 1; m < 6; ++m) { am = max_nn(am, lm[m]); a0 = max_nn(a0, l0[m]); ap = max_nn(ap, lp[m]); }
        } else if (a.split == SPLIT_RF) {
            am = absT(r.u[0] - r.c);
            a0 = absT(r.u[0]);
            ap = absT(r.u[0] + r.c);
        } else {
            am = T(__longlong_as_double((long long)a.alpha_g[0]));
            a0 = T(__longlong_as_double((long long)a.alpha_g[1]));
            ap = T(__longlong_as_double((long long)a.alpha_g[2]));
        }
        if (smooth) {
            // Eq. linearupwind, times 60
            T Fo[NV];
#pragma unroll
            for (int v = 0; v < NV; ++v) {
                const T* f = cq + (CL::F + v) * NT + i;
                if (FX && a.fx) {
                    const double x[6] = {f[0], f[1], f[2], f[3], f[4], f[5]};
                    Fo[v] = T(fx_central_flux(x));
                } else {
                    const T f05 = f[0] + f[5], f14 = f[1] + f[4], f23 = f[2] + f[3];
                    Fo[v] = fmaT(T(37), f23, fmaT(T(-8), f14, f05));
                }
            }
            ups_dissipation_add<T, 1, 0>(r, dU, w, am, a0, ap, Fo);
#pragma unroll
            for (int v = 0; v < NV; ++v) fh[v * NT + i] = Fo[v];
        } else {
            weno = true;
            fr[FR::U * NT + i] = r.u[0];
            fr[FR::C * NT + i] = r.c;
            fr[FR::IC * NT + i] = r.ic;
            fr[FR::H * NT + i] = r.H;
            fr[FR::B1 * NT + i] = r.b1;
            fr[FR::HQ2 * NT + i] = r.hq2;
#pragma unroll
            for (int s = 0; s < NV; ++s) fr[(FR::W + s) * NT + i] = w[s];
            fr[FR::IRT2 * NT + i] = Ar<T>::rcp_f(r.rt * r.rt);
            fr[FR::AM * NT + i] = halve(am);
            fr[FR::A0 * NT + i] = halve(a0);
            fr[FR::AP * NT + i] = halve(ap);
            fr[FR::MASK * NT + i] = T(a.hybrid == 2 ? fmask : 0);
            // a face is owned by the tile left of it, the last face by the last tile
            if (i < LT::SEG || c0 + i == nd) ++wenos;
        }
    }
    const unsigned int mask = __ballot_sync(0xffffffffu, weno);
    if (mask) {
        const int lane = i & 31, leader = __ffs(mask) - 1;
        int base = 0;
        if (lane == leader) base = atomicAdd(&qcount, __popc(mask));
        base = __shfl_sync(0xffffffffu, base, leader);
        if (weno) queue[base + __popc(mask & ((1u << lane) - 1u))] = i;
    }
    __syncthreads();
    const int nq = qcount;
    if (nq > 0) {
        weno_queue<T, 1, 0, NT, NT, LT::QC, NT>(a, nq, cq, fh, fr, fpm, res, queue,
                                                [](int f, int m) -> int { return f + m; });
        __syncthreads();
    }

    bool bad = false;
    if (out) {
        const T inv_dx = pick<T>(a.inv_dx * (1.0 / 60.0), a.inv_dx_f);
        T* p = reinterpret_cast<T*>(a.out) + a.off0 + c0 + i;
        T nu[NV];
#pragma unroll
        for (int v = 0; v < NV; ++v) {
            const T rv = (fh[v * NT + i] - fh[v * NT + i + 1]) * inv_dx;
            T val = rkb * fmaT(dt, rv, cq[(CL::U + v) * NT + i + 3]);
            if (rka != T(0)) val = fmaT(rka, un[v], val);
            nu[v] = val;
            p[v * a.sv] = val;
        }
        // admissibility: rho > 0, p > 0  <=>  2 rho E > |m|^2, finite
        const T m2 = fmaT(nu[1], nu[1], T(0));
        const T chk = T(2) * nu[0] * nu[2] - m2;
        if (!(nu[0] > T(0)) || !(chk > T(0)) || !isfinite(chk)) bad = true;
        if (cfl != nullptr) {
            T sp;
            if (!cell_speed<T, 1>(nu, gamma, cfl->inv_dx, sp)) cfl->bad = true;
            else cfl->smax = max_nn(cfl->smax, sp);
        }
    }
    __syncthreads();
    return bad;
}

}  // namespace wis
