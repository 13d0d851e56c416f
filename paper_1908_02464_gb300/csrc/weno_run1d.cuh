// Many RK3 steps of one small 1D problem in one launch.
//
//   k_run1d   a cluster of up to 16 CTAs; each holds a segment of the line in
//             shared memory for the whole launch.  Per stage (Sec. 4) it
//             stages its cells' records (the three cells beyond each end come
//             from its neighbours' shared memory or the boundary conditions),
//             computes its faces and updates its cells; one cluster barrier
//             ends the stage.  The CFL maximum of a finished step and the
//             admissibility flags are pushed into every CTA's shared memory
//             before that barrier, so every CTA takes the same step.
//
// What bounds it: latency.  A few hundred cells fill neither pipe; as a chain
// of six kernels per step (CFL, dt, three sweeps, bookkeeping) a step of 200
// cells in FP64 took 49 us and one of 400 cells in FP32 20 us, spread over
// launches, global-memory round trips and one SM's FP64 pipe (a WENO face
// costs ten times a linear one, and a 127-cell tile holds them all).  Sixteen
// short segments divide that arithmetic over sixteen SMs and exchange it in
// shared memory: 200 cells in FP64 31.8 us a step, 400 in FP32 7.9 us.  What
// is left in FP64 is one warp's chain of about 270 instructions a stage, one
// per 64 clocks and SM quarter.  The faces take the routines and the operand order of
// sweep_tile, and give the same bits.
#pragma once

#include <cooperative_groups.h>

#include "weno_kernels.cuh"

namespace wis {

struct Run1DArgs {
    SweepArgs a;            // constants and boundary conditions
    void* buf[3];           // state buffers; a step moves the state to the next one
    int nsteps;             // at most
    double cfl, smax_floor;
};

constexpr int kRun1DThreads = 128;
// Cells of one CTA, which end where the kernels per step are as fast.  FP64, one
// round of faces: 40 steps of a line of 2000 cells 54 us each against 67 (27
// against 35 on a smooth state), of 2500, which took a second round, 66 against
// 66 (38 against 35), of 4000 70 against 57.  FP32, four rounds: 14 us against 19
// at 4000 cells, 18 against 19 at 8000 (calls of one step 51 against 46 there,
// 42 against 46 at 4000).
template <typename T> constexpr int run1d_cells() { return sizeof(T) == 8 ? 128 : 512; }
// the fewest cells worth a CTA of its own
constexpr int kRun1DMinCells = 12;
constexpr int kRun1DMaxCluster = 16;

template <typename T>
struct Run1DSmem {
    static constexpr int M = run1d_cells<T>(), NV = 3, NQ = CellLayout<1>::NQ, NR = FaceRec<T, 1>::NR;
    static constexpr int NCELL = M + 6, NFACE = M + 1;
    static constexpr int QC = kRun1DThreads / 6;
    static constexpr size_t bytes = sizeof(T) * ((size_t)3 * NV * M + (size_t)NQ * NCELL + (size_t)(NV + NR) * NFACE +
                                                 (size_t)QC * NV * 2 * 6 + (size_t)QC * NV * 2) +
                                    sizeof(int) * (size_t)NFACE;
};

// by every thread of the CTA; the aligned forms want a converged warp
__device__ __forceinline__ void cluster_arrive()
{
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait()
{
    __syncwarp();
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_barrier()
{
    cluster_arrive();
    cluster_wait();
}

template <typename T, bool EXACTDET>
__global__ void __launch_bounds__(kRun1DThreads) k_run1d(Run1DArgs r)
{
    using CL = CellLayout<1>;
    using FR = FaceRec<T, 1>;
    using SM = Run1DSmem<T>;
    constexpr int NT = kRun1DThreads, NV = 3, NQ = SM::NQ, M = SM::M, NCELL = SM::NCELL, NFACE = SM::NFACE;
    namespace cg = cooperative_groups;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T* ub = reinterpret_cast<T*>(smem_raw);   // [3][NV][M] states: current, other, second stage
    T* cq = ub + 3 * NV * M;                  // [NQ][NCELL] cell records
    T* fh = cq + NQ * NCELL;                  // [NV][NFACE] face fluxes
    T* fr = fh + NV * NFACE;                  // [NR][NFACE] WENO face records
    T* fpm = fr + SM::NR * NFACE;
    T* res = fpm + SM::QC * NV * 2 * 6;
    int* queue = reinterpret_cast<int*>(res + SM::QC * NV * 2);
    // what every CTA of the cluster tells the others at the end of a stage,
    // in two turns: a CTA may end the next stage before another has read this
    __shared__ double x_smax[2][kRun1DMaxCluster];
    __shared__ int x_bad[2][kRun1DMaxCluster];
    __shared__ double s_dt;
    __shared__ T s_red[NT / 32];
    __shared__ int s_stop, s_bad, qcount;

    cg::cluster_group cluster = cg::this_cluster();
    const int C = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
    const SweepArgs& a = r.a;
    DevTime* tm = a.tm;
    const int tid = threadIdx.x, lane = tid & 31;
    const int n = a.n[0];
    const int lo = (int)((long long)rank * n / C), hi = (int)((long long)(rank + 1) * n / C), m = hi - lo;
    const T gamma = pick<T>(a.gamma, a.gamma_f), gm1 = gamma - T(1);
    const T inv_dx = pick<T>(a.inv_dx * (1.0 / 60.0), a.inv_dx_f);
    const T inv_dx1[1] = {T(a.inv_dx)};
    const T slim = pick<T>(a.slim, a.slim_f);
    const long long steps0 = tm->steps;
    const int phase0 = tm->phase;
    const double t_end = tm->t_end;
    const bool live = tm->status == 0;
    // time of the current state, kept by the last thread (its staging share is
    // the smallest), which takes the steps
    double t = tm->t;
    int clipped = 0, status = 0, turn = 0;
    unsigned int wenos = 0;

    // ends a stage: this CTA's admissibility and CFL maximum to all CTAs
    auto tell = [&](bool bad, bool cbad, T smax) {
        const T mw = warp_max_nn(smax);
        if (lane == 0) s_red[tid >> 5] = mw;
        if (bad || cbad) atomicOr(&s_bad, (bad ? 1 : 0) | (cbad ? 2 : 0));
        __syncthreads();
        if (tid < C) {
            T mx = s_red[0];
#pragma unroll
            for (int w = 1; w < NT / 32; ++w) mx = max_nn(mx, s_red[w]);
            *cluster.map_shared_rank(&x_smax[turn][rank], tid) = (double)mx;
            *cluster.map_shared_rank(&x_bad[turn][rank], tid) = s_bad;
        }
        cluster_barrier();
    };

    // The state, and its CFL wave speeds.  A CTA may store to another's shared
    // memory (the first tell) only once that CTA has started: every CTA says so
    // here, and the loads of the state cover the wait.
    cluster_arrive();
    if (tid == 0) s_bad = 0;
    __syncthreads();
    {
        const T* p = reinterpret_cast<const T*>(r.buf[phase0]) + a.off0 + lo;
        T smax = T(0);
        bool cbad = false;
        for (int i = tid; i < m; i += NT) {
            T u[NV], sp;
#pragma unroll
            for (int v = 0; v < NV; ++v) { u[v] = p[i + v * a.sv]; ub[v * M + i] = u[v]; }
            if (!cell_speed<T, 1>(u, gamma, inv_dx1, sp)) cbad = true;
            else smax = max_nn(smax, sp);
        }
        cluster_wait();
        tell(false, cbad, smax);
    }

    int cur = 0, done = 0;
    while (live && done < r.nsteps) {
        T dt = T(0);
        bool failed = false;
#pragma unroll 1
        for (int st = 0; st < 3; ++st) {
            const int in = st == 0 ? cur : (st == 1 ? 1 - cur : 2), out = st == 1 ? 2 : 1 - cur;
            const T* Uin = ub + in * NV * M;
            // cell records of lo - 3 .. hi + 2
            for (int idx = tid; idx < m + 6; idx += NT) {
                long long g = 0;
                bool flip = false;
                const int fixed = cell_source<0>(a, 0, 0, lo - 3 + idx, n, g, flip);
                T U[NV], q[NQ];
                if (fixed >= 0) {
#pragma unroll
                    for (int v = 0; v < NV; ++v) U[v] = pick<T>(a.bc_state[fixed][v], a.bc_state_f[fixed][v]);
                } else {
                    const int c = (int)g;
                    const T* src = Uin;
                    int first = lo;
                    if (c < lo || c >= hi) {
                        // a neighbour's cell, or across a periodic end
                        const int own = c < lo ? (lo - c <= 3 ? rank - 1 : 0) : (c - hi < 3 ? rank + 1 : C - 1);
                        src = cluster.map_shared_rank(const_cast<T*>(Uin), own);
                        first = (int)((long long)own * n / C);
                    }
#pragma unroll
                    for (int v = 0; v < NV; ++v) U[v] = src[v * M + c - first];
                    if (flip) U[1] = -U[1];
                }
                cell_prepare<T, 1, 0>(U, gamma, gm1, q);
#pragma unroll
                for (int k = 0; k < NQ; ++k) cq[k * NCELL + idx] = q[k];
            }
            if (tid == 0) { qcount = 0; s_bad = 0; }
            __syncthreads();
            if (st == 0 && tid >= NT - 32) {
                // The step, taken by the last warp (short lines give it no
                // faces) from the same numbers in every CTA; the other warps
                // go on and need it at the update
                const int kk = lane < C ? lane : 0;
                const int bad = __reduce_or_sync(0xffffffffu, (unsigned int)x_bad[turn][kk]);
                const double smax = warp_max_nn(max_nn(r.smax_floor, x_smax[turn][kk]));
                if (lane == 31) {
                    double d = 0.0;
                    if (bad & 2) status = 1;
                    else d = cfl_step(r.cfl, smax, t, t_end, &clipped);
                    s_dt = d;
                    s_stop = !(d > 0.0);
                }
            }
            unsigned int stage_wenos = 0;
            // faces lo - 1/2 .. hi - 1/2
            for (int f0 = 0; f0 < m + 1; f0 += NT) {
                const int f = f0 + tid;
                bool weno = false;
                if (f < m + 1) {
                    auto ga = [&](int k) -> T { return cq[k * NCELL + f + 2]; };
                    auto gb = [&](int k) -> T { return cq[k * NCELL + f + 3]; };
                    const Roe<T, 1> ro = roe_state<T, 1>(ga, gb, gm1);
                    T dU[NV], w[NV];
#pragma unroll
                    for (int v = 0; v < NV; ++v) {
                        const T* u = cq + (CL::U + v) * NCELL + f;
                        if (EXACTDET) dU[v] = -fifth_difference(u[0], u[1], u[2], u[3], u[4], u[5]);
                        else dU[v] = fmaT(T(10), u[2] - u[3], fmaT(T(5), u[4] - u[1], u[0] - u[5]));
                    }
                    proj_all<T, 1, 0>(ro, dU, w);
                    const T lim = slim * ro.rt;
                    int fmask = 0;
#pragma unroll
                    for (int s = 0; s < NV; ++s) fmask |= abs_lt(w[s], lim) ? (1 << s) : 0;
                    const bool smooth = a.hybrid != 0 && fmask == (1 << NV) - 1;
                    T am, a0, ap;
                    if (a.split == SPLIT_LLF) {
                        const T *lm = cq + CL::LM * NCELL + f, *l0 = cq + CL::L0 * NCELL + f,
                                *lp = cq + CL::LP * NCELL + f;
                        am = lm[0]; a0 = l0[0]; ap = lp[0];
#pragma unroll
                        for (int k = 1; k < 6; ++k) {
                            am = max_nn(am, lm[k]); a0 = max_nn(a0, l0[k]); ap = max_nn(ap, lp[k]);
                        }
                    } else {   // SPLIT_RF (the host keeps global Lax-Friedrichs off this kernel)
                        am = absT(ro.u[0] - ro.c);
                        a0 = absT(ro.u[0]);
                        ap = absT(ro.u[0] + ro.c);
                    }
                    if (smooth) {
                        T Fo[NV];
#pragma unroll
                        for (int v = 0; v < NV; ++v) {
                            const T* x = cq + (CL::F + v) * NCELL + f;
                            const T f05 = x[0] + x[5], f14 = x[1] + x[4], f23 = x[2] + x[3];
                            Fo[v] = fmaT(T(37), f23, fmaT(T(-8), f14, f05));
                        }
                        ups_dissipation_add<T, 1, 0>(ro, dU, w, am, a0, ap, Fo);
#pragma unroll
                        for (int v = 0; v < NV; ++v) fh[v * NFACE + f] = Fo[v];
                    } else {
                        weno = true;
                        fr[FR::U * NFACE + f] = ro.u[0];
                        fr[FR::C * NFACE + f] = ro.c;
                        fr[FR::IC * NFACE + f] = ro.ic;
                        fr[FR::H * NFACE + f] = ro.H;
                        fr[FR::B1 * NFACE + f] = ro.b1;
                        fr[FR::HQ2 * NFACE + f] = ro.hq2;
#pragma unroll
                        for (int s = 0; s < NV; ++s) fr[(FR::W + s) * NFACE + f] = w[s];
                        fr[FR::IRT2 * NFACE + f] = Ar<T>::rcp_f(ro.rt * ro.rt);
                        fr[FR::AM * NFACE + f] = halve(am);
                        fr[FR::A0 * NFACE + f] = halve(a0);
                        fr[FR::AP * NFACE + f] = halve(ap);
                        fr[FR::MASK * NFACE + f] = T(a.hybrid == 2 ? fmask : 0);
                        // a face is owned by the segment right of it, the last one by the last segment
                        if (f < m || hi == n) ++stage_wenos;
                    }
                }
                const unsigned int mask = __ballot_sync(0xffffffffu, weno);
                if (mask) {
                    const int leader = __ffs(mask) - 1;
                    int base = 0;
                    if (lane == leader) base = atomicAdd(&qcount, __popc(mask));
                    base = __shfl_sync(0xffffffffu, base, leader);
                    if (weno) queue[base + __popc(mask & ((1u << lane) - 1u))] = f;
                }
            }
            __syncthreads();
            if (st == 0) {
                if (s_stop) { failed = true; break; }
                dt = T(s_dt);
            }
            wenos += stage_wenos;
            const int nq = qcount;
            if (nq > 0) {
                weno_queue<T, 1, 0, NCELL, NFACE, SM::QC, NT>(a, nq, cq, fh, fr, fpm, res, queue,
                                                              [](int f, int k) -> int { return f + k; });
                __syncthreads();
            }
            // divergence and the RK3 combination
            const T rka = pick<T>(st == 0 ? 0.0 : (st == 1 ? 0.75 : 1.0 / 3.0),
                                  st == 0 ? 0.0f : (st == 1 ? 0.75f : (float)(1.0 / 3.0)));
            const T rkb = pick<T>(st == 0 ? 1.0 : (st == 1 ? 0.25 : 2.0 / 3.0),
                                  st == 0 ? 1.0f : (st == 1 ? 0.25f : (float)(2.0 / 3.0)));
            bool bad = false, cbad = false;
            T smax = T(0);
            for (int i = tid; i < m; i += NT) {
                T nu[NV];
#pragma unroll
                for (int v = 0; v < NV; ++v) {
                    const T rv = (fh[v * NFACE + i] - fh[v * NFACE + i + 1]) * inv_dx;
                    T val = rkb * fmaT(dt, rv, cq[(CL::U + v) * NCELL + i + 3]);
                    if (rka != T(0)) val = fmaT(rka, ub[(cur * NV + v) * M + i], val);
                    nu[v] = val;
                    ub[(out * NV + v) * M + i] = val;
                }
                // admissibility: rho > 0, p > 0  <=>  2 rho E > |m|^2, finite
                const T m2 = fmaT(nu[1], nu[1], T(0));
                const T chk = T(2) * nu[0] * nu[2] - m2;
                if (!(nu[0] > T(0)) || !(chk > T(0)) || !isfinite(chk)) bad = true;
                if (st == 2) {
                    T sp;
                    if (!cell_speed<T, 1>(nu, gamma, inv_dx1, sp)) cbad = true;
                    else smax = max_nn(smax, sp);
                }
            }
            turn ^= 1;
            tell(bad, cbad, smax);
            int any = 0;
            for (int k = 0; k < C; ++k) any |= x_bad[turn][k];
            if (any & 1) {   // the state before the step stays
                status = 1;
                failed = true;
                break;
            }
        }
        if (failed) break;
        cur = 1 - cur;
        ++done;
        if (tid == NT - 1) t = clipped ? t_end : t + s_dt;
    }

    if (live && done > 0) {
        T* p = reinterpret_cast<T*>(r.buf[(phase0 + done) % 3]) + a.off0 + lo;
        for (int i = tid; i < m; i += NT)
#pragma unroll
            for (int v = 0; v < NV; ++v) p[i + v * a.sv] = ub[(cur * NV + v) * M + i];
    }
    if (a.weno_count != nullptr) {
        const unsigned int w = __reduce_add_sync(0xffffffffu, wenos);
        if (lane == 0 && w != 0u) atomicAdd(a.weno_count, (unsigned long long)w);
    }
    // every CTA has read the time and the state, and no CTA leaves while
    // another may still read its shared memory
    cluster_barrier();
    if (rank == 0 && tid == NT - 1 && live) {
        tm->t = t;
        tm->steps = steps0 + done;
        tm->phase = (phase0 + done) % 3;
        tm->dt = 0.0;
        tm->clipped = clipped;
        if (status != 0) tm->status = 1;
    }
}

// CTAs of a line of n cells: at least kRun1DMinCells and less than `cells`
// cells each; 0 if the line is too long.  n >= 3, and with more than one CTA each has more than three
// cells, so that a stencil reaches no further than the neighbour.
inline int run1d_ctas(int n, int cells, int max_cluster)
{
    int c = 1;
    while (2 * c <= max_cluster && n / (2 * c) >= kRun1DMinCells) c *= 2;
    return n <= c * (cells - 1) ? c : 0;
}

template <typename T, bool EXACTDET>
cudaError_t run1d_prepare(int* max_cluster)
{
    auto kern = k_run1d<T, EXACTDET>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Run1DSmem<T>::bytes);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    *max_cluster = 0;
    for (int c = kRun1DMaxCluster; c >= 1 && *max_cluster == 0; c /= 2) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)c);
        cfg.blockDim = dim3(kRun1DThreads);
        cfg.dynamicSmemBytes = Run1DSmem<T>::bytes;
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = (unsigned)c;
        at[0].val.clusterDim.y = 1;
        at[0].val.clusterDim.z = 1;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        int fit = 0;
        if (cudaOccupancyMaxActiveClusters(&fit, kern, &cfg) == cudaSuccess && fit > 0) *max_cluster = c;
        else cudaGetLastError();
    }
    return cudaSuccess;
}

template <typename T, bool EXACTDET>
cudaError_t launch_run1d(const Run1DArgs& r, int ctas, cudaStream_t s)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)ctas);
    cfg.blockDim = dim3(kRun1DThreads);
    cfg.dynamicSmemBytes = Run1DSmem<T>::bytes;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)ctas;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_run1d<T, EXACTDET>, r);
}

}  // namespace wis
