// Persistent batched solver (1D instances: weno_batch.cu, 2D instances:
// weno_batch2d.cu): many independent Euler problems of uneven sizes, each
// advanced to its own end time with its own CFL step.
//
// One launch of CTAs works through a queue of tasks.  A task is a run of
// consecutive tiles of one sweep of one instance.  The CTA that
// finishes the last run of a sweep goes on with the instance's next sweep,
// putting parts of it into the queue when other CTAs have nothing to do, and
// after the last sweep of a step (Sec. 4 of the paper) it also advances the
// instance's time and takes the next CFL step.  Instances wait
// only for their own previous sweep.  A CTA without a task polls its place in
// the queue; it holds nothing that another CTA waits for, and a CTA that does
// not run yet holds nothing at all (instances to prepare come from a counter,
// tasks from the queue), so the polls end whichever CTAs are resident.
//
// What bounds it: the FP64 pipe (FP64), instruction issue and shared-memory
// loads (FP32).  In the first form of this solver one CTA integrated one
// instance from start to end.  The steps of an instance vary by a factor of
// twenty, and a CTA alone uses a third of its SM, so the heaviest of 1024
// Riemann problems (1913 cells, 224 steps, 0.7% of the work) took 80 of 125
// ms.  The figures stand beside the launch shapes in weno_batch.cu and
// weno_batch2d.cu.
//
// The tiles are the grid solver's (sweep_tile, line_tile), so every face is
// computed by identical arithmetic; maxima and flags do not depend on the
// order in which tiles finish.
#pragma once

#include <cuda_runtime.h>

#include "../../include/weno_is.h"
#include "weno_kernels.cuh"
#include "weno_line.cuh"

namespace wis {

// constants of one instance (written by the host)
struct BatchInst {
    int nx, ny;                  // ny = 1 in 1D
    long long off;               // its states [nvar][ny][nx] start here in U and in the work arrays
    double inv_dx[2], slim[2];   // per direction: 1 / dx, 60 sqrt(eps_h)
    float inv_dx_f[2], inv_dx60_f[2], slim_f[2];
};

// progress of one instance (zeroed before each run)
struct BatchState {
    double t, dt;                // dt = 0: finished
    unsigned long long smax;     // CFL wave speed of the current state (bits)
    long long steps;
    int left;                    // runs of the current sweep not yet finished
    int runs;                    // and how many there are
    int run;                     // tiles per run of the current sweep
    int phase;                   // sweep of the step: 1D the stage, 2D 2 stage + (0 y, 1 x)
    int cur;                     // work array (0 or 1) of the current state
    int clipped;                 // the step in progress ends at t_end
    int bad;                     // BAD_STAGE, BAD_CFL
    float dt_f;
};
enum { BAD_STAGE = 1, BAD_CFL = 2 };

// one place of the task queue
struct BatchTask {
    int inst, run;
    unsigned int turn;           // how often the place has been filled
    unsigned int taken;          // and how often read
};

// counters of one run (zeroed before each run)
struct BatchCtrl {
    unsigned long long head;           // places taken by CTAs
    unsigned long long tail;           // tasks put into the queue
    unsigned long long progress;       // sweeps of all instances so far, and parts of long ones
    unsigned int prepared;             // instances taken for preparation
    // polled by CTAs without a task, so not beside the counters they take from
    alignas(128) int finished;         // instances
    int abort;                         // a wait for a task ran out
};

struct BatchArgs {
    int count;
    const int* order;            // instance ids, most work first
    const BatchInst* inst;
    BatchCtrl* ctrl;
    BatchState* state;
    BatchTask* queue;            // one place per tile of the batch
    long long places;
    const double* t_end;
    void* U;
    void* work[3];               // two rotating states and the second stage
    void* acc;                   // 2D: divergence of the y sweep
    void* prim;                  // 2D FP64: cell primitives of the stage's state (PrimLayout records);
                                 // null: both sweeps compute them
    int* status;                 // per instance: 0 ok, WENO_ERR_NONPHYSICAL
    long long* steps;
    double* t_out;
    unsigned long long* weno_count;
    int max_steps;
    int polls;                   // of a wait before it runs out (kTaskPolls)
    const int* trial_caps;       // autotuner trial runs: step cap per instance (null otherwise)
    int write_back;              // 0: trial run, the caller's states are not touched
    double gamma, cfl, eps, c_lambda;
    float gamma_f, eps_f, lam_scale_f;
    int hybrid, wmode, split;
    int bc_lo[2], bc_hi[2];
};

// polls of a CTA for its next task, while no other makes progress, before it
// gives up (some seconds at 100 ns each); weno_batch_set_wait sets another number
constexpr int kTaskPolls = 1 << 26;
// A sweep that is one run (every CTA had work when it began) of an instance of
// millions of cells can outlast those polls: a run counts as progress every
// kBeat tiles (about a millisecond), and so do the copies of the states.
constexpr int kBeat = 32;

// tiles of nx x ny cells along direction d
template <typename CFG>
__host__ __device__ inline int batch_tiles(int dim, int nx, int ny, int d)
{
    if (dim == 1) return (nx + CFG::XS - 1) / CFG::XS;
    return d == 0 ? ((nx + CFG::XS - 1) / CFG::XS) * ((ny + CFG::XL - 1) / CFG::XL)
                  : ((ny + CFG::YS - 1) / CFG::YS) * ((nx + CFG::YL - 1) / CFG::YL);
}

// sweep arguments of one instance along direction d
template <int DIM, bool FX>
__device__ __forceinline__ SweepArgs batch_sweep_args(const BatchArgs& b, const BatchInst& q, int d)
{
    SweepArgs a;
    const long long cells = (long long)q.nx * q.ny;
    a.n[0] = q.nx; a.n[1] = q.ny; a.n[2] = 1;
    a.sy = q.nx; a.sz = cells; a.sv = cells; a.off0 = 0;
    a.acc = nullptr; a.Un = nullptr; a.out = nullptr;
    a.tm = nullptr;
    a.weno_count = b.weno_count;
    a.flags = nullptr;
    a.alpha_g = nullptr;
    a.inv_dx = q.inv_dx[d];
    a.slim = q.slim[d];
    a.gamma = b.gamma; a.eps = b.eps; a.c_lambda = b.c_lambda; a.hybrid = b.hybrid;
    a.wmode = b.wmode; a.split = b.split;
    a.inv_dx_f = q.inv_dx60_f[d];
    a.slim_f = q.slim_f[d];
    a.gamma_f = b.gamma_f; a.eps_f = b.eps_f; a.lam_scale_f = b.lam_scale_f;
    a.bc_lo = b.bc_lo[d]; a.bc_hi = b.bc_hi[d];
    a.stage = 0;
    a.fx = FX && use_fx(cells);
    return a;
}

// Time bookkeeping of one instance between two steps (first: before the
// first one): takes over the step just made, then the next CFL step.
__device__ __forceinline__ void batch_next_step(const BatchArgs& b, int inst, bool first)
{
    BatchState& s = b.state[inst];
    const double t_end = b.t_end[inst];
    const long long max_steps = b.trial_caps != nullptr ? (long long)b.trial_caps[inst] : (long long)b.max_steps;
    int status = 0;
    double t = s.t, dt = 0.0;
    long long steps = s.steps;
    int clipped = s.clipped;
    // what the sweep's warps noted by atomics, past this SM's L1
    const int bad = *(volatile int*)&s.bad;
    const unsigned long long smax = *(volatile unsigned long long*)&s.smax;
    if (!first) {
        if (bad & BAD_STAGE) {
            status = WENO_ERR_NONPHYSICAL;   // the state before the step stays
        } else {
            s.cur = 1 - s.cur;
            t = clipped ? t_end : t + s.dt;
            ++steps;
        }
    }
    if (status == 0 && steps < max_steps) {
        if (bad & BAD_CFL) status = WENO_ERR_NONPHYSICAL;
        else dt = cfl_step(b.cfl, __longlong_as_double((long long)smax), t, t_end, &clipped);
    }
    s.t = t;
    s.steps = steps;
    s.clipped = clipped;
    s.dt = dt;
    s.dt_f = (float)dt;
    s.smax = 0ull;
    s.bad = 0;
    if (!(dt > 0.0)) {
        b.status[inst] = status;
        b.steps[inst] = steps;
        b.t_out[inst] = t;
    }
}

// Most tiles of a sweep that is never split: a run that another CTA takes costs
// some 2 us in the queue and at the sweep's end, as much as a 1D tile in FP32
// (one line of 200 cells: 136 us in runs of one tile, 113 us in one run).
template <typename T, int DIM> constexpr int kBatchUnsplit = DIM == 1 && sizeof(T) == 4 ? 2 : 1;

// One thread: moves an instance to its next sweep and reserves its places in
// the queue: nr runs from place number `at` on.  Returns true when the
// instance has finished instead.
template <typename T, int DIM, typename CFG>
__device__ bool batch_next_sweep(const BatchArgs& b, int inst, bool first, int& nr, unsigned long long& at)
{
    BatchState& s = b.state[inst];
    // read beside the instance's progress, not after it
    const unsigned long long head = *(volatile unsigned long long*)&b.ctrl->head,
                             tail = *(volatile unsigned long long*)&b.ctrl->tail;
    const int nx = b.inst[inst].nx, ny = b.inst[inst].ny;
    atomicAdd(&b.ctrl->progress, 1ull);
    if (!first && s.phase + 1 < 3 * DIM) {
        s.phase += 1;
    } else {
        batch_next_step(b, inst, first);
        s.phase = 0;
        if (!(s.dt > 0.0)) {
            nr = 0;
            return true;
        }
    }
    const int nt = batch_tiles<CFG>(DIM, nx, ny, DIM == 2 && (s.phase & 1) == 0 ? 1 : 0);
    // While tasks wait for a CTA, the whole sweep is one run, which this CTA
    // goes on with: the instance stays in L1 and L2, and nothing waits for the
    // queue (runs of 8 tiles, all through the queue: 4096 Riemann problems in
    // FP32 148 ms against 121 ms here, 4096 boxes in FP32 75 against 70 ms, both
    // FP64 batches alike).  When CTAs wait for tasks, it is split for as many of
    // them as there are.
    const long long idle = (long long)(head - tail);
    const int most = idle <= 0 || nt <= kBatchUnsplit<T, DIM> ? 1 : (idle + 1 < nt ? (int)idle + 1 : nt);
    const int run = (nt + most - 1) / most;
    nr = (nt + run - 1) / run;
    s.run = run;
    s.runs = nr;
    s.left = nr;
    // before the first sweep every run goes to the queue, later ones keep run 0
    if (first || nr > 1) at = atomicAdd(&b.ctrl->tail, (unsigned long long)(first ? nr : nr - 1));
    return false;
}

// One warp: fills the places reserved by batch_next_sweep with the runs r0 ..
// nr - 1 (its stores, and those the block made before, are visible to the CTAs
// that take the tasks).  A place is filled again only when its last task has
// been read: no more tasks than places are outstanding, so that task has been
// claimed by a running CTA.
__device__ __forceinline__ void batch_put(const BatchArgs& b, int inst, int r0, int nr, unsigned long long at)
{
    const unsigned long long places = (unsigned long long)b.places;
    for (int r = r0 + (int)(threadIdx.x & 31); r < nr; r += 32) {
        const unsigned long long k = at + (unsigned long long)(r - r0), turn = k / places;
        BatchTask* q = b.queue + (long long)(k - turn * places);
        bool free = false;
        for (int w = 0; w < b.polls && !free; ++w) {
            unsigned int v;
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(&q->taken) : "memory");
            free = v == (unsigned int)turn;
            if (!free && *(volatile int*)&b.ctrl->abort != 0) return;
        }
        if (!free) {   // the place still holds a task that nobody has read
            atomicExch(&b.ctrl->abort, 1);
            return;
        }
        q->inst = inst;
        q->run = r;
        __threadfence();
        *(volatile unsigned int*)&q->turn = (unsigned int)turn + 1u;
    }
}

// One thread: the next task; false when every instance has finished (or a
// wait ran out).
__device__ __forceinline__ bool batch_take(const BatchArgs& b, int& inst, int& run)
{
    const unsigned long long at = atomicAdd(&b.ctrl->head, 1ull);
    const unsigned long long turn = at / (unsigned long long)b.places;
    BatchTask* q = b.queue + (long long)(at - turn * (unsigned long long)b.places);
    unsigned long long seen = 0ull;
    for (int k = 0;; ++k) {
        unsigned int v;
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(&q->turn) : "memory");
        if (v == (unsigned int)turn + 1u) break;
        if ((k & 3) == 0) {   // at once, so that a run ends soon after its last instance
            if (*(volatile int*)&b.ctrl->finished >= b.count || *(volatile int*)&b.ctrl->abort != 0) return false;
            if (k >= b.polls) {
                const unsigned long long now = *(volatile unsigned long long*)&b.ctrl->progress;
                if (now == seen) {
                    atomicExch(&b.ctrl->abort, 1);
                    return false;
                }
                seen = now;
                k = 32;
            }
        }
        if (k > 32) __nanosleep(40);
    }
    inst = q->inst;
    run = q->run;
    asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(&q->taken), "r"((unsigned int)turn + 1u) : "memory");
    return true;
}

template <typename T, int DIM, typename CFG, bool EXACTDET, bool FX>
__global__ void __launch_bounds__(CFG::NT, CFG::template min_blocks<T>()) k_batch(BatchArgs b)
{
    constexpr int NT = CFG::NT, NV = DIM + 2;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int s_inst, s_run, s_done;
    __shared__ bool s_alone;
    unsigned int wenos = 0;
    const int lane = threadIdx.x & 31;
    const T gamma = pick<T>(b.gamma, b.gamma_f);
    T* W[3] = {reinterpret_cast<T*>(b.work[0]), reinterpret_cast<T*>(b.work[1]), reinterpret_cast<T*>(b.work[2])};
    T* U = reinterpret_cast<T*>(b.U);
    // CFL wave speeds and flags of cells of one instance into its progress
    auto note_cfl = [&](BatchState& s, T smax, bool bad) {
        const T m = warp_max_nn(smax);
        if (lane == 0 && m > T(0)) atomicMax(&s.smax, (unsigned long long)__double_as_longlong((double)m));
        if (bad) atomicOr(&s.bad, BAD_CFL);
    };
    auto beat = [&](long long i, long long every) {
        if (threadIdx.x == 0 && i % every == every - 1) atomicAdd(&b.ctrl->progress, 1ull);
    };
    // the first warp queues the instance's next sweep; the states of a finished
    // instance go back to the caller.  Every thread calls it; the sweep's (or
    // the preparation's) stores come before.  True if this CTA goes on with
    // run 0 of the next sweep.
    auto next_sweep = [&](int inst, bool first) -> bool {
        __syncthreads();
        if (threadIdx.x < 32) {
            int done = 0, nr = 0;   // done: 0 others still work on the sweep, 1 finished, 2 go on
            unsigned long long at = 0ull;
            if (threadIdx.x == 0) {
                // A sweep of one run has nothing to take over from other CTAs
                // and, if the next one is too, nothing to publish (2000 lines
                // of 20 to 60 cells in FP32 127 us with them, 98 us without).
                const bool alone = !first && s_alone;
                if (!alone) __threadfence();
                if (first || alone || atomicSub(&b.state[inst].left, 1) == 1) {
                    if (!alone) __threadfence();
                    done = batch_next_sweep<T, DIM, CFG>(b, inst, first, nr, at) ? 1 : 2;
                    if (first || nr > 1) __threadfence();
                }
                s_done = done;
            }
            nr = __shfl_sync(0xffffffffu, nr, 0);
            at = __shfl_sync(0xffffffffu, at, 0);
            // the shuffles order no memory: the tasks that the other lanes
            // publish come after lane 0's stores, and the stores it acquired
            __syncwarp();
            if (first || nr > 1) batch_put(b, inst, first ? 0 : 1, nr, at);
        }
        __syncthreads();
        const int done = s_done;
        if (done == 1) {
            if (b.write_back) {
                const BatchInst q = b.inst[inst];
                const T* w = W[b.state[inst].cur] + q.off;
                for (long long c = threadIdx.x; c < (long long)NV * q.nx * q.ny; c += NT) {
                    U[q.off + c] = w[c];
                    beat(c / NT, 64 * kBeat);
                }
            }
            __syncthreads();
            if (threadIdx.x == 0) atomicAdd(&b.ctrl->finished, 1);
        }
        return done == 2;
    };

    // Initial states, and their CFL wave speeds.  The instances come from a
    // counter, so that only a running CTA holds one that is not in the queue yet.
    for (;;) {
        if (threadIdx.x == 0) s_inst = (int)atomicAdd(&b.ctrl->prepared, 1u);
        __syncthreads();
        const unsigned int k = (unsigned int)s_inst;
        if (k >= (unsigned int)b.count) break;
        const int inst = b.order[k];
        const BatchInst q = b.inst[inst];
        const long long cells = (long long)q.nx * q.ny;
        T ih[DIM];
#pragma unroll
        for (int d = 0; d < DIM; ++d) ih[d] = pick<T>(q.inv_dx[d], q.inv_dx_f[d]);
        T m = T(0);
        bool bad = false;
        for (long long c = threadIdx.x; c < cells; c += NT) {
            T u[NV], sp;
#pragma unroll
            for (int v = 0; v < NV; ++v) {
                u[v] = U[q.off + v * cells + c];
                W[0][q.off + v * cells + c] = u[v];
            }
            if (!cell_speed<T, DIM>(u, gamma, ih, sp)) bad = true;
            else m = max_nn(m, sp);
            beat(c / NT, 16 * kBeat);
        }
        note_cfl(b.state[inst], m, bad);
        next_sweep(inst, true);
    }
    __syncthreads();   // every thread has read s_inst

    int inst = -1, run = 0;
    bool go_on = false;
    for (;;) {
        if (go_on) {
            run = 0;
        } else {
            if (threadIdx.x == 0) {
                int i = -1, k = 0;
                if (!batch_take(b, i, k)) i = -1;
                s_inst = i;
                s_run = k;
            }
            __syncthreads();
            inst = s_inst;
            run = s_run;
            if (inst < 0) break;
        }
        BatchState& s = b.state[inst];
        const BatchInst q = b.inst[inst];
        const int phase = s.phase, cur = s.cur, len = s.run;
        if (threadIdx.x == 0) s_alone = s.runs == 1;
        const T dt = pick<T>(s.dt, s.dt_f);
        const int t0 = run * len;
        // three stages: x = cur + dt L(cur); y = 3/4 cur + 1/4 (x + dt L(x));
        // x = 1/3 cur + 2/3 (y + dt L(y)), x the other one of work arrays 0
        // and 1, y work array 2
        const int st = DIM == 2 ? phase >> 1 : phase;
        const int in = st == 0 ? cur : (st == 1 ? 1 - cur : 2), out = st == 1 ? 2 : 1 - cur;
        if (DIM == 2 && (phase & 1) == 0) {
            SweepArgs a = batch_sweep_args<DIM, FX>(b, q, 1);
            a.mode = MODE_ACC_SET;
            a.U = W[in] + q.off;
            a.acc = reinterpret_cast<T*>(b.acc) + q.off;
            // as in a step of the grid solver, the y sweep computes and stores
            // the cell primitives and the x sweep reads them
            if (sizeof(T) == 8 && b.prim != nullptr)
                a.Pout = reinterpret_cast<T*>(b.prim) + q.off / NV * PrimLayout<DIM>::STRIDE;
            const int t1 = min(t0 + len, batch_tiles<CFG>(DIM, q.nx, q.ny, 1)), ns = (q.ny + CFG::YS - 1) / CFG::YS;
            if constexpr (DIM == 2) {
                for (int t = t0; t < t1; ++t) {
                    const int lg = t / ns;
                    sweep_tile<T, DIM, 1, CFG::YL, CFG::YS, NT, EXACTDET, false, FX, true>(a, t - lg * ns, lg * CFG::YL,
                                                                                           0, T(0), smem_raw);
                    beat(t - t0, kBeat);
                }
            }
        } else {
            SweepArgs a = batch_sweep_args<DIM, FX>(b, q, 0);
            a.mode = MODE_COMBINE;
            a.U = W[in] + q.off;
            a.Un = W[cur] + q.off;
            a.out = W[out] + q.off;
            a.rk_a = st == 0 ? 0.0 : (st == 1 ? 0.75 : 1.0 / 3.0);
            a.rk_b = st == 0 ? 1.0 : (st == 1 ? 0.25 : 2.0 / 3.0);
            a.rk_a_f = st == 0 ? 0.0f : (st == 1 ? 0.75f : (float)(1.0 / 3.0));
            a.rk_b_f = st == 0 ? 1.0f : (st == 1 ? 0.25f : (float)(2.0 / 3.0));
            TileCfl<T, DIM> cfl;
#pragma unroll
            for (int d = 0; d < DIM; ++d) cfl.inv_dx[d] = pick<T>(q.inv_dx[d], q.inv_dx_f[d]);
            cfl.smax = T(0);
            cfl.bad = false;
            TileCfl<T, DIM>* const cp = st == 2 ? &cfl : nullptr;
            const int t1 = min(t0 + len, batch_tiles<CFG>(DIM, q.nx, q.ny, 0));
            bool bad = false;
            if constexpr (DIM == 1) {
                T u[3];
                line_load(a, t0 * CFG::XS, u);
                for (int t = t0; t < t1; ++t) {
                    bad |= line_tile<T, NT, EXACTDET, FX>(a, t * CFG::XS, t + 1 < t1 ? (t + 1) * CFG::XS : -1, dt, u,
                                                          smem_raw, cp, wenos);
                    beat(t - t0, kBeat);
                }
            } else {
                a.acc = reinterpret_cast<T*>(b.acc) + q.off;
                a.acc_scale = q.inv_dx[1] * (1.0 / 60.0);   // the y sweep stores unscaled flux differences
                a.acc_scale_f = q.inv_dx60_f[1];
                if (sizeof(T) == 8 && b.prim != nullptr) a.P = reinterpret_cast<const T*>(b.prim) + q.off / NV * PrimLayout<DIM>::STRIDE;
                const int ns = (q.nx + CFG::XS - 1) / CFG::XS;
                for (int t = t0; t < t1; ++t) {
                    const int lg = t / ns;
                    bad |= sweep_tile<T, DIM, 0, CFG::XL, CFG::XS, NT, EXACTDET, false, FX>(a, t - lg * ns, lg * CFG::XL,
                                                                                            0, dt, smem_raw, cp);
                    beat(t - t0, kBeat);
                }
            }
            if (bad) atomicOr(&s.bad, BAD_STAGE);
            if (st == 2) note_cfl(s, cfl.smax, cfl.bad);
        }
        go_on = next_sweep(inst, false);
    }

    if (DIM == 1 && b.weno_count != nullptr) {   // the 2D tiles count their own
        const unsigned int w = __reduce_add_sync(0xffffffffu, wenos);
        if (lane == 0 && w != 0u) atomicAdd(b.weno_count, (unsigned long long)w);
    }
}

// CTAs per SM and shared memory of a configuration
template <typename T, int DIM, typename CFG, bool EXACTDET, bool FX>
cudaError_t batch_config(int* blocks_per_sm, size_t* smem)
{
    auto kern = k_batch<T, DIM, CFG, EXACTDET, FX>;
    constexpr size_t bytes = CFG::template smem_bytes<T>();
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
    if (e != cudaSuccess) return e;
    *smem = bytes;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, kern, CFG::NT, bytes);
}

template <typename T, int DIM, typename CFG, bool EXACTDET, bool FX>
cudaError_t batch_launch(const BatchArgs& b, int blocks, cudaStream_t s)
{
    k_batch<T, DIM, CFG, EXACTDET, FX><<<blocks, CFG::NT, CFG::template smem_bytes<T>(), s>>>(b);
    return cudaGetLastError();
}

// Host entry points of the two kernels; variant v in [0, kBatchVariants), fx:
// an FP64 instance of the batch takes the integer six-point sums (use_fx).
// batch*_tiles: tiles of one instance along direction d.
constexpr int kBatchVariants = 3;
cudaError_t batch1d_config(int prec, bool fx, int v, int* blocks_per_sm, size_t* smem);
cudaError_t batch1d_launch(int prec, bool fx, int v, const BatchArgs& b, int blocks, cudaStream_t s);
int batch1d_tiles(int v, int nx);
cudaError_t batch2d_config(int prec, bool fx, int v, int* blocks_per_sm, size_t* smem);
cudaError_t batch2d_launch(int prec, bool fx, int v, const BatchArgs& b, int blocks, cudaStream_t s);
int batch2d_tiles(int v, int nx, int ny, int d);

// the dispatch over precision and variant, shared by the two translation
// units; CFG<V> is the unit's configuration template
template <int DIM, template <int> class CFG, typename T, bool EXACTDET, bool FX>
cudaError_t batch_config_v(int v, int* bps, size_t* smem)
{
    if (v == 1) return batch_config<T, DIM, CFG<1>, EXACTDET, FX>(bps, smem);
    if (v == 2) return batch_config<T, DIM, CFG<2>, EXACTDET, FX>(bps, smem);
    return batch_config<T, DIM, CFG<0>, EXACTDET, FX>(bps, smem);
}
template <int DIM, template <int> class CFG>
cudaError_t batch_config_p(int prec, bool fx, int v, int* bps, size_t* smem)
{
    if (prec == WENO_FP64)
        return fx ? batch_config_v<DIM, CFG, double, false, true>(v, bps, smem)
                  : batch_config_v<DIM, CFG, double, false, false>(v, bps, smem);
    return prec == WENO_MIXED ? batch_config_v<DIM, CFG, float, true, false>(v, bps, smem)
                              : batch_config_v<DIM, CFG, float, false, false>(v, bps, smem);
}
template <int DIM, template <int> class CFG, typename T, bool EXACTDET, bool FX>
cudaError_t batch_launch_v(int v, const BatchArgs& b, int blocks, cudaStream_t s)
{
    if (v == 1) return batch_launch<T, DIM, CFG<1>, EXACTDET, FX>(b, blocks, s);
    if (v == 2) return batch_launch<T, DIM, CFG<2>, EXACTDET, FX>(b, blocks, s);
    return batch_launch<T, DIM, CFG<0>, EXACTDET, FX>(b, blocks, s);
}
template <int DIM, template <int> class CFG>
cudaError_t batch_launch_p(int prec, bool fx, int v, const BatchArgs& b, int blocks, cudaStream_t s)
{
    if (prec == WENO_FP64)
        return fx ? batch_launch_v<DIM, CFG, double, false, true>(v, b, blocks, s)
                  : batch_launch_v<DIM, CFG, double, false, false>(v, b, blocks, s);
    return prec == WENO_MIXED ? batch_launch_v<DIM, CFG, float, true, false>(v, b, blocks, s)
                              : batch_launch_v<DIM, CFG, float, false, false>(v, b, blocks, s);
}

}  // namespace wis
