// Batched solver: the host object of the persistent batch kernel
// (weno_batch.cuh) for 1D and 2D instances, and the 1D instantiations.
#include <cuda_runtime.h>

#include <algorithm>
#include <climits>
#include <cmath>
#include <cstring>
#include <new>
#include <numeric>
#include <string>
#include <vector>

#include "../../include/weno_is.h"
#include "weno_batch.cuh"

namespace wis {

// Line tiles on 128, 64 and 256 threads (LineTile).  1024 Riemann problems of
// 100 to 2000 cells in FP64: 63, 68 and 61 ms, with the FP64 pipe 85% busy
// over the first steps (one CTA per instance: 125, 192 and 75 ms, the
// heaviest instance alone 80 ms against 12 ms here); 4096 of 100 to 4000
// cells in FP32: 123, 142 and 129 ms (231, 380 and 146 ms).  128 threads are
// the default.
template <int V>
struct Batch1Cfg {
    static constexpr int NT = V == 0 ? 128 : (V == 1 ? 64 : 256);
    static constexpr int XS = NT - 6, XL = 1, YL = 1, YS = 1;
    template <typename T> static constexpr size_t smem_bytes() { return LineTile<T, NT>::bytes; }
    template <typename T> static constexpr int min_blocks() { return (sizeof(T) == 8 ? 640 : 1024) / NT; }
};

cudaError_t batch1d_config(int prec, bool fx, int v, int* blocks_per_sm, size_t* smem)
{
    return batch_config_p<1, Batch1Cfg>(prec, fx, v, blocks_per_sm, smem);
}
cudaError_t batch1d_launch(int prec, bool fx, int v, const BatchArgs& b, int blocks, cudaStream_t s)
{
    return batch_launch_p<1, Batch1Cfg>(prec, fx, v, b, blocks, s);
}
int batch1d_tiles(int v, int nx)
{
    if (v == 1) return batch_tiles<Batch1Cfg<1>>(1, nx, 1, 0);
    if (v == 2) return batch_tiles<Batch1Cfg<2>>(1, nx, 1, 0);
    return batch_tiles<Batch1Cfg<0>>(1, nx, 1, 0);
}

}  // namespace wis

using wis::BatchArgs;

struct weno_batch {
    int dim = 1;   // 1: [3][n] instances, 2: [4][ny][nx] instances
    int count = 0, prec = 0, dev = 0, nsm = 1;
    size_t esz = 8;
    weno_params p;
    int bc_lo[2] = {0, 0}, bc_hi[2] = {0, 0}, max_steps = 0;
    cudaStream_t stream = nullptr;
    cudaStream_t cap = nullptr;
    long long total = 0;          // elements of the states of all instances
    int* order = nullptr;
    wis::BatchInst* inst = nullptr;
    double* t_end = nullptr;
    void* work[4] = {nullptr, nullptr, nullptr, nullptr};   // the fourth: 2D accumulator
    void* prim = nullptr;           // 2D FP64: cell primitives
    unsigned char* run = nullptr;   // BatchCtrl, the BatchState of every instance, the task queue
    size_t run_bytes = 0;
    long long places = 0;           // of the queue: the tiles of all instances
    long long tiles_of[wis::kBatchVariants] = {};    // tiles of the longer direction, per variant
    int* status = nullptr;
    long long* steps = nullptr;
    double* t_out = nullptr;
    unsigned long long* wcount = nullptr;
    int* trial_caps = nullptr;
    std::vector<int> n_host;      // steps grow with this size: n (1D), max(nx, ny) (2D)
    bool fx = false;              // an FP64 instance takes the integer six-point sums
    int variant = 0;
    int residency = 0;            // most CTAs per SM, 0 = as many as fit
    int blocks = 0;               // reported: min(count, residency x SMs)
    int grid = 0;                 // CTAs launched: min(tiles, residency x SMs), or ctas
    int ctas = 0;                 // weno_batch_set_launch
    int polls = wis::kTaskPolls;  // weno_batch_set_wait
    cudaGraphExec_t graph = nullptr;
    void* graph_U = nullptr;
    std::string err;
};

// the BatchState array starts here in weno_batch::run
constexpr size_t kCtrlBytes = 256;
static_assert(sizeof(wis::BatchCtrl) <= kCtrlBytes, "control block");

static std::string g_batch_err;

#define BCK(call)                                                                           \
    do {                                                                                    \
        cudaError_t e_ = (call);                                                            \
        if (e_ != cudaSuccess) {                                                            \
            bt->err = std::string(#call) + ": " + cudaGetErrorString(e_);                   \
            return WENO_ERR_CUDA;                                                           \
        }                                                                                   \
    } while (0)

static cudaError_t dispatch_config(weno_batch* bt, int v, int* bps, size_t* smem)
{
    return bt->dim == 2 ? wis::batch2d_config(bt->prec, bt->fx, v, bps, smem)
                        : wis::batch1d_config(bt->prec, bt->fx, v, bps, smem);
}

static BatchArgs batch_args(weno_batch* bt, void* U, int max_steps, int write_back)
{
    BatchArgs b;
    std::memset(&b, 0, sizeof(b));
    b.count = bt->count;
    b.order = bt->order;
    b.inst = bt->inst;
    b.ctrl = reinterpret_cast<wis::BatchCtrl*>(bt->run);
    b.state = reinterpret_cast<wis::BatchState*>(bt->run + kCtrlBytes);
    b.queue = reinterpret_cast<wis::BatchTask*>(bt->run + kCtrlBytes + sizeof(wis::BatchState) * (size_t)bt->count);
    b.places = bt->places;
    b.t_end = bt->t_end;
    b.U = U;
    for (int k = 0; k < 3; ++k) b.work[k] = bt->work[k];
    b.acc = bt->work[3];
    b.prim = bt->prim;
    b.status = bt->status; b.steps = bt->steps; b.t_out = bt->t_out;
    b.weno_count = bt->wcount;
    b.max_steps = max_steps;
    b.polls = bt->polls;
    b.write_back = write_back;
    b.gamma = bt->p.gamma; b.cfl = bt->p.cfl; b.eps = bt->p.eps; b.c_lambda = bt->p.c_lambda;
    b.gamma_f = (float)bt->p.gamma;
    b.eps_f = (float)bt->p.eps;
    b.lam_scale_f = (float)(bt->p.c_lambda * (1.0 / 3600.0));
    b.hybrid = bt->p.hybrid;
    b.wmode = bt->p.weights; b.split = bt->p.splitting;
    for (int d = 0; d < 2; ++d) { b.bc_lo[d] = bt->bc_lo[d]; b.bc_hi[d] = bt->bc_hi[d]; }
    return b;
}

static weno_status set_variant(weno_batch* bt, int v, int blocks_per_sm_cap)
{
    int bps = 0;
    size_t smem = 0;
    BCK(dispatch_config(bt, v, &bps, &smem));
    if (bps < 1) { bt->err = "batch kernel cannot be resident"; return WENO_ERR_CUDA; }
    if (blocks_per_sm_cap > 0 && bps > blocks_per_sm_cap) bps = blocks_per_sm_cap;
    bt->variant = v;
    bt->residency = blocks_per_sm_cap;
    const long long resident = (long long)bps * bt->nsm;
    bt->blocks = (int)std::min<long long>(resident, bt->count);
    bt->grid = bt->ctas > 0 ? bt->ctas : (int)std::min<long long>(resident, bt->tiles_of[v]);
    if (bt->graph) cudaGraphExecDestroy(bt->graph);
    bt->graph = nullptr;
    return WENO_OK;
}

// one run on stream s (optionally under capture): counters and progress
// zeroed, then the kernel
static cudaError_t launch_run(weno_batch* bt, const BatchArgs& b, cudaStream_t s)
{
    cudaError_t e = cudaMemsetAsync(bt->run, 0, bt->run_bytes, s);
    if (e != cudaSuccess) return e;
    return bt->dim == 2 ? wis::batch2d_launch(bt->prec, bt->fx, bt->variant, b, bt->grid, s)
                        : wis::batch1d_launch(bt->prec, bt->fx, bt->variant, b, bt->grid, s);
}

static cudaError_t enqueue_run(weno_batch* bt, void* U, int max_steps, int write_back, cudaStream_t s,
                               const int* trial_caps = nullptr)
{
    BatchArgs b = batch_args(bt, U, max_steps, write_back);
    b.trial_caps = trial_caps;
    return launch_run(bt, b, s);
}

static void batch_free(weno_batch* bt)
{
    if (bt->graph) cudaGraphExecDestroy(bt->graph);
    void* ptrs[] = {bt->order, bt->inst, bt->t_end, bt->work[0], bt->work[1], bt->work[2], bt->work[3], bt->prim, bt->run,
                    bt->status, bt->steps, bt->t_out, bt->wcount, bt->trial_caps};
    for (void* q : ptrs)
        if (q) cudaFree(q);
    if (bt->cap) cudaStreamDestroy(bt->cap);
}

// Allocations and device tables of a batch whose dim, count, prec, p, bc_*,
// max_steps, stream and n_host are set: nx, ny (null in 1D), the spacings and
// end times per instance, and the schedule (most work first).
static cudaError_t batch_setup(weno_batch* bt, const int* nx, const int* ny, const std::vector<double>& dx,
                               const std::vector<double>& dy, const double* t_end, const std::vector<int>& order)
{
    const int cnt = bt->count, nv = bt->dim + 2;
    bt->esz = bt->prec == WENO_FP64 ? sizeof(double) : sizeof(float);
    std::vector<wis::BatchInst> inst(cnt);
    std::memset(inst.data(), 0, sizeof(wis::BatchInst) * cnt);
    long long off = 0;
    for (int i = 0; i < cnt; ++i) {
        wis::BatchInst& q = inst[i];
        q.nx = nx[i];
        q.ny = ny ? ny[i] : 1;
        q.off = off;
        const long long cells = (long long)q.nx * q.ny;
        off += nv * cells;
        for (int d = 0; d < bt->dim; ++d) {
            const double h = d == 0 ? dx[i] : dy[i];
            // Eq. eq31 with the spacing of the direction
            double eps_h = bt->p.C_thr;
            for (int k = 0; k < bt->p.alpha_thr; ++k) eps_h *= h / bt->p.L_char;
            q.inv_dx[d] = 1.0 / h;
            q.inv_dx_f[d] = (float)q.inv_dx[d];
            q.inv_dx60_f[d] = (float)(q.inv_dx[d] * (1.0 / 60.0));
            q.slim[d] = std::sqrt(3600.0 * eps_h);
            q.slim_f[d] = (float)q.slim[d];
        }
        bt->fx = bt->fx || (bt->prec == WENO_FP64 && wis::use_fx(cells));
        for (int v = 0; v < wis::kBatchVariants; ++v)
            bt->tiles_of[v] += bt->dim == 1 ? wis::batch1d_tiles(v, q.nx)
                                            : std::max(wis::batch2d_tiles(v, q.nx, q.ny, 0),
                                                       wis::batch2d_tiles(v, q.nx, q.ny, 1));
    }
    bt->total = off;
    for (int v = 0; v < wis::kBatchVariants; ++v) bt->places = std::max(bt->places, bt->tiles_of[v]);
    if (bt->places > INT_MAX) return cudaErrorInvalidValue;

    cudaError_t e = cudaGetDevice(&bt->dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&bt->nsm, cudaDevAttrMultiProcessorCount, bt->dev);
    auto alloc = [&](void** p, size_t bytes) {
        if (e == cudaSuccess) e = cudaMalloc(p, bytes);
    };
    bt->run_bytes = kCtrlBytes + sizeof(wis::BatchState) * (size_t)cnt + sizeof(wis::BatchTask) * (size_t)bt->places;
    alloc((void**)&bt->order, sizeof(int) * cnt);
    alloc((void**)&bt->inst, sizeof(wis::BatchInst) * cnt);
    alloc((void**)&bt->t_end, sizeof(double) * cnt);
    for (int k = 0; k < (bt->dim == 2 ? 4 : 3); ++k) alloc(&bt->work[k], bt->esz * (size_t)bt->total);
    alloc((void**)&bt->run, bt->run_bytes);
    alloc((void**)&bt->status, sizeof(int) * cnt);
    alloc((void**)&bt->steps, sizeof(long long) * cnt);
    alloc((void**)&bt->t_out, sizeof(double) * cnt);
    alloc((void**)&bt->wcount, sizeof(unsigned long long));
    alloc((void**)&bt->trial_caps, sizeof(int) * cnt);
    // The primitives are half as much again as the work arrays.  They are taken
    // where they leave at least as much memory free; without them the x sweeps
    // compute them too, with the same results (1024 explosions in FP64 58.9 ms
    // against 55.0).
    if (e == cudaSuccess && bt->dim == 2 && bt->prec == WENO_FP64) {
        const size_t bytes = bt->esz * (size_t)(bt->total / nv) * wis::PrimLayout<2>::STRIDE;
        size_t left = 0, all = 0;
        e = cudaMemGetInfo(&left, &all);
        if (e == cudaSuccess && left >= 2 * bytes && cudaMalloc(&bt->prim, bytes) != cudaSuccess) {
            cudaGetLastError();
            bt->prim = nullptr;
        }
    }
    if (e == cudaSuccess) e = cudaMemcpy(bt->order, order.data(), sizeof(int) * cnt, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(bt->inst, inst.data(), sizeof(wis::BatchInst) * cnt, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(bt->t_end, t_end, sizeof(double) * cnt, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemset(bt->wcount, 0, sizeof(unsigned long long));
    if (e == cudaSuccess) e = cudaMemset(bt->run, 0, bt->run_bytes);
    if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&bt->cap, cudaStreamNonBlocking);
    return e;
}

// the last part of both create calls
static weno_status finish_create(weno_batch* bt, cudaError_t e, const char* what, weno_batch** out)
{
    weno_status st = WENO_OK;
    if (e != cudaSuccess) {
        bt->err = std::string(what) + ": " + cudaGetErrorString(e);
        st = WENO_ERR_CUDA;
    } else {
        st = set_variant(bt, 0, 0);
    }
    if (st != WENO_OK) {
        g_batch_err = bt->err;
        batch_free(bt);
        delete bt;
        return st;
    }
    *out = bt;
    return WENO_OK;
}

extern "C" {

weno_status weno_batch_create(const weno_batch_desc* d, const weno_params* params, void* stream, weno_batch** out)
{
    if (out) *out = nullptr;
    if (!d || !params || !out || d->count < 1 || !d->n || !d->lo || !d->hi || !d->t_end) {
        g_batch_err = "invalid batch description";
        return WENO_ERR_INVALID_ARG;
    }
    if (params->precision < WENO_FP64 || params->precision > WENO_MIXED || d->max_steps < 0 ||
        params->weights < 0 || params->weights > 3 || params->splitting < 0 || params->splitting > 2) {
        g_batch_err = "invalid precision, weights, splitting or max_steps";
        return WENO_ERR_INVALID_ARG;
    }
    if (params->splitting == 1) {
        g_batch_err = "global Lax-Friedrichs splitting is not available for batches (use LLF or Roe)";
        return WENO_ERR_UNSUPPORTED;
    }
    for (int s = 0; s < 2; ++s) {
        const int bc = s == 0 ? d->bc_lo : d->bc_hi;
        if (bc != WENO_BC_TRANSMISSIVE && bc != WENO_BC_REFLECT && bc != WENO_BC_PERIODIC) {
            g_batch_err = "batched problems take transmissive, reflecting or periodic boundaries";
            return WENO_ERR_INVALID_ARG;
        }
    }
    if ((d->bc_lo == WENO_BC_PERIODIC) != (d->bc_hi == WENO_BC_PERIODIC)) {
        g_batch_err = "periodic boundaries must be paired";
        return WENO_ERR_INVALID_ARG;
    }
    const int cnt = d->count;
    std::vector<double> dx(cnt);
    for (int i = 0; i < cnt; ++i) {
        if (d->n[i] < 3 || !(d->hi[i] > d->lo[i]) || !(d->t_end[i] >= 0.0)) {
            g_batch_err = "instance with n < 3, hi <= lo or negative t_end";
            return WENO_ERR_INVALID_ARG;
        }
        dx[i] = (d->hi[i] - d->lo[i]) / d->n[i];
    }
    std::vector<int> order(cnt);
    std::iota(order.begin(), order.end(), 0);
    std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return d->n[a] > d->n[b]; });

    weno_batch* bt = new (std::nothrow) weno_batch();
    if (!bt) { g_batch_err = "out of host memory"; return WENO_ERR_CUDA; }
    bt->count = cnt;
    bt->p = *params;
    bt->prec = params->precision;
    bt->bc_lo[0] = d->bc_lo;
    bt->bc_hi[0] = d->bc_hi;
    bt->max_steps = d->max_steps > 0 ? d->max_steps : 0x7fffffff;
    bt->stream = (cudaStream_t)stream;
    bt->n_host.assign(d->n, d->n + cnt);
    return finish_create(bt, batch_setup(bt, d->n, nullptr, dx, dx, d->t_end, order), "weno_batch_create", out);
}

weno_status weno_batch2d_create(const weno_batch2d_desc* d, const weno_params* params, void* stream,
                                weno_batch** out)
{
    if (out) *out = nullptr;
    if (!d || !params || !out || d->count < 1 || !d->nx || !d->ny || !d->lo_x || !d->hi_x || !d->lo_y ||
        !d->hi_y || !d->t_end) {
        g_batch_err = "invalid 2D batch description";
        return WENO_ERR_INVALID_ARG;
    }
    if (params->precision < WENO_FP64 || params->precision > WENO_MIXED || d->max_steps < 0 ||
        params->weights < 0 || params->weights > 3 || params->splitting < 0 || params->splitting > 2) {
        g_batch_err = "invalid precision, weights, splitting or max_steps";
        return WENO_ERR_INVALID_ARG;
    }
    if (params->splitting == 1) {
        g_batch_err = "global Lax-Friedrichs splitting is not available for batches (use LLF or Roe)";
        return WENO_ERR_UNSUPPORTED;
    }
    for (int a = 0; a < 2; ++a) {
        for (int s = 0; s < 2; ++s) {
            const int bc = s == 0 ? d->bc_lo[a] : d->bc_hi[a];
            if (bc != WENO_BC_TRANSMISSIVE && bc != WENO_BC_REFLECT && bc != WENO_BC_PERIODIC) {
                g_batch_err = "batched problems take transmissive, reflecting or periodic boundaries";
                return WENO_ERR_INVALID_ARG;
            }
        }
        if ((d->bc_lo[a] == WENO_BC_PERIODIC) != (d->bc_hi[a] == WENO_BC_PERIODIC)) {
            g_batch_err = "periodic boundaries must be paired";
            return WENO_ERR_INVALID_ARG;
        }
    }
    const int cnt = d->count;
    std::vector<double> dx(cnt), dy(cnt), work(cnt);
    std::vector<int> lin(cnt);
    for (int i = 0; i < cnt; ++i) {
        if (d->nx[i] < 3 || d->ny[i] < 3 || !(d->hi_x[i] > d->lo_x[i]) || !(d->hi_y[i] > d->lo_y[i]) ||
            !(d->t_end[i] >= 0.0)) {
            g_batch_err = "instance with nx or ny < 3, hi <= lo or negative t_end";
            return WENO_ERR_INVALID_ARG;
        }
        dx[i] = (d->hi_x[i] - d->lo_x[i]) / d->nx[i];
        dy[i] = (d->hi_y[i] - d->lo_y[i]) / d->ny[i];
        lin[i] = std::max(d->nx[i], d->ny[i]);
        // work of a run ~ cells x steps, and the steps grow with the finer spacing
        work[i] = (double)d->nx[i] * d->ny[i] * lin[i];
    }
    std::vector<int> order(cnt);
    std::iota(order.begin(), order.end(), 0);
    std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return work[a] > work[b]; });

    weno_batch* bt = new (std::nothrow) weno_batch();
    if (!bt) { g_batch_err = "out of host memory"; return WENO_ERR_CUDA; }
    bt->dim = 2;
    bt->count = cnt;
    bt->p = *params;
    bt->prec = params->precision;
    for (int k = 0; k < 2; ++k) { bt->bc_lo[k] = d->bc_lo[k]; bt->bc_hi[k] = d->bc_hi[k]; }
    bt->max_steps = d->max_steps > 0 ? d->max_steps : 0x7fffffff;
    bt->stream = (cudaStream_t)stream;
    bt->n_host = lin;
    return finish_create(bt, batch_setup(bt, d->nx, d->ny, dx, dy, d->t_end, order), "weno_batch2d_create", out);
}

void weno_batch_destroy(weno_batch* bt)
{
    if (!bt) return;
    if (bt->stream) cudaStreamSynchronize(bt->stream);
    else cudaDeviceSynchronize();
    batch_free(bt);
    delete bt;
}

const char* weno_batch_last_error(const weno_batch* bt) { return bt ? bt->err.c_str() : g_batch_err.c_str(); }

weno_status weno_batch_run(weno_batch* bt, void* U_dev)
{
    if (!bt || !U_dev) return WENO_ERR_INVALID_ARG;
    if (!bt->graph || bt->graph_U != U_dev) {
        if (bt->graph) cudaGraphExecDestroy(bt->graph);
        bt->graph = nullptr;
        cudaGraph_t g = nullptr;
        BCK(cudaStreamBeginCapture(bt->cap, cudaStreamCaptureModeRelaxed));
        cudaError_t e = enqueue_run(bt, U_dev, bt->max_steps, 1, bt->cap);
        cudaError_t e2 = cudaStreamEndCapture(bt->cap, &g);
        if (e != cudaSuccess || e2 != cudaSuccess) {
            if (g) cudaGraphDestroy(g);
            bt->err = std::string("batch graph capture: ") + cudaGetErrorString(e != cudaSuccess ? e : e2);
            return WENO_ERR_CUDA;
        }
        e = cudaGraphInstantiate(&bt->graph, g, 0);
        cudaGraphDestroy(g);
        if (e != cudaSuccess) {
            bt->err = std::string("cudaGraphInstantiate: ") + cudaGetErrorString(e);
            return WENO_ERR_CUDA;
        }
        bt->graph_U = U_dev;
    }
    BCK(cudaGraphLaunch(bt->graph, bt->stream));
    return WENO_OK;
}

weno_status weno_batch_results(weno_batch* bt, int* status, long long* steps, double* t)
{
    if (!bt) return WENO_ERR_INVALID_ARG;
    if (status) BCK(cudaMemcpyAsync(status, bt->status, sizeof(int) * bt->count, cudaMemcpyDeviceToHost, bt->stream));
    if (steps) BCK(cudaMemcpyAsync(steps, bt->steps, sizeof(long long) * bt->count, cudaMemcpyDeviceToHost, bt->stream));
    if (t) BCK(cudaMemcpyAsync(t, bt->t_out, sizeof(double) * bt->count, cudaMemcpyDeviceToHost, bt->stream));
    int abort = 0;
    BCK(cudaMemcpyAsync(&abort, &reinterpret_cast<wis::BatchCtrl*>(bt->run)->abort, sizeof(int),
                        cudaMemcpyDeviceToHost, bt->stream));
    BCK(cudaStreamSynchronize(bt->stream));
    if (abort) {
        bt->err = "a wait of the batch kernel for its next task ran out; the states are not valid";
        return WENO_ERR_TIMEOUT;
    }
    if (status)
        for (int i = 0; i < bt->count; ++i)
            if (status[i] != WENO_OK) {
                bt->err = "at least one instance reached a non-physical state";
                return WENO_ERR_NONPHYSICAL;
            }
    return WENO_OK;
}

weno_status weno_batch_weno_face_count(weno_batch* bt, unsigned long long* count, int reset)
{
    if (!bt) return WENO_ERR_INVALID_ARG;
    unsigned long long v = 0;
    BCK(cudaMemcpyAsync(&v, bt->wcount, sizeof(v), cudaMemcpyDeviceToHost, bt->stream));
    BCK(cudaStreamSynchronize(bt->stream));
    if (count) *count = v;
    if (reset) {
        BCK(cudaMemsetAsync(bt->wcount, 0, sizeof(unsigned long long), bt->stream));
        BCK(cudaStreamSynchronize(bt->stream));
    }
    return WENO_OK;
}

weno_status weno_batch_set_config(weno_batch* bt, int variant, int blocks_per_sm, int* blocks)
{
    if (!bt) return WENO_ERR_INVALID_ARG;
    if (variant < 0 || variant >= wis::kBatchVariants || blocks_per_sm < 0) {
        bt->err = "set_config: variant must be 0, 1 or 2 and blocks_per_sm >= 0";
        return WENO_ERR_INVALID_ARG;
    }
    const weno_status st = set_variant(bt, variant, blocks_per_sm);
    if (st == WENO_OK && blocks) *blocks = bt->blocks;
    return st;
}

weno_status weno_batch_set_launch(weno_batch* bt, int ctas)
{
    if (!bt) return WENO_ERR_INVALID_ARG;
    if (ctas < 0) {
        bt->err = "set_launch: negative number of CTAs";
        return WENO_ERR_INVALID_ARG;
    }
    bt->ctas = ctas;
    return set_variant(bt, bt->variant, bt->residency);
}

weno_status weno_batch_set_wait(weno_batch* bt, int polls)
{
    if (!bt) return WENO_ERR_INVALID_ARG;
    if (polls < 0) {
        bt->err = "set_wait: negative number of polls";
        return WENO_ERR_INVALID_ARG;
    }
    bt->polls = polls > 0 ? std::min(polls, 1 << 30) : wis::kTaskPolls;   // the counter of polls stays an int
    if (bt->graph) cudaGraphExecDestroy(bt->graph);   // it holds the old number
    bt->graph = nullptr;
    return WENO_OK;
}

weno_status weno_batch_autotune(weno_batch* bt, const void* U_dev, int trial_steps, int* choice)
{
    if (!bt || !U_dev || trial_steps < 1) return WENO_ERR_INVALID_ARG;
    // trial steps per instance in proportion to its cells: a full run's step
    // count grows with the cell count (the CFL step shrinks with dx), so its
    // work grows like N^2, and the trial keeps that shape
    const int nmax = *std::max_element(bt->n_host.begin(), bt->n_host.end());
    std::vector<int> tc(bt->count);
    for (int i = 0; i < bt->count; ++i)
        tc[i] = std::max(1, (int)std::ceil((double)trial_steps * bt->n_host[i] / nmax));
    BCK(cudaMemcpy(bt->trial_caps, tc.data(), sizeof(int) * bt->count, cudaMemcpyHostToDevice));
    // the trials start from a scratch copy advanced to half of each
    // instance's end time: the cost of a step depends on how far the waves
    // have spread, and trials from the initial jumps rank the configurations
    // unlike full runs do (they favour small tiles that lose on developed
    // solutions)
    const size_t sbytes = (size_t)bt->total * bt->esz;
    void* Us = nullptr;
    double* t_half = nullptr;
    BCK(cudaMalloc(&Us, sbytes));
    if (cudaMalloc(&t_half, sizeof(double) * bt->count) != cudaSuccess) {
        cudaFree(Us);
        bt->err = "autotune: out of device memory";
        return WENO_ERR_CUDA;
    }
    std::vector<double> th(bt->count);
    cudaError_t ce = cudaMemcpy(th.data(), bt->t_end, sizeof(double) * bt->count, cudaMemcpyDeviceToHost);
    for (double& x : th) x *= 0.5;
    if (ce == cudaSuccess)
        ce = cudaMemcpy(t_half, th.data(), sizeof(double) * bt->count, cudaMemcpyHostToDevice);
    if (ce == cudaSuccess) ce = cudaMemcpyAsync(Us, U_dev, sbytes, cudaMemcpyDeviceToDevice, bt->stream);
    if (ce == cudaSuccess) {
        BatchArgs b = batch_args(bt, Us, bt->max_steps, 1);
        b.t_end = t_half;
        ce = launch_run(bt, b, bt->stream);
    }
    if (ce == cudaSuccess) ce = cudaStreamSynchronize(bt->stream);
    cudaFree(t_half);
    if (ce != cudaSuccess) {
        cudaFree(Us);
        bt->err = std::string("autotune: developing the trial state: ") + cudaGetErrorString(ce);
        return WENO_ERR_CUDA;
    }
    cudaEvent_t e0, e1;
    if (cudaEventCreate(&e0) != cudaSuccess) { cudaFree(Us); bt->err = "cudaEventCreate"; return WENO_ERR_CUDA; }
    if (cudaEventCreate(&e1) != cudaSuccess) {
        cudaEventDestroy(e0); cudaFree(Us); bt->err = "cudaEventCreate"; return WENO_ERR_CUDA;
    }
    float best = 1e30f;
    int best_v = bt->variant, best_cap = 0;
    const int caps[3] = {0, 4, 2};   // 0 = as many CTAs per SM as fit
    weno_status st = WENO_OK;
    for (int v = 0; v < wis::kBatchVariants && st == WENO_OK; ++v) {
        for (int c = 0; c < 3 && st == WENO_OK; ++c) {
            st = set_variant(bt, v, caps[c]);
            if (st != WENO_OK) break;
            float ms = 1e30f;
            for (int r = 0; r < 2; ++r) {   // first run loads the kernel
                if (cudaEventRecord(e0, bt->stream) != cudaSuccess ||
                    enqueue_run(bt, Us, trial_steps, 0, bt->stream, bt->trial_caps) != cudaSuccess ||
                    cudaEventRecord(e1, bt->stream) != cudaSuccess || cudaEventSynchronize(e1) != cudaSuccess) {
                    bt->err = "batch autotune launch failed";
                    st = WENO_ERR_CUDA;
                    break;
                }
                cudaEventElapsedTime(&ms, e0, e1);
            }
            if (st == WENO_OK && ms < best) { best = ms; best_v = v; best_cap = caps[c]; }
        }
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    cudaFree(Us);
    if (st != WENO_OK) return st;
    st = set_variant(bt, best_v, best_cap);
    if (choice) { choice[0] = best_v; choice[1] = bt->blocks; }
    return st;
}

weno_status weno_batch_solve(const weno_batch_desc* d, const weno_params* params, void* stream, void* U_dev,
                             int* per_instance)
{
    weno_batch* bt = nullptr;
    weno_status st = weno_batch_create(d, params, stream, &bt);
    if (st != WENO_OK) return st;
    st = weno_batch_run(bt, U_dev);
    if (st == WENO_OK) st = weno_batch_results(bt, per_instance, nullptr, nullptr);
    if (st != WENO_OK && st != WENO_ERR_NONPHYSICAL) g_batch_err = bt->err;
    weno_batch_destroy(bt);
    return st;
}

}  // extern "C"
