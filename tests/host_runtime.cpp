// A CUDA runtime of host memory for testing the library's host code
// (csrc/recon_api.cu, csrc/recon_sched.cu) without a GPU: the runtime calls those
// files make, and stand-ins for the kernels' launchers. It is as late as CUDA
// allows: queued work runs, in the order in which it was queued, only when a
// call waits for it, so a source that is refilled or freed too early shows in the
// result. Freed memory stays mapped but is poisoned, and an access to it is counted
// (ht_faults). The stand-ins reconstruct by J <- I (a violation is found first).
#include <algorithm>
#include <climits>
#include <cstdlib>
#include <cstring>
#include <deque>
#include <functional>
#include <map>
#include <vector>
#include <cuda.h>
#include <cuda_runtime_api.h>

#include "recon.h"
#include "recon_internal.h"
#include "recon_dt.h"
#include "recon_forest.h"
#include "recon_learn.h"

struct CUevent_st { size_t last = 0; double at = 0.0; };
struct Op { std::function<void()> f; cudaEvent_t records; };
struct CUstream_st {
    std::vector<Op> *capture = nullptr;
    size_t last = 0;   // number of its latest operation
};
struct CUgraph_st { std::vector<Op> ops; };
struct CUgraphExec_st { std::vector<Op> ops; };

namespace {

std::deque<std::function<void()>> queue;
size_t queued = 0, done = 0;             // operations so far; the queue holds done + 1 .. queued
std::map<unsigned char *, size_t> live, dead;
size_t dev_bytes = 0, dev_limit = SIZE_MAX, pinned_limit = SIZE_MAX;
cudaError_t last_error = cudaSuccess;
std::map<unsigned char *, size_t> dev;   // sizes of device allocations
int faults = 0;
int broken = 0;                          // waits for a stream under capture
double now_ms = 0.0;                     // device clock: a kernel takes a nanosecond a pixel
int n_merging = 0, n_wavefront = 0, n_graph = 0, n_plan = 0;
std::vector<int> orders, steps;          // sample orders of the epochs trained; numbers of the single steps
bool fits = true;                        // the training cluster can be placed

void run_to(size_t n)
{
    while (done < n && !queue.empty()) {
        auto f = std::move(queue.front());
        queue.pop_front();
        ++done;
        f();
    }
}

void put(cudaStream_t s, std::function<void()> f, cudaEvent_t records = nullptr)
{
    if (s->capture) {
        s->capture->push_back(Op{std::move(f), records});
        return;
    }
    queue.push_back(std::move(f));
    s->last = ++queued;
    if (records) records->last = queued;
}

bool overlaps(const std::map<unsigned char *, size_t> &m, const void *p, size_t n)
{
    auto it = m.upper_bound((unsigned char *)p + (n ? n - 1 : 0));
    if (it == m.begin()) return false;
    --it;
    return it->first + it->second > (unsigned char *)p;
}

void touch(const void *p, size_t n)
{
    if (overlaps(dead, p, n)) ++faults;
}

void *alloc(size_t n)
{
    n = std::max<size_t>(n, 16);
    unsigned char *p = (unsigned char *)aligned_alloc(256, (n + 255) / 256 * 256);
    memset(p, 0, n);
    live[p] = n;
    return p;
}

void release(void *p)
{
    if (!p) return;
    auto it = live.find((unsigned char *)p);
    if (it == live.end()) { ++faults; return; }
    memset(p, 0xDD, it->second);
    dead[it->first] = it->second;
    live.erase(it);
}

struct Pixels { const uint8_t *I; uint8_t *J; int H, W, pitch, dual, fill; };

// one tile: false when the marker is on the wrong side of the mask
bool reconstruct(const Pixels &t, bool check)
{
    const size_t n = (size_t)(t.H - 1) * t.pitch + t.W;
    touch(t.I, n);
    touch(t.J, n);
    if (check && !t.fill)
        for (int y = 0; y < t.H; ++y)
            for (int x = 0; x < t.W; ++x) {
                const int i = t.I[(size_t)y * t.pitch + x], j = t.J[(size_t)y * t.pitch + x];
                if (t.dual ? j < i : j > i) return false;
            }
    for (int y = 0; y < t.H; ++y) memcpy(t.J + (size_t)y * t.pitch, t.I + (size_t)y * t.pitch, t.W);
    now_ms += 1e-6 * t.H * t.W;
    return true;
}

void fail(rk::Ctl *ctl, int *tile_err, int index)
{
    tile_err[index] = RECON_EMARKER;
    ctl->err_tile = std::min(ctl->err_tile, index);
}

}  // namespace

// ---- what the tests read and set
extern "C" int ht_faults() { return faults; }
extern "C" int ht_broken_captures() { return broken; }
extern "C" int ht_graph_nodes(cudaGraph_t g) { return (int)g->ops.size(); }
extern "C" void ht_device_limit(size_t bytes) { dev_limit = bytes; }
extern "C" void ht_pinned_limit(size_t bytes) { pinned_limit = bytes; }   // of one allocation
extern "C" size_t ht_device_bytes() { return dev_bytes; }
extern "C" void ht_counts(int *out)
{
    const int v[4] = {n_merging, n_wavefront, n_graph, n_plan};
    memcpy(out, v, sizeof(v));
}
extern "C" int ht_orders(int *out, int max)
{
    memcpy(out, orders.data(), sizeof(int) * std::min<size_t>(max, orders.size()));
    return (int)orders.size();
}
extern "C" int ht_steps(int *out, int max)
{
    memcpy(out, steps.data(), sizeof(int) * std::min<size_t>(max, steps.size()));
    return (int)steps.size();
}
extern "C" void ht_train_fits(int yes) { fits = yes; }

// ---- runtime
extern "C" {
cudaError_t cudaGetDeviceCount(int *n) { *n = 1; return cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaGetLastError()
{
    const cudaError_t e = last_error;
    last_error = cudaSuccess;
    return e;
}
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr, int) { *v = 4; return cudaSuccess; }
cudaError_t cudaGetDriverEntryPointByVersion(const char *, void **, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult *)
{
    return cudaErrorNotSupported;   // no tensor maps: plain loads
}
cudaError_t cudaMalloc(void **p, size_t n)
{
    if (dev_bytes + n > dev_limit) return last_error = cudaErrorMemoryAllocation;
    *p = alloc(n);
    dev[(unsigned char *)*p] = n;
    dev_bytes += n;
    return cudaSuccess;
}
cudaError_t cudaFree(void *p)
{
    run_to(queued);
    auto it = dev.find((unsigned char *)p);
    if (it != dev.end()) {
        dev_bytes -= it->second;
        dev.erase(it);
    }
    release(p);
    return cudaSuccess;
}
cudaError_t cudaMallocHost(void **p, size_t n)
{
    if (n > pinned_limit) return last_error = cudaErrorMemoryAllocation;
    *p = alloc(n);
    return cudaSuccess;
}
cudaError_t cudaHostAlloc(void **p, size_t n, unsigned) { *p = alloc(n); return cudaSuccess; }
cudaError_t cudaFreeHost(void *p) { release(p); return cudaSuccess; }
cudaError_t cudaHostGetDevicePointer(void **d, void *h, unsigned) { *d = h; return cudaSuccess; }
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, cudaMemcpyKind)
{
    touch(d, n);
    touch(s, n);
    memcpy(d, s, n);
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind, cudaStream_t st)
{
    put(st, [=] { touch(d, n); touch(s, n); memcpy(d, s, n); });
    return cudaSuccess;
}
cudaError_t cudaMemcpy2DAsync(void *d, size_t dp, const void *s, size_t sp, size_t w, size_t h, cudaMemcpyKind,
                              cudaStream_t st)
{
    put(st, [=] {
        for (size_t y = 0; y < h; ++y) memcpy((char *)d + y * dp, (const char *)s + y * sp, w);
    });
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void *d, int v, size_t n, cudaStream_t st)
{
    put(st, [=] { touch(d, n); memset(d, v, n); });
    return cudaSuccess;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) { *s = new CUstream_st; return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t s) { delete s; return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t s)
{
    if (s->capture) {
        ++broken;
        return cudaErrorStreamCaptureUnsupported;
    }
    run_to(s->last);
    return cudaSuccess;
}
cudaError_t cudaStreamQuery(cudaStream_t s) { return s->last <= done ? cudaSuccess : cudaErrorNotReady; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }   // one queue: in order
cudaError_t cudaStreamIsCapturing(cudaStream_t s, cudaStreamCaptureStatus *st)
{
    *st = s->capture ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
    return cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t *e) { *e = new CUevent_st; return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) { *e = new CUevent_st; return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t e) { delete e; return cudaSuccess; }
cudaError_t cudaEventRecordWithFlags(cudaEvent_t e, cudaStream_t s, unsigned)
{
    put(s, [=] { e->at = now_ms; }, e);
    return cudaSuccess;
}
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) { return cudaEventRecordWithFlags(e, s, 0); }
cudaError_t cudaEventSynchronize(cudaEvent_t e) { run_to(e->last); return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t a, cudaEvent_t b)
{
    *ms = (float)(b->at - a->at);
    return cudaSuccess;
}
cudaError_t cudaStreamBeginCapture(cudaStream_t s, cudaStreamCaptureMode)
{
    s->capture = new std::vector<Op>;
    return cudaSuccess;
}
cudaError_t cudaStreamEndCapture(cudaStream_t s, cudaGraph_t *g)
{
    *g = new CUgraph_st{*s->capture};
    delete s->capture;
    s->capture = nullptr;
    return cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t *x, cudaGraph_t g, unsigned long long)
{
    *x = new CUgraphExec_st{g->ops};
    return cudaSuccess;
}
cudaError_t cudaGraphDestroy(cudaGraph_t g) { delete g; return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t x) { delete x; return cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t x, cudaStream_t s)
{
    ++n_graph;
    for (auto &op : x->ops) put(s, op.f, op.records);
    return cudaSuccess;
}

// ---- wavefront kernels
size_t rk_smem_bytes(int) { return 0; }
cudaError_t rk_configure(int, int *ctas) { *ctas = 1; return cudaSuccess; }
cudaError_t rk_launch_fill(const rk::TileDesc *, const int *, int, cudaStream_t) { return cudaSuccess; }
cudaError_t rk_launch_init(int, const rk::Params *Pp, cudaStream_t st)
{
    const rk::Params P = *Pp;
    put(st, [=] {
        memset(P.ctl, 0, sizeof(rk::Ctl));
        P.ctl->err_tile = INT_MAX;
        touch(P.tile_err, sizeof(int) * P.ntiles);
        touch(P.work, sizeof(rk::Work) * P.ntiles);
        memset(P.tile_err, 0, sizeof(int) * P.ntiles);
        memset(P.work, 0, sizeof(rk::Work) * P.ntiles);
    });
    return cudaSuccess;
}
cudaError_t rk_launch_main(int, int, const rk::Params *Pp, cudaStream_t st)
{
    const rk::Params P = *Pp;
    put(st, [=] {
        ++n_wavefront;
        for (int t = 0; t < P.ntiles; ++t) {
            const rk::TileDesc &d = P.tiles[t];
            if (!reconstruct(Pixels{d.I, d.J, d.H, d.W, d.pitch, d.dual, d.fill}, P.check)) fail(P.ctl, P.tile_err, t);
            P.work[t].visits += (unsigned long long)d.nbx * d.nby;
            P.work[t].scan_rows += d.H;
        }
    });
    return cudaSuccess;
}

// ---- merging kernels
cudaError_t rf_configure() { return cudaSuccess; }
cudaError_t rf_launch(int, const rf::Params *Pp, cudaStream_t st)
{
    const rf::Params P = *Pp;
    put(st, [=] {
        ++n_merging;
        touch(P.px, rf::scratch_bytes(P.nblocks));
        if (P.next) {
            memset(P.next, 0, sizeof(*P.next));
            P.next->ctl.err_tile = INT_MAX;
        }
        for (int t = 0; t < P.ntiles; ++t) {
            const rf::Tile &d = P.tiles ? P.tiles[t] : P.one;
            if (!reconstruct(Pixels{d.I, d.J, d.H, d.W, d.pitch, d.dual, d.fill}, P.check))
                fail(P.ctl, P.tile_err, d.index);
            P.work[d.index].visits += (unsigned long long)d.nbx * d.nby;
        }
    });
    return cudaGetLastError();   // as after a launch
}
}

// ---- cost model, distance transform
size_t rl_features_scratch(int n) { return 64 * (size_t)n; }
size_t rl_features_stage(int n) { return 64 * (size_t)n; }
cudaError_t rl_features(const rl_tile *, int n, void *, size_t, float *feat, int *, int, cudaStream_t st, void *, size_t)
{
    put(st, [=] { memset(feat, 0, sizeof(float) * NFEAT * n); });
    return cudaSuccess;
}
cudaError_t rl_forward(const float *, const float *, int n, float *Y, cudaStream_t st)
{
    ++n_plan;
    put(st, [=] { memset(Y, 0, sizeof(float) * 2 * n); });
    return cudaSuccess;
}
cudaError_t rl_grad(const float *, const float *, const float *, const int *idx, int n, float *grad, float *loss,
                    cudaStream_t st)
{
    put(st, [=] {
        touch(idx, sizeof(int) * n);
        orders.insert(orders.end(), idx, idx + n);
        grad[0] += 1.0f;
        *loss += 1.0f;
    });
    return cudaSuccess;
}
cudaError_t rl_adam(float *, float *grad, float *, float *, int t, float, cudaStream_t st)
{
    put(st, [=] {
        faults += grad[0] != 1.0f;
        grad[0] = 0.0f;
        steps.push_back(t);
    });
    return cudaSuccess;
}
bool rl_train_fits() { return fits; }
cudaError_t rl_train_epoch(float *, float *, float *, const float *, const float *, const int *idx, int n, int, int,
                           float, float *loss, cudaStream_t st)
{
    put(st, [=] {
        touch(idx, sizeof(int) * n);
        orders.insert(orders.end(), idx, idx + n);
        *loss += 1.0f;
    });
    return cudaGetLastError();
}
size_t dt_scratch_bytes(int H, int W) { return (size_t)H * W; }
int dt_run(const uint8_t *, int, int, int *, unsigned *, void *, unsigned, int, cudaStream_t) { return DT_OK; }

// ---- entry points of the other files
extern "C" int recon_run_noalloc(const uint8_t *, uint8_t *, int, int, int, void *) { return RECON_ECUDA; }
extern "C" int recon_checks(int *, unsigned *, unsigned *, int) { return 1; }
extern "C" int recon_mb_threads(int) { return -RECON_ECUDA; }
extern "C" int recon_mb_random(const void *, int, uint64_t, int, uint64_t, uint64_t *, float *) { return RECON_ECUDA; }
extern "C" int recon_mb_atomic(unsigned *, int, int, float *) { return RECON_ECUDA; }
