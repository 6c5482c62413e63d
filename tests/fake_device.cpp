// A stand-in for the CUDA runtime and the kernels, linked with the host
// runtime's own sources (cosm_runtime.cu, cosm_server.cu, cosm_graph.cpp) for
// tests that need no GPU. Device memory is host memory, copies happen at once
// and kernels do not run; every launch checks what it was given instead: that
// no copy from pageable host memory is still on its way on the legacy stream
// when another stream launches, that the tables a kernel walks are those of
// its tile width and thread count (read back edge by edge), and that a state is
// read in the layout it was written in. A test can let a later cudaMalloc or
// the creation of threads fail.
#include <cuda_runtime.h>
#include <dlfcn.h>
#include <errno.h>
#include <pthread.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

#include <algorithm>
#include <array>
#include <atomic>
#include <map>
#include <mutex>
#include <set>
#include <string>
#include <vector>

#include "cosm.h"
#include "cosm_edges.h"
#include "cosm_internal.h"
#include "cosm_patch.h"

using namespace cosm;

namespace {

std::recursive_mutex mu;
std::map<const char *, size_t> blocks;  // device allocations
int64_t live = 0, peak = 0, fail_malloc = 0;
std::atomic<int> fail_threads{0}, fail_graphs{0};
std::atomic<int64_t> queries{0};  // of occupancies, since the last report
bool pending = false;     // a legacy-stream copy or set that nothing has waited for
uintptr_t next_handle = 0x1000;
struct Report {
    int64_t unordered, bad, launches, threads, K, shape, ragged, format;
} rep;
std::string why;

void bad(const char *what)
{
    ++rep.bad;
    if (why.empty()) why = what;
}
bool inside(const void *p, size_t bytes)
{
    auto it = blocks.upper_bound(static_cast<const char *>(p));
    if (it == blocks.begin()) return false;
    --it;
    return static_cast<const char *>(p) + bytes <= it->first + it->second;
}
void launched(void *stream)
{
    ++rep.launches;
    if (stream && pending) ++rep.unordered;
}
int model_occupancy(int threads, size_t smem)
{
    ++queries;
    if (threads < 1 || threads > 1024 || smem > 227 * 1024) return 0;
    return (int)std::min<size_t>(1024 / (size_t)((threads + 31) / 32 * 32), 228 * 1024 / (smem + 1024));
}

// The state of a launch: tagged with its layout, checked where it is loaded
// (a zero tag: copied from the host).
void touch_state(const InstView &v, int K, bool loads)
{
    int64_t tag[2] = {K, v.state_tile_stride}, was[2];
    if (!inside(v.state, (size_t)v.state_tile_stride * 2)) return bad("state outside its allocation");
    memcpy(was, v.state, sizeof(was));
    if (loads && was[0] && memcmp(was, tag, sizeof(tag))) bad("state read in another layout than it was written in");
    memcpy(v.state, tag, sizeof(tag));
}

// Every edge of every colour, in the rows of the warps a launch of `threads` has.
void check_table(const InstView &v, int storage, int K, int threads, int format)
{
    const int E = K * (storage == COSM_F32 ? 4 : 2), fmt = format & ~EDGES_EACH, RW = fmt == EDGES_WEIGHT ? 2 : 1;
    const int W = threads / 32, nc = v.n_colours;
    if (threads % 32 || W < 1) return bad("a record table without whole warps");
    if (!inside(v.counts, (size_t)W * (nc + 1) * 4) || !inside(v.starts, (size_t)W * 4))
        return bad("counts or starts of another thread count");
    using Edge = std::array<int, 4>;
    std::vector<Edge> want, got;
    for (int c = 0, k = 0; c < v.C; ++c) {
        for (int e = v.off[c]; e < v.off[c + 1]; ++e)
            want.push_back({k, (int)(v.ij[e] & 0xFFFF), (int)(v.ij[e] >> 16), v.w[e]});
        k += v.off[c + 1] > v.off[c];
    }
    for (int w = 0; w < W; ++w) {
        const uint32_t *counts = v.counts + (size_t)w * (nc + 1), *p = v.rec + v.starts[w], *const first = p;
        if (counts[nc] != counts[0]) return bad("a warp's counts do not close");
        int64_t rows = 0;
        for (int k = 0; k < nc; ++k) rows += counts[k] & ~kPartial;
        const int64_t ahead = kRowsAhead * 32 * RW, words = rows * 32 * RW;
        if (v.starts[w] < 0 || !inside(p, (size_t)(words + ahead) * 4)) return bad("a warp's rows outside the table");
        for (int k = 0; k < nc; ++k) {
            const int n = (int)(counts[k] & ~kPartial);
            for (int r = 0; r < n; ++r) {
                int empty = 0;
                for (int lane = 0; lane < 32; ++lane, p += RW) {
                    const uint32_t r0 = p[0], r1 = p[RW - 1];
                    if (r0 == kNoEdge) {
                        ++empty;
                        continue;
                    }
                    Edge e{k, 0, 0, 0};
                    if (fmt == EDGES_SIGN) {
                        e = {k, (int)(r0 >> 1 & 0x7FFF), (int)(r0 >> 16), r0 & 1 ? -1 : 1};
                    } else if (fmt == EDGES_PACK) {
                        e = {k, (int)(r0 & 0x3FFFF & ~(uint32_t)(E - 1)) / E, (int)(r0 >> 18), (int)(r0 & (E - 1)) - E / 2};
                    } else {
                        const uint32_t top = r1 & 0xFFFC0000u;
                        float f;
                        memcpy(&f, &top, 4);
                        e = {k, (int)(r0 / E), (int)((r1 & 0x3FFFF) / E), storage == COSM_Q16 ? (int32_t)r1 >> 18 : (int)f};
                    }
                    got.push_back(e);
                }
                if (empty && !(r == n - 1 && (counts[k] & kPartial) && empty < 32)) return bad("an empty place in a full row");
            }
        }
        if (memcmp(p, first, (size_t)std::min(words, ahead) * 4)) return bad("the rows ahead are not the first ones");
    }
    std::sort(want.begin(), want.end());
    std::sort(got.begin(), got.end());
    if (want != got) bad("the table's edges are not the instance's");
}

void check_patch(const InstView &v, int shape, int ragged, int threads)
{
    const int R = kPatchR[shape], C = kPatchC[shape], T = v.pgr * v.pgc, words = (8 * R * C + 31) / 32;
    if (!v.pwt || !inside(v.pwt, (size_t)words * T * 4)) return bad("a patch shape without its weights");
    if (T > threads || v.pgr * R - (v.pgr - v.pfr) != v.Q / v.Wd || v.pgc * C - (v.pgc - v.pfc) != v.Wd ||
        T * (2 * R + 2 * C - 1) > v.n || ragged != (v.pgr != v.pfr || v.pgc != v.pfc))
        bad("a patch grid that is not the lattice's");
}

void check_launch(int storage, int K, int shape, int ragged, int format, int threads, const KernelArgs *run,
                  const BatchArgs *queue, void *stream)
{
    std::lock_guard<std::recursive_mutex> lock(mu);
    launched(stream);
    rep.threads = threads;
    rep.K = K;
    rep.shape = shape;
    rep.ragged = ragged;
    rep.format = format;
    if (threads < 32) bad("fewer threads than a warp");
    auto one = [&](const InstView &v, bool loads) {
        if (v.K != K) bad("a launch of another tile width");
        if (format >= 0) check_table(v, storage, K, threads, format);
        if (shape >= 0) check_patch(v, shape, ragged, threads);
        touch_state(v, K, loads);
    };
    if (run) one(run->v, (run->segs[run->seg_off[0]].flags & SEG_LOAD) != 0);
    std::set<int> seen;
    for (int u = 0; queue && u < queue->n_units; ++u)
        if (seen.insert(queue->units[u].inst).second)
            one(queue->insts[queue->units[u].inst], (queue->units[u].flags & SEG_LOAD) != 0);
}

int patch(int storage, int K, const PatchCall &c)
{
    if (c.what == PatchCall::OCCUPANCY)
        return c.threads > patch_max_threads(kPatchR[c.shape], kPatchC[c.shape], K * (storage == COSM_F32 ? 4 : 2))
                   ? 0
                   : model_occupancy(c.threads, c.smem);
    check_launch(storage, K, c.shape, c.ragged, -1, c.threads, c.run, c.queue, c.stream);
    return 0;
}
int edges(int storage, const EdgesCall &c)
{
    if (c.what == EdgesCall::OCCUPANCY) return model_occupancy(c.threads, c.smem);
    check_launch(storage, c.K, -1, 0, c.format, c.threads, c.run, c.queue, c.stream);
    return 0;
}

}  // namespace

namespace cosm {

int patch_call_f32_k2(const PatchCall &c) { return patch(COSM_F32, 2, c); }
int patch_call_f16_k2(const PatchCall &c) { return patch(COSM_F16, 2, c); }
int patch_call_f16_k4(const PatchCall &c) { return patch(COSM_F16, 4, c); }
int patch_call_bf16_k2(const PatchCall &c) { return patch(COSM_BF16, 2, c); }
int patch_call_bf16_k4(const PatchCall &c) { return patch(COSM_BF16, 4, c); }
int patch_call_q16_k2(const PatchCall &c) { return patch(COSM_Q16, 2, c); }
int patch_call_q16_k4(const PatchCall &c) { return patch(COSM_Q16, 4, c); }
int edges_call_f32(const EdgesCall &c) { return edges(COSM_F32, c); }
int edges_call_f16(const EdgesCall &c) { return edges(COSM_F16, c); }
int edges_call_bf16(const EdgesCall &c) { return edges(COSM_BF16, c); }
int edges_call_q16(const EdgesCall &c) { return edges(COSM_Q16, c); }

size_t sweep_smem_bytes(int storage, int K, int n, int P, int mode)
{
    const auto up = [](size_t b) { return (b + 15) & ~(size_t)15; };
    return up((size_t)n * K * (storage == COSM_F32 ? 4 : 2)) + (mode == MODE_ACCUM_ ? up((size_t)n * K * 4) : 0) +
           up((size_t)K * (P + 1) * 4) + 20 * (size_t)K;
}
int sweep_occupancy(int, int, int, int threads, size_t smem) { return model_occupancy(threads, smem); }
int batch_occupancy(int, int, int, int threads, size_t smem) { return model_occupancy(threads, smem); }
int sweep_launch(const LaunchCfg &c, const KernelArgs &a, void *stream)
{
    check_launch(c.storage, c.K, -1, 0, -1, c.threads, &a, nullptr, stream);
    return 0;
}
int batch_launch(int storage, int K, int, int, int threads, size_t, const BatchArgs &b, void *stream)
{
    check_launch(storage, K, -1, 0, -1, threads, nullptr, &b, stream);
    return 0;
}
int finalize_launch(const FinalArgs &a, void *stream)
{
    std::lock_guard<std::recursive_mutex> lock(mu);
    launched(stream);
    memset(a.best, 0, 32);
    memset(a.spins, 1, (size_t)a.n);
    return 0;
}
int batch_finalize_launch(int, const InstView *, const BatchFinal *, void *stream)
{
    std::lock_guard<std::recursive_mutex> lock(mu);
    launched(stream);
    return 0;
}
int opt_readout_launch(const OptArgs &, int, void *stream)
{
    std::lock_guard<std::recursive_mutex> lock(mu);
    launched(stream);
    return 0;
}
static int state_launch(const StateArgs &a, bool loads, void *stream)
{
    std::lock_guard<std::recursive_mutex> lock(mu);
    launched(stream);
    InstView v;
    memset(&v, 0, sizeof(v));
    v.state = a.state;
    v.state_tile_stride = a.stride;
    if (!a.t0) touch_state(v, a.K, loads);
    return 0;
}
int state_export_launch(const StateArgs &a, int, void *stream) { return state_launch(a, true, stream); }
int state_import_launch(const StateArgs &a, void *stream) { return state_launch(a, false, stream); }

}  // namespace cosm

// ---------------------------------------------------------------- CUDA runtime
extern "C" {

cudaError_t cudaMalloc(void **p, size_t bytes)
{
    std::lock_guard<std::recursive_mutex> lock(mu);
    if (fail_malloc > 0 && --fail_malloc == 0) return cudaErrorMemoryAllocation;
    *p = calloc(1, std::max<size_t>(bytes, 16));
    blocks[static_cast<char *>(*p)] = bytes;
    live += (int64_t)bytes;
    peak = std::max(peak, live);
    return cudaSuccess;
}
cudaError_t cudaFree(void *p)
{
    std::lock_guard<std::recursive_mutex> lock(mu);
    auto it = blocks.find(static_cast<char *>(p));
    if (it == blocks.end()) return cudaErrorInvalidValue;
    live -= (int64_t)it->second;
    blocks.erase(it);
    free(p);
    return cudaSuccess;
}
cudaError_t cudaMemcpy(void *d, const void *s, size_t bytes, cudaMemcpyKind)
{
    std::lock_guard<std::recursive_mutex> lock(mu);
    memmove(d, s, bytes);
    pending = inside(d, bytes);  // a copy to the host waits for what went before it
    return cudaSuccess;
}
cudaError_t cudaMemset(void *d, int v, size_t bytes)
{
    std::lock_guard<std::recursive_mutex> lock(mu);
    memset(d, v, bytes);
    pending = true;
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t bytes, cudaMemcpyKind, cudaStream_t)
{
    memmove(d, s, bytes);
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void *d, int v, size_t bytes, cudaStream_t)
{
    memset(d, v, bytes);
    return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t s)
{
    std::lock_guard<std::recursive_mutex> lock(mu);
    if (!s) pending = false;
    return cudaSuccess;
}
cudaError_t cudaDeviceSynchronize(void) { return cudaStreamSynchronize(nullptr); }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned)
{
    std::lock_guard<std::recursive_mutex> lock(mu);
    *s = reinterpret_cast<cudaStream_t>(next_handle += 16);
    return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned)
{
    *e = reinterpret_cast<cudaEvent_t>(0x10);
    return cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t *e) { return cudaEventCreateWithFlags(e, 0); }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t, cudaEvent_t)
{
    *ms = 1.0f;
    return cudaSuccess;
}
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t *g)
{
    *g = reinterpret_cast<cudaGraph_t>(0x20);
    return cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t *e, cudaGraph_t, unsigned long long)
{
    if (fail_graphs > 0) return cudaErrorMemoryAllocation;
    *e = reinterpret_cast<cudaGraphExec_t>(0x30);
    return cudaSuccess;
}
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t s)
{
    std::lock_guard<std::recursive_mutex> lock(mu);
    launched(s);
    return cudaSuccess;
}
cudaError_t cudaGetDevice(int *d)
{
    *d = 0;
    return cudaSuccess;
}
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr a, int)
{
    *v = a == cudaDevAttrMultiProcessorCount ? 152 : 0;
    return cudaSuccess;
}
cudaError_t cudaGetLastError(void) { return cudaSuccess; }
const char *cudaGetErrorString(cudaError_t) { return "error"; }

// std::thread's creation, bound here by -Bsymbolic and the static libstdc++.
int pthread_create(pthread_t *t, const pthread_attr_t *a, void *(*f)(void *), void *arg)
{
    if (fail_threads > 0) return EAGAIN;
    using Fn = int (*)(pthread_t *, const pthread_attr_t *, void *(*)(void *), void *);
    static const Fn real = reinterpret_cast<Fn>(dlsym(RTLD_NEXT, "pthread_create"));
    return real(t, a, f, arg);
}

// Not part of the host runtime's own sources.
int cosm_solve_static(const cosm_graph_desc *, const cosm_params *, int64_t, int32_t, uint64_t, int64_t *, int32_t *, void *)
{
    return COSM_ERR_CUDA;
}
int cosm_probe_smem(int32_t, double *, double *) { return COSM_ERR_CUDA; }
int cosm_probe_fp32(int32_t, double *, double *) { return COSM_ERR_CUDA; }

// ---------------------------------------------------------------- the test's side
void fake_fail_malloc(int64_t nth) { fail_malloc = nth; }  // the nth cudaMalloc from now on fails once
void fake_fail_threads(int on) { fail_threads = on; }
void fake_fail_graphs(int on) { fail_graphs = on; }
int64_t fake_peak_bytes(void)  // since the last call
{
    const int64_t p = peak;
    peak = live;
    return p;
}
const char *fake_message(void) { return why.c_str(); }
int64_t fake_queries(void) { return queries.exchange(0); }
void fake_report(int64_t out[8])
{
    memcpy(out, &rep, sizeof(rep));
    memset(&rep, 0, sizeof(rep));
    why.clear();
}
}
