// Host-side state of one instance and the runtime helpers shared by the
// single-instance, batch and serving code.
#pragma once

#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <cstdint>
#include <memory>
#include <new>
#include <string>
#include <system_error>
#include <thread>
#include <vector>

#include "../../include/cosm.h"
#include "cosm_internal.h"
#include "cosm_edges.h"
#include "cosm_patch.h"

#include <nvtx3/nvToolsExt.h>

namespace cosm {

// Records msg for cosm_last_error() and returns code.
int fail(int code, const std::string &msg);

// An NVTX range over the scope of one ABI call (host side: create, run,
// readout, batch and server steps), visible to profilers that attach an
// NVTX tool and free otherwise.
struct NvtxRange {
    explicit NvtxRange(const char *name) { nvtxRangePushA(name); }
    ~NvtxRange() { nvtxRangePop(); }
    NvtxRange(const NvtxRange &) = delete;
    NvtxRange &operator=(const NvtxRange &) = delete;
};

}  // namespace cosm

#define CK(call)                                                                          \
    do {                                                                                  \
        cudaError_t e_ = (call);                                                          \
        if (e_ != cudaSuccess)                                                            \
            return fail(COSM_ERR_CUDA, std::string(#call) + ": " + cudaGetErrorString(e_)); \
    } while (0)

namespace cosm {

template <typename T>
struct DevBuf {
    T *p = nullptr;
    size_t cap = 0;  // elements
    int ensure(size_t count)
    {
        if (count <= cap && p) return COSM_OK;
        if (p) cudaFree(p);
        p = nullptr;
        cap = 0;
        if (cudaMalloc((void **)&p, std::max<size_t>(count, 1) * sizeof(T)) != cudaSuccess) {
            cudaGetLastError();
            return fail(COSM_ERR_NOMEM, "cudaMalloc failed");
        }
        cap = std::max<size_t>(count, 1);
        return COSM_OK;
    }
    void release()
    {
        if (p) cudaFree(p);
        p = nullptr;
        cap = 0;
    }
};

// A sweep's edges laid out for one tile width and thread count
// (cosm_edges.h); only read once it is filled.
struct RecordTable {
    int K = 0, threads = 0, format = -1, n_colours = 0;
    DevBuf<uint32_t> rec, counts;
    DevBuf<int32_t> starts;
    void release()
    {
        rec.release();
        counts.release();
        starts.release();
    }
};

// How a handle's replicas are laid out in tiles: the kernel and tables that
// its launches take, and the layout its state is stored in.
struct TileLayout {
    int K = 0, threads = 0, occupancy = 0;
    int shape = -1;            // patch shape of the register kernels (-1: phases in shared memory)
    bool ragged = false;       // the shape does not divide the lattice
    int pgr = 0, pgc = 0, pfr = 0, pfc = 0;  // patch grid and its whole rows / columns of patches
    int format = -1;           // record-table format (-1: none)
    const RecordTable *table = nullptr;      // its table
    bool block_pairs = false;  // binary32 lattice tiles of two replicas: two 2x2 blocks per thread (even pass)
    bool staged = false;       // binary32 edge lists: colour records staged in shared memory
    size_t smem = 0;
    int64_t tile_stride = 0;   // storage elements per tile
};

}  // namespace cosm

struct cosm_handle : cosm::TileLayout {
    using Graph = cosm::Graph;
    template <typename T> using DevBuf = cosm::DevBuf<T>;
    Graph g;                        // host copy, original vertex ids
    cosm_params prm;
    int device = 0;
    int num_sms = 0;
    bool lattice = false;
    int64_t W = 0;                  // total weight
    int32_t wmax = 0;               // largest |w|
    int64_t wbound = 0;             // sum over colours of the largest |w|, plus the largest |h|
    std::vector<int32_t> slot_of;   // original id -> slot
    std::vector<int32_t> orig_of;   // slot -> original id
    int32_t off[cosm::kMaxColors + 1] = {0};
    int32_t C = 0;
    DevBuf<uint32_t> d_ij;
    DevBuf<int8_t> d_w;
    std::vector<uint32_t> h_ij;     // colour-major records and weights on the host
    std::vector<int8_t> h_wv;
    std::vector<std::unique_ptr<cosm::RecordTable>> tables;
    DevBuf<int32_t> d_orig;
    DevBuf<uint16_t> d_slot;        // original id -> slot (lattices)
    DevBuf<int32_t> d_off;          // colour offsets
    int mode = cosm::MODE_GENERAL_;       // kernel variant
    int32_t Q = 0, Wd = 0;          // 2D lattice geometry
    DevBuf<uint8_t> d_wnib;         // 2D lattice block weight bits
    std::vector<uint8_t> nib;       // the same on the host
    // 2D lattice kept in registers: weight words per patch, one table per
    // shape, filled once when the shape is first chosen and then only read
    DevBuf<uint32_t> d_pwt[cosm::kPatchShapes];
    bool fields = false;            // local fields given
    DevBuf<int32_t> d_h;            // local field per slot
    DevBuf<int2> d_hlist;           // (slot, field) of the vertices with one
    int32_t n_fields = 0;
    // per run
    DevBuf<unsigned char> d_state;
    DevBuf<int64_t> d_cut;
    DevBuf<int32_t> d_bestp;
    DevBuf<float2> d_alpha;
    DevBuf<cosm::Segment> d_segs;
    DevBuf<int32_t> d_segoff;
    DevBuf<int32_t> d_ready;
    DevBuf<int32_t> d_err;
    DevBuf<int64_t> d_best;
    DevBuf<int8_t> d_spins;
    DevBuf<int64_t> d_energy;       // per replica: energy of the kept readout
    DevBuf<uint32_t> d_bisB;        // per replica: its bisector position
    DevBuf<int64_t> d_trace;        // tracking: [replica][readout] energies
    DevBuf<uint32_t> d_bits;        // tracking: [replica][words] kept spins
    DevBuf<uint32_t> d_qbuf;        // optimal bisector scratch
    DevBuf<int32_t> d_delta;
    DevBuf<uint64_t> d_items;
    DevBuf<unsigned char> d_stage;  // rows on their way in or out (bounded, state_rows)
    int32_t n_trace = 0;            // readouts per trial of the last tracked run
    bool have_trace = false;
    bool bits_valid = false;        // d_bits holds the kept spins of the last run
    // cached host tables
    int64_t alpha_S = -1;
    double alpha_a0 = -1, alpha_ratio = -1;
    std::vector<cosm::Segment> h_segs;
    std::vector<int32_t> h_segoff;
    int64_t sched_tiles = -1, sched_S = -1, sched_G = -1, sched_s0 = -1, sched_s1 = -1;
    bool segs_uploaded = false;
    // state of the last launch
    int replicas = 0;
    int grid = 0;
    uint64_t seed = 0;
    int64_t sweep_idx = 0;          // sweeps of the current trial applied to the state
    int64_t target = INT64_MIN;     // success threshold of the last run's cuts
    uint64_t wait_limit_ns = 0;     // bounded waits between segments (0: environment / 20 s)
    int32_t fault = 0;              // host-side fault injection for the next run (COSM_FAULT_*)
    bool have_state = false, have_result = false;
    cudaStream_t stream = nullptr;
    int launches = 0;
};

namespace cosm {

int env_int(const char *name, int dflt);
// The sweep kernel of a handle's layout: resident CTAs per SM (queue: as the
// batch and serving launches run it), and its launches.
int kernel_occupancy(const cosm_handle *h, int threads, size_t smem, bool queue);
int kernel_launch(const LaunchCfg &cfg, const KernelArgs &a, cudaStream_t st);
int kernel_launch_queue(const LaunchCfg &cfg, const BatchArgs &b, cudaStream_t st);
// narrow_ties: among tiles keeping as many replicas resident, or of modelled
// costs within 10 %, the narrower one (more CTAs per SM). only_K: tiles of that
// width alone (0: any).
int choose_layout(cosm_handle *h, int replicas, bool narrow_ties = false, int only_K = 0);
// Half a thread count, in whole warps where the kernel needs them.
inline int half_threads(int threads, bool warps) { return warps ? std::max(32, threads / 64 * 32) : threads / 2; }
// A forced thread count (0: none) as the kernels take it: the readout scans the
// bisectors with all lanes of a warp.
inline int at_least_a_warp(int threads) { return threads > 0 ? std::max(32, threads) : threads; }
// The device tables of the chosen layout (h->K, h->threads, h->shape).
int ensure_tables(cosm_handle *h);
int ensure_run_buffers(cosm_handle *h, int replicas);
// Device bytes of a handle's graph, tables and run buffers.
size_t device_bytes(const cosm_handle *h);
InstView inst_view(cosm_handle *h);
int upload_alpha(cosm_handle *h, int64_t S, cudaStream_t st);
int launch_finalize(cosm_handle *h, cudaStream_t st);
int launch_opt_readout(cosm_handle *h, bool keep_better, cudaStream_t st);
int single_only(const cosm_graph_desc *g, const cosm_params *p);

// Runs work(i) for i < count on the calling thread and at most 15 more, each
// with `device` current. Where no more threads can be created the ones there do
// the work. Returns how many took part.
template <typename Work>
int side_by_side(size_t count, int device, const Work &work)
{
    std::atomic<size_t> next{0};
    const auto loop = [&] {
        for (size_t i; (i = next++) < count;) work(i);
    };
    std::vector<std::thread> pool;
    const size_t most = std::min<size_t>(count, std::max(1u, std::min(16u, std::thread::hardware_concurrency())));
    try {
        pool.reserve(most);
        while (pool.size() + 1 < most)
            pool.emplace_back([&loop, device] {
                cudaSetDevice(device);
                loop();
            });
    } catch (const std::system_error &) {
    } catch (const std::bad_alloc &) {
    }
    loop();
    for (auto &t : pool) t.join();
    return (int)pool.size() + 1;
}

}  // namespace cosm
