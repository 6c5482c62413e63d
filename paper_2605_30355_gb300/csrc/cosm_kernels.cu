// CUDA kernels of Cosm for sm_103a: the sweep kernels of edge lists and of
// lattices kept in shared memory, the finalisers, the optimal-bisector
// readout and the measurement probes.
#include <algorithm>

#include "cosm_device.cuh"

namespace cosm {

// ---------------------------------------------------------------- finalize
// Best replica (lowest energy of its kept readout, or the largest cut when
// no energies are kept; ties -> lowest index), its energy, and its spins in
// original vertex order: the saved bits of the kept readout with tracking,
// else the rounding of the final phases at the kept bisector.
__device__ __forceinline__ uint32_t stored_q(const void *state, int storage, size_t idx)
{
    if (storage == 0) return phase_q(reinterpret_cast<const float *>(state)[idx]);
    if (storage == 1) return phase_q(__half2float(reinterpret_cast<const __half *>(state)[idx]));
    if (storage == 3) return phase_q(__bfloat162float(reinterpret_cast<const __nv_bfloat16 *>(state)[idx]));
    return (uint32_t)reinterpret_cast<const uint16_t *>(state)[idx] << 16;
}

__device__ void finalize_body(int replicas, int K, int storage, int P, int n, int64_t W,
                              const void *state, int64_t stride, const int32_t *orig_of,
                              const int64_t *cut, const int32_t *bestp, const int64_t *energy,
                              const uint32_t *bisB, const uint32_t *bits, int words, int64_t *best,
                              int8_t *spins, int64_t target)
{
    // reductions in the warps, then over the warps' results (the block is 1,024
    // threads; a 64-bit shared atomic per thread took 40 of 52 us)
    __shared__ long long s_cut[32];
    __shared__ int s_rep[32], s_hits[32];
    const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31;
    long long bc = LLONG_MIN;
    int br = 0x7FFFFFFF;
    int hits = 0;  // fewer than 2^24 replicas
    for (int r = tid; r < replicas; r += nt) {
        const long long c = energy ? -energy[r] : cut[r];
        if (c > bc || (c == bc && r < br)) { bc = c; br = r; }
        hits += cut[r] >= target ? 1 : 0;
    }
    const auto reduce = [&]() {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const long long c = __shfl_xor_sync(0xFFFFFFFFu, bc, o);
            const int r = __shfl_xor_sync(0xFFFFFFFFu, br, o);
            if (c > bc || (c == bc && r < br)) { bc = c; br = r; }
            hits += __shfl_xor_sync(0xFFFFFFFFu, hits, o);
        }
    };
    reduce();
    if (lane == 0) {
        s_cut[tid >> 5] = bc;
        s_rep[tid >> 5] = br;
        s_hits[tid >> 5] = hits;
    }
    __syncthreads();
    bc = s_cut[lane];
    br = s_rep[lane];
    hits = s_hits[lane];
    reduce();
    const int rb = br;
    const long long cb = cut[rb];
    if (tid == 0) {
        best[0] = cb;
        best[1] = energy ? energy[rb] : W - 2 * cb;
        best[2] = rb;
        best[3] = (int64_t)hits;
    }
    if (bits) {
        const uint32_t *bw = bits + (size_t)rb * words;
        for (int v = tid; v < n; v += nt) spins[orig_of[v]] = ((bw[v >> 5] >> (v & 31)) & 1u) ? 1 : -1;
        return;
    }
    const int tile = rb / K, place = rb % K;
    const uint32_t B = bisB ? bisB[rb] : (uint32_t)(((uint64_t)bestp[rb] << 31) / (uint64_t)P);
    for (int v = tid; v < n; v += nt) {
        const uint32_t q = stored_q(state, storage, (size_t)tile * stride + (size_t)v * K + place);
        spins[orig_of[v]] = ((uint32_t)(q - B) < 0x80000000u) ? 1 : -1;
    }
}

__global__ void __launch_bounds__(1024) finalize_kernel(const FinalArgs a)
{
    finalize_body(a.replicas, a.K, a.storage, a.P, a.n, a.W, a.state, a.state_tile_stride, a.orig_of,
                  a.cut, a.bestp, a.energy, a.bisB, a.bits, a.words, a.best, a.spins, a.target);
}

__global__ void __launch_bounds__(1024) batch_finalize_kernel(const InstView *insts, const BatchFinal *fin)
{
    const InstView &v = insts[blockIdx.x];
    const BatchFinal &f = fin[blockIdx.x];
    finalize_body(v.replicas, v.K, f.storage, v.P, v.n, f.W, v.state, v.state_tile_stride, v.orig_of,
                  v.cut, v.bestp, v.energy, v.bisB, nullptr, 0, f.best, f.spins, LLONG_MIN);
}

// ---------------------------------------------------------------- optimal bisector
// Exact best bisector of each replica (Section II-B; the sorted sweep of
// Burer, Monteiro and Zhang 2002). With phi_v = q_v mod 2^31 and t_v the top
// bit of q_v, s_v(B) = +1 iff [B <= phi_v] xor t_v for B in [0, 2^31), so an
// edge's cut state flips on the interval (lo, hi] of its endpoints'
// positions: d_e = w_e (1 - 2 (t_i xor t_j)) enters at lo + 1 and leaves at
// hi + 1. Each vertex collects the changes that happen at its position, the
// (position, change) pairs are sorted by position, and a block-wide prefix sum
// gives the cut at every position where it can change; the best (ties: the
// smallest B) competes with the replica's kept readout.
//
// One CTA of 1,024 threads per replica at a time, one CTA per SM. The changes
// are summed with shared-memory atomics (global ones where 8 n bytes do not
// fit) and sorted by a least-significant-digit radix sort, 8 bits a pass: each
// warp ranks a contiguous chunk against per-warp digit counts in shared
// memory (match.any orders equal digits), and scatters it to one of two
// buffers in global memory, which stay in L2. Digits in which no two positions
// differ are skipped (fixed point: the lower 16 bits). A bitonic network over
// global memory with a serial block scan took 1.18 ms per replica of 20,000
// vertices and 40,000 edges.
constexpr int kOptThreads = 1024, kOptWarps = kOptThreads / 32, kDigits = 256;

__device__ __forceinline__ long long block_exclusive_sum(long long x, long long *warp_sums)
{
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    long long inc = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const long long y = __shfl_up_sync(0xFFFFFFFFu, inc, o);
        if (lane >= o) inc += y;
    }
    if (lane == 31) warp_sums[w] = inc;
    __syncthreads();
    if (w == 0) {
        long long s = warp_sums[lane];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const long long y = __shfl_up_sync(0xFFFFFFFFu, s, o);
            if (lane >= o) s += y;
        }
        warp_sums[lane] = s;
    }
    __syncthreads();
    const long long before = w ? warp_sums[w - 1] : 0;
    __syncthreads();  // warp_sums may be used again
    return before + inc - x;
}

// One pass of the sort on the digit at `shift`: elements get(i), i < n, into
// out. hist: kDigits x 33 words of shared memory.
template <typename Get>
__device__ __forceinline__ void radix_pass(int n, int shift, uint32_t *hist, long long *warp_sums, uint64_t *out,
                                           const Get &get)
{
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    for (int i = tid; i < kDigits * 33; i += kOptThreads) hist[i] = 0u;
    __syncthreads();
    const int chunk = ((n + kOptWarps - 1) / kOptWarps + 31) / 32 * 32;
    const int i0 = w * chunk, i1 = min(n, i0 + chunk);
    for (int i = i0; i < i1; i += 32) {
        const bool in = i + lane < i1;
        const uint32_t d = in ? (uint32_t)(get(i + lane) >> (32 + shift)) & 0xFFu : 0xFFFFFFFFu;
        const uint32_t same = __match_any_sync(0xFFFFFFFFu, d);
        if (in && lane == __ffs(same) - 1) hist[d * 33 + w] += __popc(same);
        __syncwarp();
    }
    __syncthreads();
    // offsets in (digit, warp) order: eight counts per thread
    {
        uint32_t *h = hist + (tid >> 2) * 33 + (tid & 3) * 8;
        uint32_t c[8], sum = 0;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            c[k] = h[k];
            sum += c[k];
        }
        uint32_t at = (uint32_t)block_exclusive_sum(sum, warp_sums);
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            h[k] = at;
            at += c[k];
        }
    }
    __syncthreads();
    for (int i = i0; i < i1; i += 32) {
        const bool in = i + lane < i1;
        const uint64_t x = in ? get(i + lane) : 0ull;
        const uint32_t d = in ? (uint32_t)(x >> (32 + shift)) & 0xFFu : 0xFFFFFFFFu;
        const uint32_t same = __match_any_sync(0xFFFFFFFFu, d);
        if (in) out[hist[d * 33 + w] + __popc(same & ((1u << lane) - 1u))] = x;
        __syncwarp();
        if (in && lane == __ffs(same) - 1) hist[d * 33 + w] += __popc(same);
        __syncwarp();
    }
    __syncthreads();
}

template <bool kShared>
__global__ void __launch_bounds__(kOptThreads) opt_readout_kernel(const OptArgs o)
{
    extern __shared__ __align__(16) uint32_t opt_smem[];
    __shared__ long long s_sums[kOptWarps], s_best[kOptWarps];
    __shared__ uint32_t s_B[kOptWarps];
    __shared__ unsigned long long s_c0;
    __shared__ uint32_t s_diff;
    __shared__ int s_take;
    const InstView &v = o.v;
    constexpr int nt = kOptThreads;
    const int tid = threadIdx.x, lane = tid & 31, n = v.n;
    uint32_t *hist = opt_smem;
    uint32_t *qb = kShared ? opt_smem + kDigits * 33 : o.qbuf + (size_t)blockIdx.x * n;
    int32_t *dl = kShared ? reinterpret_cast<int32_t *>(qb + n) : o.delta + (size_t)blockIdx.x * n;
    uint64_t *const buf0 = o.items + (size_t)blockIdx.x * 2 * n, *const buf1 = buf0 + n;
    const int m = __ldg(v.off + v.C);
    const int storage = o.storage;
    for (int r = blockIdx.x; r < v.replicas; r += gridDim.x) {
        const int tile = r / v.K, place = r % v.K;
        if (tid == 0) {
            s_c0 = 0ull;
            s_diff = 0u;
        }
        for (int u = tid; u < n; u += nt) {
            qb[u] = stored_q(v.state, storage, (size_t)tile * v.state_tile_stride + (size_t)u * v.K + place);
            dl[u] = 0;
        }
        __syncthreads();
        long long c0 = 0;
        for (int e = tid; e < m; e += nt) {
            const uint32_t rec = load_rec(v, e);
            const int wv = (int)__ldg(v.w + e);
            const int i = (int)(rec & 0xFFFFu), j = (int)(rec >> 16);
            const uint32_t qi = qb[i], qj = qb[j];
            const bool cross = ((qi ^ qj) >> 31) != 0;
            if (cross) c0 += wv;
            const uint32_t pi = qi & 0x7FFFFFFFu, pj = qj & 0x7FFFFFFFu;
            if (pi == pj) continue;
            const int d = cross ? -wv : wv;
            atomicAdd(dl + (pi < pj ? i : j), d);
            atomicAdd(dl + (pi < pj ? j : i), -d);
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) c0 += __shfl_xor_sync(0xFFFFFFFFu, c0, off);
        if (lane == 0) atomicAdd(&s_c0, (unsigned long long)c0);
        uint32_t diff = 0;
        const uint32_t first = qb[0];
        for (int u = tid; u < n; u += nt) diff |= qb[u] ^ first;
        diff = __reduce_or_sync(0xFFFFFFFFu, diff);
        if (lane == 0) atomicOr(&s_diff, diff);
        __syncthreads();
        const uint32_t digits = s_diff;
        // the sort: the first pass reads the vertices, the others a buffer
        uint64_t *it = nullptr;
#pragma unroll 1
        for (int shift = 0; shift < 32; shift += 8) {
            if (!((digits & 0x7FFFFFFFu) >> shift & 0xFFu) && !(shift == 24 && !it)) continue;
            uint64_t *out = it == buf0 ? buf1 : buf0;
            if (it) {
                const uint64_t *in = it;
                radix_pass(n, shift, hist, s_sums, out, [in](int i) { return in[i]; });
            } else {
                radix_pass(n, shift, hist, s_sums, out, [qb, dl](int i) {
                    return ((uint64_t)(qb[i] & 0x7FFFFFFFu) << 32) | (uint32_t)dl[i];
                });
            }
            it = out;
        }
        // block prefix sum over contiguous chunks of the sorted pairs
        const int chunk = (n + nt - 1) / nt;
        const int a0 = min(n, tid * chunk), a1 = min(n, a0 + chunk);
        long long sum = 0;
        for (int i = a0; i < a1; ++i) sum += (int32_t)(uint32_t)it[i];
        const long long C0 = (long long)s_c0;
        long long run = C0 + block_exclusive_sum(sum, s_sums), best = LLONG_MIN;
        uint32_t bB = 0xFFFFFFFFu;
        if (tid == 0) { best = C0; bB = 0; }
        for (int i = a0; i < a1; ++i) {
            const uint64_t x = it[i];
            run += (int32_t)(uint32_t)x;
            const uint32_t pos = (uint32_t)(x >> 32);
            const bool end = (i == n - 1) || ((uint32_t)(it[i + 1] >> 32) != pos);
            if (end && pos + 1u < 0x80000000u && run > best) {
                best = run;
                bB = pos + 1u;
            }
        }
        const auto better = [&](long long c, uint32_t b2) {
            if (c > best || (c == best && b2 < bB)) {
                best = c;
                bB = b2;
            }
        };
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            const long long c = __shfl_xor_sync(0xFFFFFFFFu, best, off);
            better(c, __shfl_xor_sync(0xFFFFFFFFu, bB, off));
        }
        if (lane == 0) {
            s_best[tid >> 5] = best;
            s_B[tid >> 5] = bB;
        }
        __syncthreads();
        if (tid < 32) {
            best = s_best[lane];
            bB = s_B[lane];
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) {
                const long long c = __shfl_xor_sync(0xFFFFFFFFu, best, off);
                better(c, __shfl_xor_sync(0xFFFFFFFFu, bB, off));
            }
            if (tid == 0) {
                s_B[0] = bB;
                const long long E = v.W - 2 * best;
                const int take = !o.keep_better || !v.energy || E < v.energy[r];
                if (take) {
                    v.cut[r] = best;
                    v.bestp[r] = -1;
                    if (v.energy) v.energy[r] = E;
                    if (v.bisB) v.bisB[r] = bB;
                }
                s_take = take;
            }
        }
        __syncthreads();
        if (s_take && v.bits) {
            const uint32_t B = s_B[0];
            for (int wi = tid; wi < v.words; wi += nt) {
                uint32_t word = 0u;
                const int v0 = wi * 32, v1 = min(n, v0 + 32);
                for (int u = v0; u < v1; ++u)
                    if ((uint32_t)(qb[u] - B) < 0x80000000u) word |= 1u << (u - v0);
                v.bits[(size_t)r * v.words + wi] = word;
            }
        }
        __syncthreads();
    }
}

// ---------------------------------------------------------------- state in and out
// A thread takes one slot of one tile: one vector access to its K phases in
// the tile layout, K scalar ones to the replicas' rows (neighbouring slots'
// vertices lie one or two apart). Bound by HBM: a few tens of microseconds
// for 256 replicas of 20,000 phases, where the host loop over the copied
// state took 12 ms.
template <typename T, int K>
struct __align__(sizeof(T) * K) Lanes {
    T v[K];
};

__device__ __forceinline__ double turn_of(double g)
{
    const double x = g - floor(g);
    return x >= 1.0 ? 0.0 : x;
}
template <int kStorage, typename T>
__device__ __forceinline__ double stored_turn(T raw)
{
    if constexpr (kStorage == 0) return turn_of((double)__uint_as_float(raw));
    else if constexpr (kStorage == 1) return turn_of((double)__half2float(__ushort_as_half(raw)));
    else if constexpr (kStorage == 3) return turn_of((double)__bfloat162float(__ushort_as_bfloat16(raw)));
    else return (double)raw / 65536.0;  // fixed point: already a turn in [0, 1)
}

// kStorage -1: the storage type itself.
template <typename T, int K, int kStorage>
__global__ void __launch_bounds__(256) state_export_kernel(const StateArgs a)
{
    const int slot = blockIdx.x * blockDim.x + threadIdx.x;
    if (slot >= a.n) return;
    const int v = a.orig_of[slot];
    for (int t = blockIdx.y; t < a.tiles; t += gridDim.y) {
        const Lanes<T, K> x = reinterpret_cast<const Lanes<T, K> *>(
            reinterpret_cast<const T *>(a.state) + (size_t)(a.t0 + t) * (size_t)a.stride)[slot];
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const int64_t r = (int64_t)t * K + k;  // row
            if ((int64_t)a.t0 * K + r >= a.replicas) break;
            if constexpr (kStorage < 0) reinterpret_cast<T *>(a.rows)[r * a.n + v] = x.v[k];
            else reinterpret_cast<double *>(a.rows)[r * a.n + v] = stored_turn<kStorage>(x.v[k]);
        }
    }
}

// Replicas past the last one, and places past the last slot, become zero.
template <typename T, int K>
__global__ void __launch_bounds__(256) state_import_kernel(const StateArgs a)
{
    const int slot = blockIdx.x * blockDim.x + threadIdx.x;
    if ((int64_t)slot * K >= a.stride) return;
    const int v = slot < a.n ? a.orig_of[slot] : 0;
    for (int t = blockIdx.y; t < a.tiles; t += gridDim.y) {
        T *tile = reinterpret_cast<T *>(a.state) + (size_t)(a.t0 + t) * (size_t)a.stride;
        Lanes<T, K> x;
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const int64_t r = (int64_t)t * K + k;
            const bool there = slot < a.n && (int64_t)a.t0 * K + r < a.replicas;
            x.v[k] = there ? reinterpret_cast<const T *>(a.rows)[r * a.n + v] : (T)0;
        }
        if ((int64_t)(slot + 1) * K <= a.stride) {
            reinterpret_cast<Lanes<T, K> *>(tile)[slot] = x;
        } else {
            for (int64_t k = 0; (int64_t)slot * K + k < a.stride; ++k) tile[(int64_t)slot * K + k] = x.v[k];
        }
    }
}

template <typename T, int K>
static int state_launch(const StateArgs &a, int what, cudaStream_t st)
{
    const int64_t slots = what < 0 ? (a.stride + K - 1) / K : a.n;
    const dim3 grid((unsigned)((slots + 255) / 256), (unsigned)std::min(a.tiles, 4096));
    if (what < 0) state_import_kernel<T, K><<<grid, 256, 0, st>>>(a);
    else if (what == STATE_RAW) state_export_kernel<T, K, -1><<<grid, 256, 0, st>>>(a);
    else if constexpr (sizeof(T) == 4) state_export_kernel<T, K, 0><<<grid, 256, 0, st>>>(a);
    else if (a.storage == 1) state_export_kernel<T, K, 1><<<grid, 256, 0, st>>>(a);
    else if (a.storage == 3) state_export_kernel<T, K, 3><<<grid, 256, 0, st>>>(a);
    else state_export_kernel<T, K, 2><<<grid, 256, 0, st>>>(a);
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

static int state_dispatch(const StateArgs &a, int what, cudaStream_t st)
{
    if (a.storage == 0) {
        if (a.K == 1) return state_launch<uint32_t, 1>(a, what, st);
        if (a.K == 2) return state_launch<uint32_t, 2>(a, what, st);
        if (a.K == 4) return state_launch<uint32_t, 4>(a, what, st);
    } else {
        if (a.K == 2) return state_launch<uint16_t, 2>(a, what, st);
        if (a.K == 4) return state_launch<uint16_t, 4>(a, what, st);
        if (a.K == 8) return state_launch<uint16_t, 8>(a, what, st);
    }
    return -1;
}

int state_export_launch(const StateArgs &a, int kind, void *stream)
{
    return state_dispatch(a, kind, reinterpret_cast<cudaStream_t>(stream));
}
int state_import_launch(const StateArgs &a, void *stream)
{
    return state_dispatch(a, -1, reinterpret_cast<cudaStream_t>(stream));
}

// ---------------------------------------------------------------- host side
template <typename Store, int K, int M>
static SmemLimit &sweep_limit()
{
    static SmemLimit lim;
    return lim;
}
template <typename Store, int K, int M>
static SmemLimit &batch_limit()
{
    static SmemLimit lim;
    return lim;
}

#define COSM_DISPATCH_M(T, KK, MODE, CALL)                 \
    do {                                                   \
        if ((MODE) == MODE_GENERAL) return CALL(T, KK, 0); \
        if ((MODE) == MODE_ACCUM) return CALL(T, KK, 1);   \
        if ((MODE) == MODE_LATTICE2D) return CALL(T, KK, 2); \
    } while (0)

#define COSM_DISPATCH(STORAGE, K, MODE, CALL)                       \
    do {                                                            \
        if ((STORAGE) == 0) {                                       \
            if ((K) == 1) COSM_DISPATCH_M(float, 1, MODE, CALL);    \
            if ((K) == 2) COSM_DISPATCH_M(float, 2, MODE, CALL);    \
            if ((K) == 4) COSM_DISPATCH_M(float, 4, MODE, CALL);    \
        } else if ((STORAGE) == 1) {                                \
            if ((K) == 2) COSM_DISPATCH_M(__half, 2, MODE, CALL);   \
            if ((K) == 4) COSM_DISPATCH_M(__half, 4, MODE, CALL);   \
            if ((K) == 8) COSM_DISPATCH_M(__half, 8, MODE, CALL);   \
        } else if ((STORAGE) == 3) {                                \
            if ((K) == 2) COSM_DISPATCH_M(__nv_bfloat16, 2, MODE, CALL); \
            if ((K) == 4) COSM_DISPATCH_M(__nv_bfloat16, 4, MODE, CALL); \
            if ((K) == 8) COSM_DISPATCH_M(__nv_bfloat16, 8, MODE, CALL); \
        } else {                                                    \
            if ((K) == 2) COSM_DISPATCH_M(uint16_t, 2, MODE, CALL); \
            if ((K) == 4) COSM_DISPATCH_M(uint16_t, 4, MODE, CALL); \
            if ((K) == 8) COSM_DISPATCH_M(uint16_t, 8, MODE, CALL); \
        }                                                           \
    } while (0)

size_t sweep_smem_bytes(int storage, int K, int n, int P, int mode)
{
#define SMEM_CALL(T, KK, M) smem_bytes<T, KK>(n, P, (M) == MODE_ACCUM)
    COSM_DISPATCH(storage, K, mode, SMEM_CALL);
#undef SMEM_CALL
    return 0;
}

int sweep_occupancy(int storage, int K, int mode, int threads, size_t smem)
{
#define OCC_CALL(T, KK, M) occupancy_of(sweep_limit<T, KK, M>(), sweep_kernel<T, KK, M>, max_threads<T, KK, M>(), threads, smem)
    COSM_DISPATCH(storage, K, mode, OCC_CALL);
#undef OCC_CALL
    return 0;
}

int sweep_launch(const LaunchCfg &cfg, const KernelArgs &a, void *stream)
{
#define LAUNCH_CALL(T, KK, M) launch_sweep(sweep_limit<T, KK, M>(), sweep_kernel<T, KK, M>, cfg, a, stream)
    COSM_DISPATCH(cfg.storage, cfg.K, cfg.mode, LAUNCH_CALL);
#undef LAUNCH_CALL
    return -1;
}

int finalize_launch(const FinalArgs &a, void *stream)
{
    finalize_kernel<<<1, 1024, 0, reinterpret_cast<cudaStream_t>(stream)>>>(a);
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

int opt_readout_launch(const OptArgs &a, int grid, void *stream)
{
    static SmemLimit shared, global;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    const size_t hist = (size_t)kDigits * 33 * 4, all = hist + (size_t)a.v.n * 8;
    if (all <= raise_smem(shared, opt_readout_kernel<true>)) {
        opt_readout_kernel<true><<<grid, kOptThreads, all, st>>>(a);
    } else {
        if (hist > raise_smem(global, opt_readout_kernel<false>)) return -1;
        opt_readout_kernel<false><<<grid, kOptThreads, hist, st>>>(a);
    }
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

int batch_occupancy(int storage, int K, int mode, int threads, size_t smem)
{
#define BOCC_CALL(T, KK, M) occupancy_of(batch_limit<T, KK, M>(), batch_kernel<T, KK, M>, max_threads<T, KK, M>(), threads, smem)
    COSM_DISPATCH(storage, K, mode, BOCC_CALL);
#undef BOCC_CALL
    return 0;
}

int batch_launch(int storage, int K, int mode, int grid, int threads, size_t smem, const BatchArgs &b,
                 void *stream)
{
#define BLAUNCH_CALL(T, KK, M) launch_batch(batch_limit<T, KK, M>(), batch_kernel<T, KK, M>, grid, threads, smem, b, stream)
    COSM_DISPATCH(storage, K, mode, BLAUNCH_CALL);
#undef BLAUNCH_CALL
    return -1;
}

int batch_finalize_launch(int count, const InstView *insts, const BatchFinal *fin, void *stream)
{
    batch_finalize_kernel<<<count, 1024, 0, reinterpret_cast<cudaStream_t>(stream)>>>(insts, fin);
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

}  // namespace cosm


// ---------------------------------------------------------------- SMEM probe
namespace cosm {

// Shared-memory read bandwidth: every thread streams 16-byte words from a
// conflict-free pattern; thread 0 records the SM clocks spent.
__global__ void __launch_bounds__(1024) smem_probe_kernel(int iters, unsigned long long *clk,
                                                          uint32_t *sink)
{
    __shared__ uint4 buf[4096];
    const int tid = threadIdx.x;
    for (int k = tid; k < 4096; k += blockDim.x) buf[k] = make_uint4(k, k + 1, k + 2, k + 3);
    __syncthreads();
    unsigned long long t0 = clock64();
    uint32_t acc = 0;
    int idx = tid;
    for (int it = 0; it < iters; ++it) {
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const uint4 v = buf[(idx + u * 512) & 4095];
            acc ^= v.x ^ v.y ^ v.z ^ v.w;
        }
        idx += 7;
    }
    __syncthreads();
    unsigned long long t1 = clock64();
    if (tid == 0) atomicMax(clk, t1 - t0);
    if (acc == 0xFFFFFFFFu) sink[0] = acc;
}

}  // namespace cosm

extern "C" int cosm_probe_smem(int32_t iters, double *bytes_per_clk_per_sm, double *gbps)
{
    using namespace cosm;
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return COSM_ERR_CUDA;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    unsigned long long *clk = nullptr;
    uint32_t *sink = nullptr;
    if (cudaMalloc(&clk, 8) != cudaSuccess || cudaMalloc(&sink, 4) != cudaSuccess) return COSM_ERR_NOMEM;
    cudaMemset(clk, 0, 8);
    cudaEvent_t e0, e1;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    const int threads = 1024, blocks = 2 * sms;
    smem_probe_kernel<<<blocks, threads>>>(iters / 4 + 1, clk, sink);  // warm-up
    cudaMemset(clk, 0, 8);
    cudaEventRecord(e0);
    smem_probe_kernel<<<blocks, threads>>>(iters, clk, sink);
    cudaEventRecord(e1);
    cudaError_t err = cudaEventSynchronize(e1);
    float ms = 0.f;
    cudaEventElapsedTime(&ms, e0, e1);
    unsigned long long cycles = 0;
    cudaMemcpy(&cycles, clk, 8, cudaMemcpyDeviceToHost);
    cudaFree(clk);
    cudaFree(sink);
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    if (err != cudaSuccess) return COSM_ERR_CUDA;
    const double bytes_per_cta = (double)threads * iters * 8 * 16;
    // two CTAs share an SM; clk is the longest CTA's span
    if (bytes_per_clk_per_sm) *bytes_per_clk_per_sm = 2.0 * bytes_per_cta / (double)cycles;
    if (gbps) *gbps = bytes_per_cta * blocks / (ms * 1e-3) / 1e9;
    return COSM_OK;
}

// ---------------------------------------------------------------- FP32 issue probe
namespace cosm {

// FP32 arithmetic issue rate: every thread runs 8 independent chains of
// fused multiply-adds, scalar (fma.rn.f32, one operation per lane) or packed
// (fma.rn.f32x2, two operations per lane); thread 0 records the SM clocks
// spent. The chains hold values near a fixed point of x -> a x + b, so no
// lane overflows or goes subnormal.
template <bool kPacked>
__global__ void __launch_bounds__(1024) fp32_probe_kernel(int iters, unsigned long long *clk, float *sink)
{
    const float a = 0.5f, b = 0.25f + 1e-3f * (float)(threadIdx.x & 7);
    f32x2 x2[8];
    float x1[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        x1[i] = 0.125f * (float)i;
        x2[i] = p_pack(x1[i], -x1[i]);
    }
    const f32x2 a2 = p_pack(a, a), b2 = p_pack(b, b);
    __syncthreads();
    const unsigned long long t0 = clock64();
    for (int it = 0; it < iters; ++it) {
#pragma unroll
        for (int u = 0; u < 8; ++u) {
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                if constexpr (kPacked) {
                    x2[i] = p_fma(x2[i], a2, b2);
                } else {
                    asm volatile("fma.rn.f32 %0, %0, %1, %2;" : "+f"(x1[i]) : "f"(a), "f"(b));
                }
            }
        }
    }
    __syncthreads();
    const unsigned long long t1 = clock64();
    if (threadIdx.x == 0) atomicMax(clk, t1 - t0);
    float s = 0.f;
#pragma unroll
    for (int i = 0; i < 8; ++i) s += kPacked ? p_lo(x2[i]) + p_hi(x2[i]) : x1[i];
    if (s == 12345.0f) sink[0] = s;
}

}  // namespace cosm

extern "C" int cosm_probe_fp32(int32_t iters, double *ops_per_clk_per_sm, double *ops_per_clk_per_sm_packed)
{
    using namespace cosm;
    if (iters < 1) return COSM_ERR_INVALID_ARG;
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return COSM_ERR_CUDA;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    unsigned long long *clk = nullptr;
    float *sink = nullptr;
    if (cudaMalloc(&clk, 8) != cudaSuccess) return COSM_ERR_NOMEM;
    if (cudaMalloc(&sink, 4) != cudaSuccess) {
        cudaFree(clk);
        return COSM_ERR_NOMEM;
    }
    const int threads = 1024, blocks = 2 * sms;
    // operations per CTA: threads x iters x 8 unrolled x 8 chains (x 2 packed)
    const double ops = (double)threads * iters * 64.0;
    double res[2] = {0.0, 0.0};
    cudaError_t err = cudaSuccess;
    for (int packed = 0; packed < 2 && err == cudaSuccess; ++packed) {
        for (int rep = 0; rep < 2; ++rep) {  // the first launch warms up
            cudaMemset(clk, 0, 8);
            if (packed) fp32_probe_kernel<true><<<blocks, threads>>>(rep ? iters : iters / 4 + 1, clk, sink);
            else fp32_probe_kernel<false><<<blocks, threads>>>(rep ? iters : iters / 4 + 1, clk, sink);
        }
        err = cudaDeviceSynchronize();
        unsigned long long cycles = 0;
        if (err == cudaSuccess) err = cudaMemcpy(&cycles, clk, 8, cudaMemcpyDeviceToHost);
        // two CTAs share an SM; clk is the longest CTA's span
        if (cycles) res[packed] = 2.0 * ops * (packed ? 2.0 : 1.0) / (double)cycles;
    }
    cudaFree(clk);
    cudaFree(sink);
    if (err != cudaSuccess) return COSM_ERR_CUDA;
    if (ops_per_clk_per_sm) *ops_per_clk_per_sm = res[0];
    if (ops_per_clk_per_sm_packed) *ops_per_clk_per_sm_packed = res[1];
    return COSM_OK;
}
