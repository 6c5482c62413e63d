// Edge lists of any graph, from record tables laid out for the launch.
//
// A table (cosm_edges.h) gives every warp one stream of rows, 32 edges each,
// colour after colour. A warp takes up to four rows of a colour at a time:
// it decodes their records, at once fetches the next rows' (of the same
// colour, the next one or the next sweep: the stream only goes on), then
// loads, updates and stores the phases. So the records' latency (L2 for
// graphs beyond L1) overlaps the updates and the barriers between colours,
// addresses are a pointer and constants, and a row of 32 edges costs what its
// edges cost: 31 warp instructions at two binary32 replicas per tile (random
// 3-regular graph of 20,000 vertices; colours, twist and wrap included), and two
// wavefronts per phase access.
#pragma once

#include "cosm_device.cuh"
#include "cosm_edges.h"

namespace cosm {

extern __shared__ __align__(16) unsigned char edges_smem[];

// Loads and stores of a slot's K phases at a byte offset of the tile, which
// starts the dynamic shared memory (its address folds into the instruction).
template <int NW>
__device__ __forceinline__ void tile_ld(uint32_t off, uint32_t (&w)[NW])
{
    const unsigned char *p = edges_smem + off;
    if constexpr (NW == 1) {
        w[0] = *reinterpret_cast<const uint32_t *>(p);
    } else if constexpr (NW == 2) {
        const uint2 v = *reinterpret_cast<const uint2 *>(p);
        w[0] = v.x; w[1] = v.y;
    } else {
        const uint4 v = *reinterpret_cast<const uint4 *>(p);
        w[0] = v.x; w[1] = v.y; w[2] = v.z; w[3] = v.w;
    }
}
template <int NW>
__device__ __forceinline__ void tile_st(uint32_t off, const uint32_t (&w)[NW])
{
    unsigned char *p = edges_smem + off;
    if constexpr (NW == 1) *reinterpret_cast<uint32_t *>(p) = w[0];
    else if constexpr (NW == 2) *reinterpret_cast<uint2 *>(p) = make_uint2(w[0], w[1]);
    else *reinterpret_cast<uint4 *>(p) = make_uint4(w[0], w[1], w[2], w[3]);
}

// Constants of one sweep.
struct EdgeStep {
    float alpha;       // float forms
    uint32_t aq;       // fixed point: grid quanta
    uint32_t pw, nw;   // fixed point: the quanta and their negation in both halves
};

// Operands of a record: byte offsets and the signed step (float bits, or the
// quanta alpha w).
template <int kFmt, uint32_t E, bool kQ>
__device__ __forceinline__ void decode(const InstView &v, uint32_t r0, uint32_t r1, const EdgeStep &c, uint32_t &oi,
                                       uint32_t &oj, uint32_t &aw)
{
    if constexpr (kFmt == EDGES_SIGN) {
        oi = (r0 & 0xFFFEu) * (E / 2);
        oj = (r0 >> 16) * E;
        if constexpr (kQ) aw = r0 & 1u;
        else aw = flip_if_odd(__float_as_uint(c.alpha), r0);
    } else if constexpr (kFmt == EDGES_PACK) {
        constexpr int S = E == 8 ? 3 : 4;
        constexpr uint32_t field = 0x3FFFu << S;
        oi = r0 & field;
        oj = (r0 >> (18 - S)) & field;
        if constexpr (kQ) {
            aw = c.aq * ((r0 & (E - 1)) - E / 2);
        } else {
            // 1.5 * 2^23 + code, less the offset: the weight, exactly
            const float w = __fadd_rn(__uint_as_float((r0 & (E - 1)) | 0x4B400000u), -(12582912.0f + (float)(E / 2)));
            aw = __float_as_uint(c.alpha * w);
        }
    } else {
        oi = r0;
        oj = r1 & 0x3FFFFu;
        if constexpr (kQ) aw = (uint32_t)((int32_t)c.aq * ((int32_t)r1 >> 18));
        else aw = __float_as_uint(c.alpha * __uint_as_float(r1 & 0xFFFC0000u));
    }
#ifdef COSM_CHECKS
    if (oi >= (uint32_t)v.n * E || oj >= (uint32_t)v.n * E) {
        if (v.check) atomicOr(v.check, 2);
        oi = oj = 0;
    }
#else
    (void)v;
#endif
}

// The next B rows of this warp's stream, one record per lane and row. They
// are fetched whole, whichever colour they belong to: rows past the ones taken
// next are fetched again (from L1).
template <int RW, int B>
struct Stream {
    const uint32_t *p;  // this lane's first word of the next rows
    uint32_t r[B * RW];
    __device__ __forceinline__ void fetch()
    {
#pragma unroll
        for (int k = 0; k < B; ++k) {
            if constexpr (RW == 1) {
                r[k] = __ldg(p + k * 32);
            } else {
                const uint2 a = __ldg(reinterpret_cast<const uint2 *>(p + k * 64));
                r[2 * k] = a.x;
                r[2 * k + 1] = a.y;
            }
        }
    }
};

// Operands of B rows: byte offsets, signed steps, and which lanes hold an edge.
template <int B>
struct Operands {
    uint32_t oi[B], oj[B], aw[B];
    bool ok[B];
};

// Loads, updates and stores of B rows (edges of one colour share no vertex).
// kAll: every place holds an edge.
template <typename Store, int K, int kFmt, bool kEach, int B, bool kAll>
__device__ __forceinline__ void edge_rows(const Operands<B> &o, const EdgeStep &c)
{
    if constexpr (sizeof(Store) == 4 && K > 1) {
        const uint32_t xb = (uint32_t)__cvta_generic_to_shared(edges_smem);
        f32x2 xi[B][K / 2], xj[B][K / 2];
#pragma unroll
        for (int q = 0; q < B; ++q) {
            if (kAll || o.ok[q]) {
                lds_p<K>(xb + o.oi[q], xi[q]);
                lds_p<K>(xb + o.oj[q], xj[q]);
            } else {
#pragma unroll
                for (int h = 0; h < K / 2; ++h) xi[q][h] = xj[q][h] = 0ull;
            }
        }
#pragma unroll
        for (int q = 0; q < B; ++q) {
            const f32x2 aw2 = ((f32x2)o.aw[q] << 32) | o.aw[q];
#pragma unroll
            for (int h = 0; h < K / 2; ++h) {
                pair_x2(xi[q][h], xj[q][h], aw2, kTwo2);
                if constexpr (kEach) {
                    xi[q][h] = p_wrap(xi[q][h]);
                    xj[q][h] = p_wrap(xj[q][h]);
                }
            }
        }
#pragma unroll
        for (int q = 0; q < B; ++q) {
            if (kAll || o.ok[q]) {
                sts_p<K>(xb + o.oi[q], xi[q]);
                sts_p<K>(xb + o.oj[q], xj[q]);
            }
        }
        return;
    }
    constexpr bool kQ = std::is_same<Store, uint16_t>::value;
    constexpr int NW = K * (int)sizeof(Store) / 4;
    uint32_t wi[B][NW], wj[B][NW];
#pragma unroll
    for (int q = 0; q < B; ++q) {
        if (kAll || o.ok[q]) {
            tile_ld<NW>(o.oi[q], wi[q]);
            tile_ld<NW>(o.oj[q], wj[q]);
        } else {
#pragma unroll
            for (int h = 0; h < NW; ++h) wi[q][h] = wj[q][h] = 0u;
        }
    }
    if constexpr (kQ) {
#pragma unroll
        for (int q = 0; q < B; ++q) {
            if constexpr (kFmt == EDGES_SIGN)
                pair_qw<NW>(wi[q], wj[q], o.aw[q] ? c.nw : c.pw, o.aw[q] ? c.pw : c.nw);
            else
                pair_qw<NW>(wi[q], wj[q], both_halves(o.aw[q]), both_halves(0u - o.aw[q]));
        }
    } else if constexpr (sizeof(Store) == 2) {
#pragma unroll
        for (int q = 0; q < B; ++q) {
            const f32x2 aw2 = ((f32x2)o.aw[q] << 32) | o.aw[q];
#pragma unroll
            for (int h = 0; h < NW; ++h) {
                f32x2 a = h2_to_p<Store>(wi[q][h]), b = h2_to_p<Store>(wj[q][h]);
                pair_x2<kAlu16<Store>()>(a, b, aw2, kTwo2);
                wi[q][h] = p_to_h2<Store>(p_wrap(a));
                wj[q][h] = p_to_h2<Store>(p_wrap(b));
            }
        }
    } else if constexpr (K == 1) {
        // two edges share the lanes (the last of an odd number is alone)
#pragma unroll
        for (int q = 0; q < B; q += 2) {
            constexpr int last = B - 1;
            const int q1 = q + 1 < B ? q + 1 : last;
            f32x2 a = ((f32x2)wi[q1][0] << 32) | wi[q][0], b = ((f32x2)wj[q1][0] << 32) | wj[q][0];
            pair_x2(a, b, ((f32x2)o.aw[q1] << 32) | o.aw[q], kTwo2);
            if constexpr (kEach) {
                a = p_wrap(a);
                b = p_wrap(b);
            }
            wi[q][0] = (uint32_t)a;
            wj[q][0] = (uint32_t)b;
            if (q + 1 < B) {
                wi[q1][0] = (uint32_t)(a >> 32);
                wj[q1][0] = (uint32_t)(b >> 32);
            }
        }
    } else {
#pragma unroll
        for (int q = 0; q < B; ++q) {
            const f32x2 aw2 = ((f32x2)o.aw[q] << 32) | o.aw[q];
#pragma unroll
            for (int h = 0; h < K / 2; ++h) {
                f32x2 a = ((f32x2)wi[q][2 * h + 1] << 32) | wi[q][2 * h];
                f32x2 b = ((f32x2)wj[q][2 * h + 1] << 32) | wj[q][2 * h];
                pair_x2(a, b, aw2, kTwo2);
                if constexpr (kEach) {
                    a = p_wrap(a);
                    b = p_wrap(b);
                }
                wi[q][2 * h] = (uint32_t)a;
                wi[q][2 * h + 1] = (uint32_t)(a >> 32);
                wj[q][2 * h] = (uint32_t)b;
                wj[q][2 * h + 1] = (uint32_t)(b >> 32);
            }
        }
    }
#pragma unroll
    for (int q = 0; q < B; ++q) {
        if (kAll || o.ok[q]) {
            tile_st<NW>(o.oi[q], wi[q]);
            tile_st<NW>(o.oj[q], wj[q]);
        }
    }
}

// The next N rows, all places filled (kAll) or checked lane by lane: decode,
// fetch the rows after them, update.
template <typename Store, int K, int kFmt, bool kEach, int RW, int B, int N, bool kAll>
__device__ __forceinline__ void take_rows(const InstView &v, Stream<RW, B> &st, const EdgeStep &c)
{
    constexpr bool kQ = std::is_same<Store, uint16_t>::value;
    constexpr uint32_t E = K * (uint32_t)sizeof(Store);
    Operands<N> o;
#pragma unroll
    for (int q = 0; q < N; ++q) {
        o.ok[q] = kAll || st.r[q * RW] != kNoEdge;
        if (!kAll) o.aw[q] = 0u;
        if (o.ok[q]) decode<kFmt, E, kQ>(v, st.r[q * RW], st.r[q * RW + RW - 1], c, o.oi[q], o.oj[q], o.aw[q]);
    }
    st.p += N * 32 * RW;
    st.fetch();
    edge_rows<Store, K, kFmt, kEach, N, kAll>(o, c);
}

// The colours of one sweep: per colour the whole batches, the rest, and a
// last row with empty places by itself. counts: this warp's; n: the first.
template <typename Store, int K, int kFmt, bool kEach, int RW, int B>
__device__ __forceinline__ void edge_sweep(const InstView &v, const uint32_t *counts, int nc, uint32_t &n,
                                           Stream<RW, B> &st, const EdgeStep &c)
{
#pragma unroll 1
    for (int k = 1; k <= nc; ++k) {
        const uint32_t next = __ldg(counts + k);
        const bool partial = (int)n < 0;
        int m = (int)(n & ~kPartial) - partial;
        for (; m >= B; m -= B) take_rows<Store, K, kFmt, kEach, RW, B, B, true>(v, st, c);
        if (m == 1) take_rows<Store, K, kFmt, kEach, RW, B, 1, true>(v, st, c);
        if constexpr (B > 2) {
            if (m == 2) take_rows<Store, K, kFmt, kEach, RW, B, 2, true>(v, st, c);
            if (m == 3) take_rows<Store, K, kFmt, kEach, RW, B, 3, true>(v, st, c);
        }
        if (partial) take_rows<Store, K, kFmt, kEach, RW, B, 1, false>(v, st, c);
        n = next;
        __syncthreads();
    }
}

// The twist and the wrap after the colours, one slot at a time.
template <typename Store, int K>
__device__ __forceinline__ void edge_twist(const InstView &v, const Tile<Store, K> &t, int k, int E, float step,
                                           bool dwt, bool wrap)
{
    const int tid = threadIdx.x, nt = blockDim.x, n = v.n, P1 = v.P + 1;
    float th[K], st[K];
#pragma unroll
    for (int r = 0; r < K; ++r) {
        const int *Dr = t.D + r * P1;
        th[r] = dwt ? __int_as_float(Dr[k]) : 0.f;
        st[r] = dwt ? ((((uint32_t)Dr[E] >> k) & 1u) ? -step : step) : 0.f;
    }
    const float W2 = 2.0f * v.window;
    if constexpr (sizeof(Store) == 4) {
        constexpr int H = K >= 2 ? K / 2 : 1;  // words per slot (K = 1: a word spans two slots)
        f32x2 th2[H], tk2[H], st2[H];
#pragma unroll
        for (int h = 0; h < H; ++h) {
            const int r0 = K >= 2 ? 2 * h : 0, r1 = K >= 2 ? 2 * h + 1 : 0;
            th2[h] = p_pack(th[r0], th[r1]);
            tk2[h] = p_pack(th[r0] - W2, th[r1] - W2);
            st2[h] = p_pack(st[r0], st[r1]);
        }
        const int groups = K >= 2 ? n : (n >> 1);
        const uint32_t xb = (uint32_t)__cvta_generic_to_shared(t.xs);
        for (int q = tid; q < groups; q += nt) {
            f32x2 x[H];
            lds_p<2 * H>(xb + (uint32_t)q * 8 * H, x);
#pragma unroll
            for (int h = 0; h < H; ++h) {
                if (dwt) dwt_x2(x[h], th2[h], tk2[h], st2[h]);
                if (wrap) x[h] = p_wrap(x[h]);
            }
            sts_p<2 * H>(xb + (uint32_t)q * 8 * H, x);
        }
        if (K == 1 && (n & 1) && tid == 0) {
            float x = t.xs[n - 1];
            if (dwt && in_windows(x, th[0], th[0] - W2)) x = __fadd_rn(x, st[0]);
            if (wrap) x = wrap_c(x);
            t.xs[n - 1] = x;
        }
    } else {
        for (int u = tid; u < n; u += nt) {
            float x[K];
            ldk<K>(t.xs + (size_t)u * K, x);
#pragma unroll
            for (int r = 0; r < K; ++r)
                if (in_windows(x[r], th[r], th[r] - W2)) x[r] = wrap_c(__fadd_rn(x[r], st[r]));
            stk<K>(t.xs + (size_t)u * K, x);
        }
    }
}

// Threads a CTA may have (16-byte slots of 16-bit floats need 92 registers),
// and rows in flight: four, or two of 16-byte slots. 128 registers for 512
// threads and four or eight rows measured no faster (gnm 10k, 1,024 replicas,
// four replicas per tile: 25.7 us per sweep against 26.6; two: 22.8 against
// 24.0 and 24.3): rows fetched and not taken next cost more than they hide.
template <typename Store, int K>
__host__ __device__ constexpr int edges_max_threads()
{
    return K * sizeof(Store) >= 16 && sizeof(Store) == 2 && !std::is_same<Store, uint16_t>::value ? 512 : 1024;
}
template <typename Store, int K>
__host__ __device__ constexpr int edges_rows()
{
    return K * sizeof(Store) >= 16 ? 2 : 4;
}

template <typename Store, int K, int kFmt, bool kEach>
__device__ __forceinline__ void run_segment_edges(const InstView &v, const Segment &sg, int *s_skip, int32_t *ready,
                                                  int32_t *err, uint64_t wait_limit_ns)
{
    constexpr bool kQ = std::is_same<Store, uint16_t>::value;
    constexpr int RW = kFmt == EDGES_WEIGHT ? 2 : 1;
    constexpr int B = edges_rows<Store, K>();
    const Tile<Store, K> t = carve<Store, K>(edges_smem, v.n, v.P, false);
    const int tid = threadIdx.x, nt = blockDim.x;
    if (!seg_begin<Store, K>(v, sg, t, s_skip, ready, err, wait_limit_ns)) return;
    Stretches st(v);
    const uint32_t rep0 = (uint32_t)sg.tile * K;
    const uint32_t s1 = (uint32_t)sg.s_end;  // below 2^31
    const int wrap_p = v.wrap_p, period = v.dwt_period;
    if (sg.s_begin <= sg.s_end) {
        static_assert(B <= kRowsAhead, "rows ahead");
        const uint32_t *const start = v.rec + __ldg(v.starts + (tid >> 5)) + (tid & 31) * RW;
        const int nc = v.n_colours;
        const uint32_t *const counts = v.counts + (tid >> 5) * (nc + 1);
        uint32_t rows = __ldg(counts);
        Stream<RW, B> stream;
        stream.p = start;
        stream.fetch();
        for (uint32_t s = (uint32_t)sg.s_begin; s <= s1;) {
            int to_twist;
            const uint32_t end = st.template begin<kQ, K>(v, t.D, s, s1, rep0, &to_twist);
            int to_wrap = sweeps_to_wrap(s, wrap_p), event = -1;
            const float2 *ap = v.alpha_tab + ((int64_t)s - v.alpha_base);
            float2 at = __ldg(ap);
#pragma unroll 1
            for (int left = (int)(end - s); left >= 0; --left) {
            const bool dwt = to_twist == 0;
            if (dwt) {
                ++event;
                to_twist = period;
            }
            --to_twist;
            EdgeStep c;
            c.alpha = at.x;
            if constexpr (kQ) {
                c.aq = (uint32_t)__float2int_rn(at.x);
                c.pw = both_halves(c.aq);
                c.nw = both_halves(0u - c.aq);
            }
            const float step = at.y;
            if (left > 0) at = __ldg(++ap);
            edge_sweep<Store, K, kFmt, kEach>(v, counts, nc, rows, stream, c);
            stream.p = start;  // the rows fetched past the end are the first ones
            if (v.hv) {
                if constexpr (kQ) field_pass_q<K>(v, t.xs, c.aq);
                else field_pass<Store, K>(v, t.xs, c.alpha);
                __syncthreads();
            }
            if constexpr (kQ) {
                if (dwt) {
                    constexpr int NW = K / 2;
                    uint32_t cq[K], sq[K], chw[NW], ntw[NW], sqw[NW];
                    const uint32_t stepq = (uint32_t)__float2int_rn(step) << 16;
#pragma unroll
                    for (int r = 0; r < K; ++r) {
                        const int *Dr = t.D + r * (v.P + 1);
                        cq[r] = (uint32_t)Dr[event];
                        sq[r] = ((uint32_t)Dr[st.E] >> event) & 1u ? 0u - stepq : stepq;
                    }
                    dwt_qw_consts<NW>(cq, v.qwin, sq, chw, ntw, sqw);
                    const uint32_t xb = (uint32_t)__cvta_generic_to_shared(t.xs);
                    for (int u = tid; u < v.n; u += nt) {
                        uint32_t x[NW];
                        lds_w<NW>(xb + (uint32_t)u * (K * 2), x);
#pragma unroll
                        for (int h = 0; h < NW; ++h) dwt_qw(x[h], chw[h], ntw[h], sqw[h]);
                        sts_w<NW>(xb + (uint32_t)u * (K * 2), x);
                    }
                    __syncthreads();
                }
            } else {
                // binary32 wraps on every wrap_p-th sweep, or with every
                // twist when each update is wrapped
                const bool wrap = sizeof(Store) == 4 && (kEach ? dwt : to_wrap == 0);
                if (to_wrap == 0) to_wrap = wrap_p;
                --to_wrap;
                if (dwt || wrap) {
                    edge_twist<Store, K>(v, t, event, (int)st.E, step, dwt, wrap);
                    __syncthreads();
                }
            }
            }
            if (st.readout_after(end)) {
                tile_readout<Store, K>(v, sg.tile, t, (int)((end - 1) / st.track), true);
                __syncthreads();
            }
            s = end + 1;
        }
    }
    seg_end<Store, K>(v, sg, t, ready);
}

// One kernel for single runs (segment lists) and queues (batch, serving).
template <typename Store, int K, int kFmt, bool kEach>
__global__ void __launch_bounds__(edges_max_threads<Store, K>()) edges_kernel(const __grid_constant__ KernelArgs a,
                                                                                    const __grid_constant__ BatchArgs b)
{
    __shared__ int s_skip, s_unit;
    if (b.units == nullptr) {
        for (int si = a.seg_off[blockIdx.x]; si < a.seg_off[blockIdx.x + 1]; ++si) {
            const Segment sg = a.segs[si];
            run_segment_edges<Store, K, kFmt, kEach>(a.v, sg, &s_skip, a.ready, a.err, a.wait_limit_ns);
        }
        return;
    }
    for (;;) {
        if (threadIdx.x == 0) s_unit = atomicAdd(b.counter, 1);
        __syncthreads();
        const int u = s_unit;
        __syncthreads();  // all threads read s_unit before it is overwritten
        if (u >= b.n_units) break;
        const BatchUnit bu = b.units[u];
        const Segment sg{bu.tile, bu.flags, bu.s_begin, bu.s_end};
        run_segment_edges<Store, K, kFmt, kEach>(b.insts[bu.inst], sg, &s_skip, nullptr, nullptr, 0);
    }
}

template <typename Store, int K, int kFmt, bool kEach>
int edges_one(const EdgesCall &c)
{
    static SmemLimit lim;
    auto fn = edges_kernel<Store, K, kFmt, kEach>;
    if (c.what == EdgesCall::OCCUPANCY) return occupancy_of(lim, fn, edges_max_threads<Store, K>(), c.threads, c.smem);
    if (c.smem > raise_smem(lim, fn)) return -1;
    static const KernelArgs no_run = {};
    static const BatchArgs no_queue = {};
    const KernelArgs &a = c.run ? *c.run : no_run;
    const BatchArgs &b = c.queue ? *c.queue : no_queue;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(c.stream);
    if (c.cooperative) {
        void *args[] = {const_cast<KernelArgs *>(&a), const_cast<BatchArgs *>(&b)};
        return cudaLaunchCooperativeKernel((const void *)fn, dim3(c.grid), dim3(c.threads), args, c.smem, st) ==
                       cudaSuccess
                   ? 0
                   : -1;
    }
    fn<<<c.grid, c.threads, c.smem, st>>>(a, b);
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

template <typename Store, int K>
int edges_format(const EdgesCall &c)
{
    constexpr bool kPack = K * sizeof(Store) >= 8;  // the code needs 3 bits
    if (c.format == EDGES_SIGN) return edges_one<Store, K, EDGES_SIGN, false>(c);
    if (c.format == EDGES_WEIGHT) return edges_one<Store, K, EDGES_WEIGHT, false>(c);
    if constexpr (kPack)
        if (c.format == EDGES_PACK) return edges_one<Store, K, EDGES_PACK, false>(c);
    if constexpr (sizeof(Store) == 4) {
        if (c.format == (EDGES_WEIGHT | EDGES_EACH)) return edges_one<Store, K, EDGES_WEIGHT, true>(c);
        if constexpr (kPack)
            if (c.format == (EDGES_PACK | EDGES_EACH)) return edges_one<Store, K, EDGES_PACK, true>(c);
    }
    return c.what == EdgesCall::OCCUPANCY ? 0 : -1;
}

template <typename Store, int K0, int K1, int K2>
int edges_dispatch(const EdgesCall &c)
{
    if (c.K == K0) return edges_format<Store, K0>(c);
    if (c.K == K1) return edges_format<Store, K1>(c);
    if (c.K == K2) return edges_format<Store, K2>(c);
    return c.what == EdgesCall::OCCUPANCY ? 0 : -1;
}

}  // namespace cosm
