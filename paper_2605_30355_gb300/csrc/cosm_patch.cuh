// 2D lattices held in registers ("patch" kernels).
//
// A thread owns a patch of PR x PC 2x2 blocks (2 PR x 2 PC sites) of one
// replica tile and keeps its phases in registers for the whole segment. The
// colours 0 and 1 of a sweep act inside the patch's own blocks. Colours 2
// and 3 act inside the blocks shifted by one site in both directions, which
// reach into the patches to the right and below: every thread publishes its
// first row and first column of sites in shared memory, reads the
// neighbours' ones it needs, updates the shifted blocks, writes the borrowed
// sites back and reads its own again. So a sweep moves 4 (2 PR + 2 PC - 1)
// sites per patch through shared memory instead of 16 PR PC, two barriers as
// in the shared-memory passes, with the same operations per lane in the same
// order: the phases are bit-identical to block_pass_even / block_pass_odd.
//
// What bounds the sweep is instruction issue: the FMA pipe for the float forms
// (62 % busy, 59 % of issue slots; a pair update alone runs in 12.1 cycles per
// warp and scheduler against 8 for its four packed instructions), the logic
// pipe and the integer multiply-add pipe for fixed point (59 % each). The
// passes on shared memory spent a third of their instructions on loads,
// stores, addresses and weight bits per block. Measured per sweep of 1,024
// replicas, shared memory against registers: 100 x 200 binary32 13.7 -> 11.3
// us, fixed point 9.9 -> 6.9; 100 x 100 7.2 -> 5.5 and 6.4 -> 3.4 (binary16
// 8.6 -> 7.3); one wave of 16 x 16 0.57 -> 0.28 and 0.63 -> 0.20. The register
// file (256 KB) holds a tile of 160 KB of phases; the patch shapes trade
// exchanged sites (large patches) for threads and latency (small ones).
// Publishing early and splitting the barrier into arrival and wait (mbarrier)
// was slower (its wait costs 400 cycles).
//
// Sides that the shape does not divide: patches at the end of a row (column)
// of patches are one block shorter; their last block column (row) is a
// phantom computed on and thrown away (kRagged).
#pragma once

#include "cosm_device.cuh"
#include "cosm_patch.h"

namespace cosm {

// ---------------------------------------------------------------- sites
// A site's K phases in the storage type: one f32x2 (binary32, K = 2) or
// K / 2 packed words (16-bit storage).
template <typename Store, int K>
struct Site {
    static constexpr int NW = K / 2;
    uint32_t w[NW];
};
template <>
struct Site<float, 2> {
    static constexpr int NW = 1;
    f32x2 w[1];
};

template <typename Store, int K>
__device__ __forceinline__ Site<Store, K> lds_site(uint32_t a)
{
    Site<Store, K> s;
    if constexpr (sizeof(Store) == 4) lds_p<2>(a, s.w);
    else lds_w<K / 2>(a, s.w);
    return s;
}
template <typename Store, int K>
__device__ __forceinline__ void sts_site(uint32_t a, const Site<Store, K> &s)
{
    if constexpr (sizeof(Store) == 4) sts_p<2>(a, s.w);
    else sts_w<K / 2>(a, s.w);
}

// Twist constants of one event, per pair of replicas: the float forms' window
// offsets and step, the fixed-point form's words (dwt_qw).
template <int H>
struct TwistF {
    f32x2 th[H], tk[H], st[H];
};
template <int H>
struct TwistQ {
    uint32_t ch[H], nt[H], st[H];
};

// Constants of one sweep; the twist's are read from its window where they
// are used (registers are what limits the patch).
struct SweepConsts {
    uint32_t a1;     // float forms: bits of alpha; fixed point: quanta in both halves
    uint32_t n1;     // fixed point: the negated quanta
    bool dwt, wrap;
    const int *D;    // twist window (TwistWindow): event k of E, P1 words per replica
    int k, E, P1;
    float W2, step;
    uint32_t qwin;
};

template <int K>
__device__ __forceinline__ TwistF<K / 2> twist_f(const SweepConsts &c)
{
    TwistF<K / 2> t;
#pragma unroll
    for (int h = 0; h < K / 2; ++h) {
        float th[2], st[2];
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const int *Dr = c.D + (2 * h + r) * c.P1;
            th[r] = __int_as_float(Dr[c.k]);
            st[r] = ((uint32_t)Dr[c.E] >> c.k) & 1u ? -c.step : c.step;
        }
        t.th[h] = p_pack(th[0], th[1]);
        t.tk[h] = p_pack(th[0] - c.W2, th[1] - c.W2);
        t.st[h] = p_pack(st[0], st[1]);
    }
    return t;
}
template <int K>
__device__ __forceinline__ TwistQ<K / 2> twist_q(const SweepConsts &c)
{
    TwistQ<K / 2> t;
    const uint32_t stepq = (uint32_t)__float2int_rn(c.step) << 16;
    uint32_t cq[K], sq[K];
#pragma unroll
    for (int r = 0; r < K; ++r) {
        const int *Dr = c.D + r * c.P1;
        cq[r] = (uint32_t)Dr[c.k];
        sq[r] = ((uint32_t)Dr[c.E] >> c.k) & 1u ? 0u - stepq : stepq;
    }
    dwt_qw_consts<K / 2>(cq, c.qwin, sq, t.ch, t.nt, t.st);
    return t;
}

// ---------------------------------------------------------------- blocks
// One 2x2 block {tl, tr, bl, br} and two colours: tl-tr and bl-br, then
// tl-bl and tr-br; bits SH .. SH + 3 of w are the weight bits of the four
// edges in that order. ch / cv: 2, or -2 where the horizontal / vertical
// pairs cross the torus seam (the weight bits are flipped there already).
// kVH, kVV: ch, cv vary (else 2).
template <int SH>
__device__ __forceinline__ f32x2 signed_step2(uint32_t w, uint32_t a1)
{
    const uint32_t aw = a1 ^ ((SH < 31 ? w << (31 - SH) : w) & 0x80000000u);
    return ((f32x2)aw << 32) | aw;
}

template <int SH, bool kVH, bool kVV, int kAlu>
__device__ __forceinline__ void block_x2(f32x2 &tl, f32x2 &tr, f32x2 &bl, f32x2 &br, uint32_t w, uint32_t a1,
                                         f32x2 ch, f32x2 cv)
{
    const f32x2 h2 = kVH ? ch : kTwo2, v2 = kVV ? cv : kTwo2;
    pair_x2<kAlu>(tl, tr, signed_step2<SH>(w, a1), h2);
    pair_x2<kAlu>(bl, br, signed_step2<SH + 1>(w, a1), h2);
    pair_x2<kAlu>(tl, bl, signed_step2<SH + 2>(w, a1), v2);
    pair_x2<kAlu>(tr, br, signed_step2<SH + 3>(w, a1), v2);
}

// Fixed point in a staggered form. Every edge of the lattice joins a site of
// even (row + column) to one of odd; the even ones are held as their
// complement X = ~x, the odd ones as W = x. With u = X + W per half:
//   the even site is x_i of eq. (6): ~(x_i - x_j) = u,     so sgn_b = +1 iff u < 0
//   the odd site is x_i:               x_i - x_j = u + 1,  so sgn_b = -1 iff u + 1 < 0
// and in both cases X and W take the same increment, -alpha w where the sign
// bit of u (u + 1) is set and +alpha w elsewhere (all modulo 2^16, ties and
// the exactly-opposite value included). One byte permute and one select per
// word replace the complement, the permute and the two selects of pair_qw,
// whose logic pipe bounds it (76 % busy in the patch kernel). k: the 0 or 1
// added to u in both halves; pairs across the torus seam swap the two cases.
template <int NW, bool kAdd>
__device__ __forceinline__ void pair_staggered(uint32_t (&X)[NW], uint32_t (&W)[NW], uint32_t pq, uint32_t nq,
                                               uint32_t k)
{
#pragma unroll
    for (int h = 0; h < NW; ++h) {
        uint32_t u = add_u16x2(X[h], W[h]);
        if constexpr (kAdd) u = add_u16x2(u, k);
        const uint32_t neg = half_signs(u);
        const uint32_t inc = (nq & neg) | (pq & ~neg);
        X[h] = add_u16x2(X[h], inc);
        W[h] = add_u16x2(W[h], inc);
    }
}

constexpr int kPatchAlu16 = 2;
// kDwt: the twist follows (16-bit floats take it before they are rounded).
template <typename Store, int K, int SH, bool kVH, bool kVV, bool kDwt>
__device__ __forceinline__ void patch_block(Site<Store, K> &tl, Site<Store, K> &tr, Site<Store, K> &bl,
                                            Site<Store, K> &br, uint32_t w, const SweepConsts &c, f32x2 ch, f32x2 cv,
                                            const TwistF<K / 2> &tf)
{
    if constexpr (sizeof(Store) == 4) {
        block_x2<SH, kVH, kVV, 1>(tl.w[0], tr.w[0], bl.w[0], br.w[0], w, c.a1, ch, cv);
    } else if constexpr (std::is_same<Store, uint16_t>::value) {
        // the block's corners tl and br are even sites, tr and bl odd ones
        constexpr int NW = K / 2;
        constexpr uint32_t one = 0x00010001u;
        const uint32_t sh = (uint32_t)ch, sv = (uint32_t)cv;  // 1 in both halves on seam pairs, else 0
        const bool s0 = (w >> SH) & 1u, s1 = (w >> (SH + 1)) & 1u, s2 = (w >> (SH + 2)) & 1u,
                   s3 = (w >> (SH + 3)) & 1u;
        const uint32_t a = c.a1, n = c.n1;
        pair_staggered<NW, kVH>(tl.w, tr.w, s0 ? n : a, s0 ? a : n, sh);
        pair_staggered<NW, true>(br.w, bl.w, s1 ? n : a, s1 ? a : n, kVH ? sh ^ one : one);
        pair_staggered<NW, kVV>(tl.w, bl.w, s2 ? n : a, s2 ? a : n, sv);
        pair_staggered<NW, true>(br.w, tr.w, s3 ? n : a, s3 ? a : n, kVV ? sv ^ one : one);
    } else {
        // 16-bit floats: widened, two colours (and the twist) in binary32,
        // wrapped and rounded once, as the shared-memory passes
#pragma unroll
        for (int h = 0; h < K / 2; ++h) {
            f32x2 a = h2_to_p<Store>(tl.w[h]), b = h2_to_p<Store>(tr.w[h]);
            f32x2 d = h2_to_p<Store>(bl.w[h]), e = h2_to_p<Store>(br.w[h]);
            block_x2<SH, kVH, kVV, kPatchAlu16>(a, b, d, e, w, c.a1, ch, cv);
            if constexpr (kDwt) {
                dwt_x2(a, tf.th[h], tf.tk[h], tf.st[h]);
                dwt_x2(b, tf.th[h], tf.tk[h], tf.st[h]);
                dwt_x2(d, tf.th[h], tf.tk[h], tf.st[h]);
                dwt_x2(e, tf.th[h], tf.tk[h], tf.st[h]);
            }
            tl.w[h] = p_to_h2<Store>(p_wrap(a));
            tr.w[h] = p_to_h2<Store>(p_wrap(b));
            bl.w[h] = p_to_h2<Store>(p_wrap(d));
            br.w[h] = p_to_h2<Store>(p_wrap(e));
        }
    }
}

// ---------------------------------------------------------------- patch
template <typename Store, int K, int PR, int PC, bool kRagged>
struct Patch {
    static constexpr int SR = 2 * PR, SC = 2 * PC, NS = SR * SC;
    static constexpr int NE = SR + SC - 1;            // published sites (odd: conflict-free stride)
    static constexpr uint32_t E = K * sizeof(Store);  // bytes per site
    static constexpr int NWT = (8 * PR * PC + 31) / 32;  // weight words
    using S = Site<Store, K>;
    static constexpr bool kRR = kRagged && PR > 1, kRC = kRagged && PC > 1;

    S x[NS];
    uint32_t wt[NWT];
    uint32_t own, right, below, diag;  // shared addresses of the published sites of four patches
    bool shortR, shortC;
    f32x2 ch0, ch1, cv0, cv1;  // c of the last / second-to-last block column and row of shifted blocks

    // fixed point: sites held as their complement (pair_staggered)
    __device__ static constexpr bool even_site(int k) { return ((k / SC + k % SC) & 1) == 0; }
    __device__ static constexpr int at(int r, int c) { return (r % SR) * SC + (c % SC); }
    // published site (0, c) or (r, 0)
    __device__ static constexpr uint32_t pub(int r, int c) { return (uint32_t)(r == 0 ? c : SC + r - 1) * E; }

    // Even block (i, j).
    template <int i, int j>
    __device__ __forceinline__ void even(const SweepConsts &c)
    {
        constexpr int b = 4 * (i * PC + j);
        patch_block<Store, K, b % 32, false, false, false>(
            x[at(2 * i, 2 * j)], x[at(2 * i, 2 * j + 1)], x[at(2 * i + 1, 2 * j)], x[at(2 * i + 1, 2 * j + 1)],
            wt[b / 32], c, kTwo2, kTwo2, TwistF<K / 2>());
    }
    // Shifted block (i, j): its right sites are in the next patch for the
    // last block column, its bottom sites for the last block row.
    template <int i, int j, bool kDwt>
    __device__ __forceinline__ void odd(const SweepConsts &c, const TwistF<K / 2> &tf)
    {
        constexpr int b = 4 * (PR * PC + i * PC + j);
        constexpr bool h0 = j == PC - 1, h1 = kRC && j == PC - 2, v0 = i == PR - 1, v1 = kRR && i == PR - 2;
        patch_block<Store, K, b % 32, h0 || h1, v0 || v1, kDwt>(
            x[at(2 * i + 1, 2 * j + 1)], x[at(2 * i + 1, 2 * j + 2)], x[at(2 * i + 2, 2 * j + 1)],
            x[at(2 * i + 2, 2 * j + 2)], wt[b / 32], c, h0 ? ch0 : ch1, v0 ? cv0 : cv1, tf);
    }
    // Blocks without a published site (even) or a borrowed one (shifted) come
    // first: they cover the latency of the shared loads before them.
    static constexpr int IR = kRR ? PR - 2 : PR - 1, IC = kRC ? PC - 2 : PC - 1;
    template <bool kInner, int b = 0>
    __device__ __forceinline__ void evens(const SweepConsts &c)
    {
        if constexpr (b < PR * PC) {
            if constexpr ((b / PC > 0 && b % PC > 0) == kInner) even<b / PC, b % PC>(c);
            evens<kInner, b + 1>(c);
        }
    }
    template <bool kInner, bool kDwt, int b = 0>
    __device__ __forceinline__ void odds(const SweepConsts &c, const TwistF<K / 2> &tf)
    {
        if constexpr (b < PR * PC) {
            if constexpr ((b / PC < IR && b % PC < IC) == kInner) odd<b / PC, b % PC, kDwt>(c, tf);
            odds<kInner, kDwt, b + 1>(c, tf);
        }
    }
    // The shifted blocks with the sweep's twist and wrap: every site held now
    // sits in exactly one of them. 16-bit floats take the twist block by block,
    // before they are rounded.
    __device__ __forceinline__ void odd_pass(const SweepConsts &c)
    {
        if constexpr (sizeof(Store) == 2 && !std::is_same<Store, uint16_t>::value) {
            if (c.dwt) {
                const TwistF<K / 2> tf = twist_f<K>(c);
                odds<true, true>(c, tf);
                odds<false, true>(c, tf);
            } else {
                odds<true, false>(c, TwistF<K / 2>());
                odds<false, false>(c, TwistF<K / 2>());
            }
        } else {
            odds<true, false>(c, TwistF<K / 2>());
            odds<false, false>(c, TwistF<K / 2>());
            if (c.dwt) {
                if constexpr (sizeof(Store) == 4) {
                    const TwistF<K / 2> t = twist_f<K>(c);
#pragma unroll
                    for (int k = 0; k < NS; ++k) dwt_x2(x[k].w[0], t.th[0], t.tk[0], t.st[0]);
                } else {
                    const TwistQ<K / 2> t = twist_q<K>(c);
#pragma unroll
                    for (int k = 0; k < NS; ++k) {
#pragma unroll
                        for (int h = 0; h < K / 2; ++h) {
                            uint32_t q = even_site(k) ? ~x[k].w[h] : x[k].w[h];
                            dwt_qw(q, t.ch[h], t.nt[h], t.st[h]);
                            x[k].w[h] = even_site(k) ? ~q : q;
                        }
                    }
                }
            }
            if constexpr (sizeof(Store) == 4) {
                if (c.wrap) {
#pragma unroll
                    for (int k = 0; k < NS; ++k) x[k].w[0] = p_wrap(x[k].w[0]);
                }
            }
        }
    }

    __device__ __forceinline__ void publish()
    {
#pragma unroll
        for (int c = 0; c < SC; ++c) sts_site<Store, K>(own + pub(0, c), x[at(0, c)]);
#pragma unroll
        for (int r = 1; r < SR; ++r) sts_site<Store, K>(own + pub(r, 0), x[at(r, 0)]);
    }
    __device__ __forceinline__ void take_back()
    {
#pragma unroll
        for (int c = 0; c < SC; ++c) x[at(0, c)] = lds_site<Store, K>(own + pub(0, c));
#pragma unroll
        for (int r = 1; r < SR; ++r) x[at(r, 0)] = lds_site<Store, K>(own + pub(r, 0));
    }
    // The neighbours' sites of the shifted blocks. They take the places of
    // row 0 and column 0, which are published; in a short patch the phantom
    // row SR - 2 (column SC - 2) is the one after its last own row (column).
    __device__ __forceinline__ void borrow()
    {
#pragma unroll
        for (int c = 1; c < SC; ++c) x[at(0, c)] = lds_site<Store, K>(below + pub(0, c));
#pragma unroll
        for (int r = 1; r < SR; ++r) x[at(r, 0)] = lds_site<Store, K>(right + pub(r, 0));
        x[at(0, 0)] = lds_site<Store, K>(diag + pub(0, 0));
        if constexpr (kRC) {
            if (shortC) {
#pragma unroll
                for (int r = 1; r < SR; ++r) x[at(r, SC - 2)] = x[at(r, 0)];
                x[at(0, SC - 2)] = x[at(0, 0)];
            }
        }
        if constexpr (kRR) {
            // row 0 already holds the row below, its corner included
            if (shortR) {
#pragma unroll
                for (int c = 0; c < SC; ++c) x[at(SR - 2, c)] = x[at(0, c)];
            }
        }
    }
    __device__ __forceinline__ void give_back()
    {
        if constexpr (kRR) {
            if (shortR) {
#pragma unroll
                for (int c = 0; c < SC; ++c) x[at(0, c)] = x[at(SR - 2, c)];
            }
        }
        if constexpr (kRC) {
            if (shortC) {
#pragma unroll
                for (int r = 1; r < SR; ++r) x[at(r, 0)] = x[at(r, SC - 2)];
                x[at(0, 0)] = x[at(0, SC - 2)];
            }
        }
#pragma unroll
        for (int c = 1; c < SC; ++c) sts_site<Store, K>(below + pub(0, c), x[at(0, c)]);
#pragma unroll
        for (int r = 1; r < SR; ++r) sts_site<Store, K>(right + pub(r, 0), x[at(r, 0)]);
        sts_site<Store, K>(diag + pub(0, 0), x[at(0, 0)]);
    }

    __device__ __forceinline__ static void flip(S &s, bool even)
    {
        if constexpr (std::is_same<Store, uint16_t>::value) {
            if (even) {
#pragma unroll
                for (int h = 0; h < S::NW; ++h) s.w[h] = ~s.w[h];
            }
        }
    }
    // Own sites from / to the tile in shared memory ([slot][K], four
    // sublattices of Q slots).
    template <bool kLoad>
    __device__ __forceinline__ void tile(uint32_t xs, const InstView &v, int br0, int bc0)
    {
        const uint32_t qb = (uint32_t)v.Q * E;
#pragma unroll
        for (int i = 0; i < PR; ++i) {
#pragma unroll
            for (int j = 0; j < PC; ++j) {
                const bool there = !(kRR && i == PR - 1 && shortR) && !(kRC && j == PC - 1 && shortC);
                const uint32_t a = xs + (uint32_t)((br0 + i) * v.Wd + bc0 + j) * E;
#pragma unroll
                for (int g = 0; g < 4; ++g) {
                    S &s = x[at(2 * i + (g >> 1), 2 * j + (g & 1))];
                    if constexpr (kLoad) {
                        if (there) {
                            s = lds_site<Store, K>(a + g * qb);
                            flip(s, g == 0 || g == 3);
                        } else {
#pragma unroll
                            for (int h = 0; h < S::NW; ++h) s.w[h] = 0;
                        }
                    } else {
                        S o = s;
                        flip(o, g == 0 || g == 3);
                        if (there) sts_site<Store, K>(a + g * qb, o);
                    }
                }
            }
        }
    }
};

template <typename Store, int K, int PR, int PC, bool kRagged>
__device__ __forceinline__ void run_segment_patch(const InstView &v, const Segment &sg, unsigned char *smem,
                                                  int *s_skip, int32_t *ready, int32_t *err, uint64_t wait_limit_ns)
{
    using Pt = Patch<Store, K, PR, PC, kRagged>;
    constexpr bool kQ = std::is_same<Store, uint16_t>::value;
    const Tile<Store, K> t = carve<Store, K>(smem, v.n, v.P, false);
    const int tid = threadIdx.x;
    if (!seg_begin<Store, K>(v, sg, t, s_skip, ready, err, wait_limit_ns)) return;
    if (sg.s_begin > sg.s_end) {  // a readout of the stored state
        seg_end<Store, K>(v, sg, t, ready);
        return;
    }
    const int GR = v.pgr, GC = v.pgc;
#ifdef COSM_CHECKS
    // the patches tile the blocks, one thread each, and their published sites
    // fit the tile
    if (tid == 0 && v.check) {
        const bool bad = GR < 1 || GC < 1 || GR * GC > (int)blockDim.x || v.Wd < 1 || v.Q * 4 != v.n ||
                         GR * PR - (GR - v.pfr) != v.Q / v.Wd || GC * PC - (GC - v.pfc) != v.Wd ||
                         GR * GC * Pt::NE > v.n || (!kRagged && (GR != v.pfr || GC != v.pfc));
        if (bad) atomicOr(v.check, 2);
    }
#endif
    const bool active = tid < GR * GC;
    const int pr = active ? tid / GC : 0, pc = active ? tid - pr * GC : 0;
    const uint32_t xs = (uint32_t)__cvta_generic_to_shared(t.xs);
    Pt p;
    // the first pfr rows (pfc columns) of patches are whole, the rest one block shorter
    const int br0 = pr * PR - max(0, pr - v.pfr), bc0 = pc * PC - max(0, pc - v.pfc);
    p.shortR = Pt::kRR && pr >= v.pfr;
    p.shortC = Pt::kRC && pc >= v.pfc;
    {
        const bool seamC = pc == GC - 1, seamR = pr == GR - 1;
        if constexpr (kQ) {
            // one in both halves where the pair's roles swap
            p.ch0 = seamC ? 0x00010001ull : 0ull;
            p.ch1 = seamC && p.shortC ? 0x00010001ull : 0ull;
            p.cv0 = seamR ? 0x00010001ull : 0ull;
            p.cv1 = seamR && p.shortR ? 0x00010001ull : 0ull;
        } else {
            p.ch0 = seamC ? kMinusTwo2 : kTwo2;
            p.ch1 = seamC && p.shortC ? kMinusTwo2 : kTwo2;
            p.cv0 = seamR ? kMinusTwo2 : kTwo2;
            p.cv1 = seamR && p.shortR ? kMinusTwo2 : kTwo2;
        }
        const int rr = pr + 1 == GR ? 0 : pr + 1, cc = pc + 1 == GC ? 0 : pc + 1;
        constexpr uint32_t stride = Pt::NE * Pt::E;
        p.own = xs + (uint32_t)(pr * GC + pc) * stride;
        p.right = xs + (uint32_t)(pr * GC + cc) * stride;
        p.below = xs + (uint32_t)(rr * GC + pc) * stride;
        p.diag = xs + (uint32_t)(rr * GC + cc) * stride;
    }
    if (active) {
        const int T = GR * GC;
#pragma unroll
        for (int k = 0; k < Pt::NWT; ++k) p.wt[k] = __ldg(v.pwt + k * T + tid);
        p.template tile<true>(xs, v, br0, bc0);
    }
    __syncthreads();  // the published sites take the place of the tile
    Stretches st(v);
    const uint32_t rep0 = (uint32_t)sg.tile * K;
    const uint32_t s1 = (uint32_t)sg.s_end;  // below 2^31
    const int wrap_p = sizeof(Store) == 2 ? 1 : max(v.wrap_p, 1);
    SweepConsts c;
    c.D = t.D;
    c.E = (int)st.E;
    c.P1 = v.P + 1;
    c.W2 = 2.0f * v.window;
    c.qwin = v.qwin;
    for (uint32_t s = (uint32_t)sg.s_begin; s <= s1;) {
        int to_twist;
        const uint32_t end = st.template begin<kQ, K>(v, t.D, s, s1, rep0, &to_twist);
        int to_wrap = sweeps_to_wrap(s, wrap_p);
        const float2 *ap = v.alpha_tab + ((int64_t)s - v.alpha_base);
        float2 at = __ldg(ap);
        const int period = (int)st.period;
        c.k = -1;
#pragma unroll 1
        for (int left = (int)(end - s); left >= 0; --left) {
            c.dwt = to_twist == 0;
            c.wrap = to_wrap == 0;
            if (c.dwt) {
                ++c.k;
                to_twist = period;
            }
            if (c.wrap) to_wrap = wrap_p;
            --to_twist;
            --to_wrap;
            if constexpr (kQ) {
                const uint32_t aq = (uint32_t)__float2int_rn(at.x);
                c.a1 = both_halves(aq);
                c.n1 = both_halves(0u - aq);
            } else {
                c.a1 = __float_as_uint(at.x);
            }
            c.step = at.y;
            if (left > 0) at = __ldg(++ap);
            if (active) {
                p.template evens<true>(c);
                p.template evens<false>(c);
                p.publish();
            }
            __syncthreads();
            if (active) {
                p.borrow();
                p.odd_pass(c);
                p.give_back();
            }
            __syncthreads();
            if (active) p.take_back();
        }
        if (st.readout_after(end)) {
            __syncthreads();  // the tile takes the place of the published sites
            if (active) p.template tile<false>(xs, v, br0, bc0);
            tile_readout<Store, K>(v, sg.tile, t, (int)((end - 1) / st.track), true);
            __syncthreads();
        }
        s = end + 1;
    }
    __syncthreads();
    if (active) p.template tile<false>(xs, v, br0, bc0);
    __syncthreads();
    seg_end<Store, K>(v, sg, t, ready);
}

// One kernel for single runs (segment lists) and queues (batch, serving).
template <typename Store, int K, int PR, int PC, bool kRagged>
__global__ void __launch_bounds__(patch_max_threads(PR, PC, K *(int)sizeof(Store)))
    patch_kernel(const KernelArgs a, const BatchArgs b)
{
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int s_skip, s_unit;
    if (b.units == nullptr) {
        for (int si = a.seg_off[blockIdx.x]; si < a.seg_off[blockIdx.x + 1]; ++si) {
            const Segment sg = a.segs[si];
            run_segment_patch<Store, K, PR, PC, kRagged>(a.v, sg, smem, &s_skip, a.ready, a.err, a.wait_limit_ns);
            __syncthreads();
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
        run_segment_patch<Store, K, PR, PC, kRagged>(b.insts[bu.inst], sg, smem, &s_skip, nullptr, nullptr, 0);
    }
}

template <typename Store, int K, int PR, int PC, bool kRagged>
int patch_call(const PatchCall &c)
{
    static SmemLimit lim;
    auto fn = patch_kernel<Store, K, PR, PC, kRagged>;
    constexpr int most = patch_max_threads(PR, PC, K * (int)sizeof(Store));
    if (c.what == PatchCall::OCCUPANCY) return occupancy_of(lim, fn, most, c.threads, c.smem);
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
int patch_dispatch(const PatchCall &c)
{
    constexpr bool float16 = sizeof(Store) == 2 && !std::is_same<Store, uint16_t>::value;
#define PATCH_CASE(I, R, C)                                                                  \
    if constexpr (patch_built(float16, K, R, C))                                             \
        if (c.shape == (I))                                                                  \
            return c.ragged ? patch_call<Store, K, R, C, (R) * (C) != 1>(c) : patch_call<Store, K, R, C, false>(c);
    COSM_PATCH_SHAPES(PATCH_CASE)
#undef PATCH_CASE
    return c.what == PatchCall::OCCUPANCY ? 0 : -1;
}

}  // namespace cosm
