// Host runtime behind the C ABI of include/cosm.h: handles, device layout,
// the work schedule of replica tiles over resident CTAs, and launches.
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdlib>
#include <cstring>
#include <string>
#include <vector>

#include "../../include/cosm.h"
#include "cosm_handle.h"
#include "cosm_internal.h"

using namespace cosm;

static thread_local std::string g_err;

int cosm::fail(int code, const std::string &msg)
{
    g_err = msg;
    return code;
}

extern "C" const char *cosm_last_error(void) { return g_err.c_str(); }

void cosm::set_last_error(const std::string &msg) { g_err = msg; }

extern "C" void cosm_default_params(cosm_params *p)
{
    if (!p) return;
    std::memset(p, 0, sizeof(*p));
    p->alpha0_deg = 14.0;
    p->dwt_ratio = 0.5;
    p->dwt_period = 3;
    p->window_deg = 90.0;
    p->n_bisectors = 100;
    p->storage = COSM_F32;
    p->flags = 0;
}

static int check_params(const cosm_params *p)
{
    if (!p) return fail(COSM_ERR_INVALID_ARG, "params is NULL");
    if (!(p->alpha0_deg >= 0.0 && p->alpha0_deg < 180.0))
        return fail(COSM_ERR_INVALID_ARG, "alpha0_deg must be in [0, 180)");
    if (!(p->dwt_ratio >= 0.0 && p->dwt_ratio <= 16.0))
        return fail(COSM_ERR_INVALID_ARG, "dwt_ratio must be in [0, 16]");
    if (p->dwt_period < 0) return fail(COSM_ERR_INVALID_ARG, "dwt_period must be >= 0");
    if (!(p->window_deg > 0.0 && p->window_deg <= 180.0))
        return fail(COSM_ERR_INVALID_ARG, "window_deg must be in (0, 180]");
    if (p->n_bisectors < 1 || p->n_bisectors > kMaxBisectors)
        return fail(COSM_ERR_INVALID_ARG, "n_bisectors must be in [1, 256]");
    if (p->storage != COSM_F32 && p->storage != COSM_F16 && p->storage != COSM_Q16 && p->storage != COSM_BF16)
        return fail(COSM_ERR_INVALID_ARG, "storage must be COSM_F32, COSM_F16, COSM_Q16 or COSM_BF16");
    if (p->flags & ~(COSM_NO_DWT | COSM_NO_SCS | COSM_DWT_RANDOM_DIR | COSM_OPT_BISECTOR))
        return fail(COSM_ERR_INVALID_ARG, "unknown flags");
    if (p->track_period < 0) return fail(COSM_ERR_INVALID_ARG, "track_period must be >= 0");
    return COSM_OK;
}

// Features of single-instance runs only (local fields, tracking, optimal
// bisector): the batch and serving paths reject them up front.
int cosm::single_only(const cosm_graph_desc *g, const cosm_params *p)
{
    if (g && g->h) return fail(COSM_ERR_INVALID_ARG, "local fields are supported by single instances only");
    if (p && p->track_period > 0)
        return fail(COSM_ERR_INVALID_ARG, "mid-anneal tracking is supported by single instances only");
    if (p && (p->flags & COSM_OPT_BISECTOR))
        return fail(COSM_ERR_INVALID_ARG, "the optimal bisector is supported by single instances only");
    return COSM_OK;
}

extern "C" int cosm_validate_partition(int32_t n, int64_t m, const int32_t *src, const int32_t *dst,
                                       int32_t n_colors, const int32_t *color)
{
    if (!src || !dst || !color || n < 1 || m < 0) return fail(COSM_ERR_INVALID_ARG, "bad arguments");
    std::string why;
    int rc = validate_partition(n, m, src, dst, n_colors, color, why);
    if (rc) return fail(rc, why);
    return COSM_OK;
}

extern "C" int cosm_color_greedy(int32_t n, int64_t m, const int32_t *src, const int32_t *dst,
                                 int32_t *color, int32_t *n_colors)
{
    if (!src || !dst || !color || !n_colors || n < 1 || m < 0)
        return fail(COSM_ERR_INVALID_ARG, "bad arguments");
    for (int64_t e = 0; e < m; ++e)
        if (src[e] < 0 || src[e] >= n || dst[e] < 0 || dst[e] >= n || src[e] == dst[e])
            return fail(COSM_ERR_INVALID_ARG, "edge endpoint out of range or loop");
    return color_greedy(n, m, src, dst, color, n_colors);
}

extern "C" int cosm_color_misra_gries(int32_t n, int64_t m, const int32_t *src, const int32_t *dst,
                                      int32_t *color, int32_t *n_colors)
{
    if (!src || !dst || !color || !n_colors || n < 1 || m < 0)
        return fail(COSM_ERR_INVALID_ARG, "bad arguments");
    for (int64_t e = 0; e < m; ++e)
        if (src[e] < 0 || src[e] >= n || dst[e] < 0 || dst[e] >= n || src[e] == dst[e])
            return fail(COSM_ERR_INVALID_ARG, "edge endpoint out of range or loop");
    int rc = color_misra_gries(n, m, src, dst, color, n_colors);
    if (rc) return fail(rc, "Misra-Gries colouring failed (multigraph?)");
    return COSM_OK;
}

extern "C" int cosm_color_torus2d(int32_t L1, int32_t L2, int64_t m, const int32_t *src,
                                  const int32_t *dst, int32_t *color)
{
    if (!src || !dst || !color) return fail(COSM_ERR_INVALID_ARG, "bad arguments");
    int rc = color_torus2d(L1, L2, m, src, dst, color);
    if (rc) return fail(rc, "not an even-sided 2D torus edge list");
    return COSM_OK;
}

extern "C" int cosm_color_torus3d(int32_t L1, int32_t L2, int32_t L3, int64_t m, const int32_t *src,
                                  const int32_t *dst, int32_t *color)
{
    if (!src || !dst || !color) return fail(COSM_ERR_INVALID_ARG, "bad arguments");
    int rc = color_torus3d(L1, L2, L3, m, src, dst, color);
    if (rc) return fail(rc, "not an even-sided 3D torus edge list");
    return COSM_OK;
}

// ------------------------------------------------------------------ create

// Waits for the copies made on the legacy stream. cudaMemcpy from pageable
// memory may return while its transfer is still queued there, and a stream
// created non-blocking -- a batch's, a server's, a caller's -- does not wait
// for the legacy stream: whatever is copied this way for a later launch has
// arrived before the call that copies it returns.
static int settle()
{
    CK(cudaStreamSynchronize(nullptr));
    return COSM_OK;
}

extern "C" void cosm_destroy(cosm_handle *h)
{
    if (!h) return;
    if (h->stream || h->have_state) cudaStreamSynchronize(h->stream);
    h->d_ij.release(); h->d_w.release(); h->d_orig.release(); h->d_slot.release(); h->d_off.release(); h->d_state.release();
    h->d_cut.release(); h->d_bestp.release(); h->d_alpha.release(); h->d_segs.release();
    h->d_segoff.release(); h->d_ready.release(); h->d_err.release(); h->d_best.release();
    h->d_spins.release();
    h->d_wnib.release();
    for (auto &b : h->d_pwt) b.release();
    for (auto &t : h->tables) t->release();
    h->d_h.release(); h->d_hlist.release(); h->d_energy.release(); h->d_bisB.release(); h->d_trace.release();
    h->d_bits.release(); h->d_qbuf.release(); h->d_delta.release(); h->d_items.release(); h->d_stage.release();
    delete h;
}

// The implicit-index 2D lattice kernel applies when the graph is an
// even-sided torus given with the regular 4-colour pattern, all weights are
// +-1 and the update is the sequential one. It walks 2x2 blocks in two
// passes; this builds each block's four weight bits from the edge list, in
// the kernel's edge order (even pass: A-B, C-D, A-C, B-D; odd pass: D-C,
// B-A, D-B, C-A over the shifted block).
static int setup_lattice2d(cosm_handle *h, const std::vector<int32_t> &pattern)
{
    const Graph &g = h->g;
    h->mode = (h->prm.flags & COSM_NO_SCS) ? MODE_ACCUM_ : MODE_GENERAL_;
    if (std::getenv("COSM_NO_LATTICE") || h->fields) return COSM_OK;
    // the full torus only (every block needs its four edges)
    if (!h->lattice || g.dims[2] != 0 || h->mode != MODE_GENERAL_ || h->C != 4 || g.m != 2 * (int64_t)g.n)
        return COSM_OK;
    for (int64_t e = 0; e < g.m; ++e)
        if (g.w[(size_t)e] != 1 && g.w[(size_t)e] != -1) return COSM_OK;
    if (pattern != g.color) return COSM_OK;  // another colour order changes the dynamics
    const int32_t Q = g.n / 4, Wd = g.dims[1] / 2;
    // a slot's edge of each colour: the other end and the weight (a vertex
    // of the torus has one edge of each of the four colours)
    std::vector<int32_t> other((size_t)g.n * 4, -1);
    std::vector<int8_t> wt((size_t)g.n * 4);
    for (int64_t e = 0; e < g.m; ++e) {
        const int32_t a = h->slot_of[(size_t)g.src[(size_t)e]], b = h->slot_of[(size_t)g.dst[(size_t)e]];
        const size_t ka = (size_t)a * 4 + g.color[(size_t)e], kb = (size_t)b * 4 + g.color[(size_t)e];
        other[ka] = b;
        other[kb] = a;
        wt[ka] = wt[kb] = (int8_t)g.w[(size_t)e];
    }
    auto weight = [&](int32_t slot_a, int32_t slot_b) -> int32_t {
        for (size_t k = (size_t)slot_a * 4; k < (size_t)slot_a * 4 + 4; ++k)
            if (other[k] == slot_b) return wt[k];
        return 0;
    };
    std::vector<uint8_t> nib((size_t)2 * Q, 0);
    for (int32_t f = 0; f < Q; ++f) {
        const int32_t A = f, B = Q + f, Cc = 2 * Q + f, D = 3 * Q + f;
        const int32_t even[4][2] = {{A, B}, {Cc, D}, {A, Cc}, {B, D}};
        const int32_t gcol = (f % Wd == Wd - 1) ? f + 1 - Wd : f + 1;
        const int32_t hrow = (f + Wd) % Q, gh = (gcol + Wd) % Q;
        const int32_t odd[4][2] = {{D, 2 * Q + gcol}, {Q + hrow, gh}, {D, Q + hrow}, {2 * Q + gcol, gh}};
        for (int k = 0; k < 4; ++k) {
            const int32_t we = weight(even[k][0], even[k][1]), wo = weight(odd[k][0], odd[k][1]);
            if (we == 0 || wo == 0) return fail(COSM_ERR_INVALID_ARG, "lattice block edge missing");
            if (we == -1) nib[(size_t)f] |= (uint8_t)(1u << k);
            if (wo == -1) nib[(size_t)Q + f] |= (uint8_t)(1u << k);
        }
    }
    int rc = h->d_wnib.ensure(nib.size());
    if (rc) return rc;
    CK(cudaMemcpy(h->d_wnib.p, nib.data(), nib.size(), cudaMemcpyHostToDevice));
    h->nib.swap(nib);
    h->Q = Q;
    h->Wd = Wd;
    h->mode = MODE_LATTICE2D_;
    return COSM_OK;
}

// Order of one colour class's edges for the edge-list kernel. A warp takes
// 32 consecutive edges; with two binary32 replicas per slot (8 bytes) a
// half-warp's 16 loads of source phases, and its 16 loads of destination
// phases, are each conflict-free in shared memory when their slots are
// distinct modulo 16. Edges are grouped accordingly: the class is read as a
// bipartite multigraph between source residues and destination residues
// (slot mod 16), properly edge-coloured with its maximum degree of colours
// by Konig's alternating-path method, and each colour class (at most one
// edge per residue on either side) becomes a run of consecutive edges,
// largest first, in source-residue order. Edges of one colour share no
// vertex, so their order changes no result; it only changes which phases a
// half-warp touches together.
static void balance_banks(int64_t *e, int64_t cnt, const std::vector<int32_t> &ss,
                          const std::vector<int32_t> &ds)
{
    constexpr int R = 16;
    if (cnt < 32 || cnt > ((int64_t)1 << 20)) return;
    std::vector<int32_t> A((size_t)cnt), B((size_t)cnt);
    int deg[2 * R] = {0};
    for (int64_t k = 0; k < cnt; ++k) {
        A[(size_t)k] = ss[(size_t)e[k]] & (R - 1);
        B[(size_t)k] = R + (ds[(size_t)e[k]] & (R - 1));
        ++deg[A[(size_t)k]];
        ++deg[B[(size_t)k]];
    }
    int D = 0;
    for (int v = 0; v < 2 * R; ++v) D = std::max(D, deg[v]);
    const int Wd = (D + 63) / 64;
    std::vector<int32_t> at((size_t)2 * R * D, -1);  // at[v D + c]: edge of colour c at residue v
    std::vector<uint64_t> freeb((size_t)2 * R * Wd, ~0ull);
    std::vector<int32_t> color((size_t)cnt, -1);
    auto mark = [&](int v, int c, bool used) {
        uint64_t &w = freeb[(size_t)v * Wd + c / 64];
        if (used) w &= ~(1ull << (c % 64));
        else w |= 1ull << (c % 64);
    };
    auto first_free = [&](int v, int u) {  // first colour free at v (and at u when u >= 0)
        for (int w = 0; w < Wd; ++w) {
            uint64_t f = freeb[(size_t)v * Wd + w];
            if (u >= 0) f &= freeb[(size_t)u * Wd + w];
            if (w == Wd - 1 && D % 64) f &= (1ull << (D % 64)) - 1;
            if (f) return w * 64 + __builtin_ctzll(f);
        }
        return -1;
    };
    auto put = [&](int32_t k, int c) {
        color[(size_t)k] = c;
        at[(size_t)A[(size_t)k] * D + c] = k;
        at[(size_t)B[(size_t)k] * D + c] = k;
        mark(A[(size_t)k], c, true);
        mark(B[(size_t)k], c, true);
    };
    auto take = [&](int32_t k) {
        const int c = color[(size_t)k];
        at[(size_t)A[(size_t)k] * D + c] = -1;
        at[(size_t)B[(size_t)k] * D + c] = -1;
        mark(A[(size_t)k], c, false);
        mark(B[(size_t)k], c, false);
    };
    std::vector<int32_t> path;
    for (int32_t k = 0; k < (int32_t)cnt; ++k) {
        const int a = A[(size_t)k], b = B[(size_t)k];
        int c = first_free(a, b);
        if (c < 0) {
            // colour al free at a, be free at b; swap al/be along the
            // alternating path that starts at b with its al-edge (it never
            // reaches a), after which al is free at both ends
            const int al = first_free(a, -1), be = first_free(b, -1);
            path.clear();
            int v = b, cur = al;
            for (;;) {
                const int32_t k2 = at[(size_t)v * D + cur];
                if (k2 < 0) break;
                path.push_back(k2);
                v = (B[(size_t)k2] == v) ? A[(size_t)k2] : B[(size_t)k2];
                cur = (cur == al) ? be : al;
            }
            std::vector<int> old(path.size());
            for (size_t i = 0; i < path.size(); ++i) {
                old[i] = color[(size_t)path[i]];
                take(path[i]);
            }
            for (size_t i = 0; i < path.size(); ++i) put(path[i], old[i] == al ? be : al);
            c = al;
        }
        put(k, c);
    }
    std::vector<std::vector<int32_t>> groups((size_t)D);
    for (int32_t k = 0; k < (int32_t)cnt; ++k) groups[(size_t)color[(size_t)k]].push_back(k);
    std::stable_sort(groups.begin(), groups.end(),
                     [](const std::vector<int32_t> &x, const std::vector<int32_t> &y) { return x.size() > y.size(); });
    std::vector<int64_t> out;
    out.reserve((size_t)cnt);
    for (auto &g : groups) {
        std::sort(g.begin(), g.end(), [&](int32_t x, int32_t y) { return A[(size_t)x] < A[(size_t)y]; });
        for (int32_t k : g) out.push_back(e[k]);
    }
    std::copy(out.begin(), out.end(), e);
}

extern "C" int cosm_create(const cosm_graph_desc *gd, const cosm_params *p, cosm_handle **out)
{
    NvtxRange range("cosm_create");
    if (!gd || !out) return fail(COSM_ERR_INVALID_ARG, "NULL argument");
    *out = nullptr;
    int rc = check_params(p);
    if (rc) return rc;
    if (!gd->src || !gd->dst || !gd->w) return fail(COSM_ERR_INVALID_ARG, "NULL edge arrays");
    if (gd->n < 2 || gd->n > kMaxVertices) return fail(COSM_ERR_INVALID_ARG, "n must be in [2, 65536]");
    if (gd->m < 1 || gd->m > ((int64_t)1 << 26)) return fail(COSM_ERR_INVALID_ARG, "m must be in [1, 2^26]");
    cosm_handle *h = new (std::nothrow) cosm_handle();
    if (!h) return fail(COSM_ERR_NOMEM, "host allocation failed");
    h->prm = *p;
    Graph &g = h->g;
    g.n = gd->n;
    g.m = gd->m;
    g.src.assign(gd->src, gd->src + gd->m);
    g.dst.assign(gd->dst, gd->dst + gd->m);
    g.w.assign(gd->w, gd->w + gd->m);
    for (int k = 0; k < 3; ++k) g.dims[k] = gd->dims[k];
    std::string why;
    rc = validate_graph(g, why);
    if (rc) { delete h; return fail(rc, why); }
    if (gd->h) {
        if (p->flags & COSM_OPT_BISECTOR) {
            delete h;
            return fail(COSM_ERR_INVALID_ARG, "local fields fix the readout; COSM_OPT_BISECTOR does not apply");
        }
        int64_t mag = 0;
        for (int64_t e = 0; e < g.m; ++e) mag += std::abs(g.w[(size_t)e]);
        for (int32_t v = 0; v < g.n; ++v) {
            if (gd->h[v] > 32767 || gd->h[v] < -32767) {
                delete h;
                return fail(COSM_ERR_INVALID_ARG, "local field " + std::to_string(v) + " exceeds 32767 in magnitude");
            }
            mag += std::abs(gd->h[v]);
        }
        if (mag >= ((int64_t)1 << 31)) {
            delete h;
            return fail(COSM_ERR_INVALID_ARG, "sum of |w| and |h| must be below 2^31");
        }
        h->fields = true;
    }
    // partition: given, or coloured here (lattice pattern, else greedy)
    g.color.assign((size_t)g.m, 0);
    if (gd->color) {
        g.color.assign(gd->color, gd->color + gd->m);
        g.C = gd->n_colors;
    } else if (g.dims[0] > 0 && g.dims[2] == 0 &&
               color_torus2d(g.dims[0], g.dims[1], g.m, g.src.data(), g.dst.data(), g.color.data()) == 0) {
        g.C = 4;
    } else if (g.dims[0] > 0 && g.dims[2] > 0 &&
               color_torus3d(g.dims[0], g.dims[1], g.dims[2], g.m, g.src.data(), g.dst.data(),
                             g.color.data()) == 0) {
        g.C = 6;
    } else {
        color_greedy(g.n, g.m, g.src.data(), g.dst.data(), g.color.data(), &g.C);
    }
    rc = validate_partition(g.n, g.m, g.src.data(), g.dst.data(), g.C, g.color.data(), why);
    if (rc) { delete h; return fail(rc, why); }
    h->C = g.C;
    // shared-memory layout: lattice sublattices when the hint matches
    h->slot_of.resize((size_t)g.n);
    std::vector<int32_t> pattern;
    if (g.dims[0] > 0) {
        if (!lattice_relabel(g, h->slot_of, pattern, why)) { delete h; return fail(COSM_ERR_INVALID_ARG, why); }
        h->lattice = true;
    } else {
        for (int32_t v = 0; v < g.n; ++v) h->slot_of[(size_t)v] = v;
    }
    h->orig_of.assign((size_t)g.n, 0);
    for (int32_t v = 0; v < g.n; ++v) h->orig_of[(size_t)h->slot_of[(size_t)v]] = v;
    // colour-major edge records, each colour sorted by the slot of src
    // (stable counting sorts by slot, then by colour: comparing edges through
    // their indices was half of creating a 100 x 100 instance)
    std::vector<int64_t> order((size_t)g.m);
    {
        std::vector<int64_t> by_slot((size_t)g.m);
        std::vector<int64_t> at((size_t)std::max(g.n, g.C) + 1, 0);
        for (int64_t e = 0; e < g.m; ++e) ++at[(size_t)h->slot_of[(size_t)g.src[(size_t)e]] + 1];
        for (int32_t v = 0; v < g.n; ++v) at[(size_t)v + 1] += at[(size_t)v];
        for (int64_t e = 0; e < g.m; ++e)
            by_slot[(size_t)at[(size_t)h->slot_of[(size_t)g.src[(size_t)e]]]++] = e;
        std::fill(at.begin(), at.end(), 0);
        for (int64_t e = 0; e < g.m; ++e) ++at[(size_t)g.color[(size_t)e] + 1];
        for (int32_t c = 0; c < g.C; ++c) at[(size_t)c + 1] += at[(size_t)c];
        for (int64_t e : by_slot) order[(size_t)at[(size_t)g.color[(size_t)e]]++] = e;
    }
    // instances that never take record tables (whose rows are arranged for
    // their own tile width) have their colours' edges ordered here
    int32_t wmax = 0;
    for (int64_t e = 0; e < g.m; ++e) wmax = std::max(wmax, std::abs(g.w[(size_t)e]));
    const bool plain = (p->flags & COSM_NO_SCS) || (p->storage != COSM_Q16 && wmax > 63) ||
                       std::getenv("COSM_STAGE") || std::getenv("COSM_SPLIT_W");
    {
        std::vector<int32_t> ss((size_t)g.m), ds((size_t)g.m);
        for (int64_t e = 0; e < g.m; ++e) {
            ss[(size_t)e] = h->slot_of[(size_t)g.src[(size_t)e]];
            ds[(size_t)e] = h->slot_of[(size_t)g.dst[(size_t)e]];
        }
        int64_t a = 0;
        while (a < g.m) {
            int64_t z = a;
            while (z < g.m && g.color[(size_t)order[(size_t)z]] == g.color[(size_t)order[(size_t)a]]) ++z;
            if (plain && !std::getenv("COSM_SRC_ORDER")) balance_banks(order.data() + a, z - a, ss, ds);
            a = z;
        }
    }
    std::vector<uint32_t> ij((size_t)g.m);
    std::vector<int8_t> wv((size_t)g.m);
    std::memset(h->off, 0, sizeof(h->off));
    for (int64_t k = 0; k < g.m; ++k) {
        const int64_t e = order[(size_t)k];
        ij[(size_t)k] = (uint32_t)h->slot_of[(size_t)g.src[(size_t)e]] |
                        ((uint32_t)h->slot_of[(size_t)g.dst[(size_t)e]] << 16);
        wv[(size_t)k] = (int8_t)g.w[(size_t)e];
        h->off[g.color[(size_t)e] + 1]++;
        h->W += g.w[(size_t)e];
    }
    for (int c = 0; c < h->C; ++c) h->off[c + 1] += h->off[c];
    h->wmax = wmax;
    h->h_ij = ij;
    h->h_wv = wv;
    h->wbound = std::min(colour_weight_bound(h->off, h->C, wv.data(), gd->h, g.n),
                         vertex_weight_bound(g.n, g.m, g.src.data(), g.dst.data(), g.w.data(), gd->h));
    // device copies
    cudaGetDevice(&h->device);
    cudaDeviceGetAttribute(&h->num_sms, cudaDevAttrMultiProcessorCount, h->device);
    // records and weights padded with zeros past a multiple of 16 edges: the
    // staged edge-list sweep copies whole 16-byte chunks around each colour
    const size_t m_pad = (((size_t)g.m + 15) & ~(size_t)15) + 16;
    ij.resize(m_pad, 0u);
    wv.resize(m_pad, 0);
    if ((rc = h->d_ij.ensure(m_pad)) || (rc = h->d_w.ensure(m_pad)) ||
        (rc = h->d_orig.ensure((size_t)g.n)) || (rc = h->d_off.ensure((size_t)h->C + 1)) ||
        (rc = h->d_err.ensure(1)) ||
        (rc = h->d_best.ensure(4)) || (rc = h->d_spins.ensure((size_t)g.n))) {
        cosm_destroy(h);
        return rc;
    }
    if (cudaMemcpy(h->d_ij.p, ij.data(), ij.size() * 4, cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemcpy(h->d_w.p, wv.data(), wv.size(), cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemcpy(h->d_orig.p, h->orig_of.data(), (size_t)g.n * 4, cudaMemcpyHostToDevice) !=
            cudaSuccess ||
        cudaMemcpy(h->d_off.p, h->off, ((size_t)h->C + 1) * 4, cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemset(h->d_err.p, 0, 4) != cudaSuccess) {
        cosm_destroy(h);
        return fail(COSM_ERR_CUDA, "copying the graph to the device failed");
    }
    if (h->lattice) {
        std::vector<uint16_t> slots(h->slot_of.begin(), h->slot_of.end());
        if ((rc = h->d_slot.ensure(slots.size()))) {
            cosm_destroy(h);
            return rc;
        }
        if (cudaMemcpy(h->d_slot.p, slots.data(), slots.size() * 2, cudaMemcpyHostToDevice) != cudaSuccess) {
            cosm_destroy(h);
            return fail(COSM_ERR_CUDA, "copying the graph to the device failed");
        }
    }
    if (h->fields) {
        std::vector<int32_t> hs((size_t)g.n);
        for (int32_t v = 0; v < g.n; ++v) hs[(size_t)h->slot_of[(size_t)v]] = gd->h[v];
        // the vertices with a field, as (slot, field) pairs for the sweeps
        std::vector<int2> list;
        for (int32_t v = 0; v < g.n; ++v)
            if (hs[(size_t)v]) list.push_back(make_int2(v, hs[(size_t)v]));
        h->n_fields = (int32_t)list.size();
        if ((rc = h->d_h.ensure((size_t)g.n)) || (rc = h->d_hlist.ensure(list.size()))) {
            cosm_destroy(h);
            return rc;
        }
        if (cudaMemcpy(h->d_h.p, hs.data(), hs.size() * 4, cudaMemcpyHostToDevice) != cudaSuccess ||
            (!list.empty() && cudaMemcpy(h->d_hlist.p, list.data(), list.size() * sizeof(int2),
                                         cudaMemcpyHostToDevice) != cudaSuccess)) {
            cosm_destroy(h);
            return fail(COSM_ERR_CUDA, "copying the local fields to the device failed");
        }
    }
    if ((rc = setup_lattice2d(h, pattern)) || (rc = settle())) {
        cosm_destroy(h);
        return rc;
    }
    *out = h;
    return COSM_OK;
}

// ------------------------------------------------------------------ layout

int cosm::env_int(const char *name, int dflt)
{
    const char *s = std::getenv(name);
    return (s && *s) ? std::atoi(s) : dflt;
}

static int patch_call_for(int storage, int K, const PatchCall &c)
{
    const int none = c.what == PatchCall::OCCUPANCY ? 0 : -1;
    switch (storage) {
    case COSM_F32: return K == 2 ? patch_call_f32_k2(c) : none;
    case COSM_F16: return K == 2 ? patch_call_f16_k2(c) : K == 4 ? patch_call_f16_k4(c) : none;
    case COSM_BF16: return K == 2 ? patch_call_bf16_k2(c) : K == 4 ? patch_call_bf16_k4(c) : none;
    default: return K == 2 ? patch_call_q16_k2(c) : K == 4 ? patch_call_q16_k4(c) : none;
    }
}

static int patch_occupancy(int storage, int K, int shape, bool ragged, int threads, size_t smem)
{
    return patch_call_for(storage, K, PatchCall{PatchCall::OCCUPANCY, shape, ragged, threads, smem, 0, false, nullptr,
                                                nullptr, nullptr});
}

static int edges_call_for(int storage, const EdgesCall &c)
{
    switch (storage) {
    case COSM_F32: return edges_call_f32(c);
    case COSM_F16: return edges_call_f16(c);
    case COSM_BF16: return edges_call_bf16(c);
    default: return edges_call_q16(c);
    }
}

static int edges_occupancy(int storage, int K, int format, int threads, size_t smem)
{
    return edges_call_for(storage, EdgesCall{EdgesCall::OCCUPANCY, K, format, threads, smem, 0, false, nullptr, nullptr,
                                             nullptr});
}

int cosm::kernel_occupancy(const cosm_handle *h, int threads, size_t smem, bool queue)
{
    if (h->format >= 0) return edges_occupancy(h->prm.storage, h->K, h->format, threads, smem);
    if (h->shape >= 0) return patch_occupancy(h->prm.storage, h->K, h->shape, h->ragged, threads, smem);
    return queue ? batch_occupancy(h->prm.storage, h->K, h->mode, threads, smem)
                 : sweep_occupancy(h->prm.storage, h->K, h->mode, threads, smem);
}

int cosm::kernel_launch(const LaunchCfg &cfg, const KernelArgs &a, cudaStream_t st)
{
    if (cfg.format >= 0)
        return edges_call_for(cfg.storage, EdgesCall{EdgesCall::LAUNCH, cfg.K, cfg.format, cfg.threads, cfg.smem,
                                                     cfg.grid, cfg.cooperative, &a, nullptr, st});
    if (cfg.shape < 0) return sweep_launch(cfg, a, st);
    return patch_call_for(cfg.storage, cfg.K, PatchCall{PatchCall::LAUNCH, cfg.shape, cfg.ragged, cfg.threads,
                                                        cfg.smem, cfg.grid, cfg.cooperative, &a, nullptr, st});
}

int cosm::kernel_launch_queue(const LaunchCfg &cfg, const BatchArgs &b, cudaStream_t st)
{
    if (cfg.format >= 0)
        return edges_call_for(cfg.storage, EdgesCall{EdgesCall::LAUNCH, cfg.K, cfg.format, cfg.threads, cfg.smem,
                                                     cfg.grid, false, nullptr, &b, st});
    if (cfg.shape < 0) return batch_launch(cfg.storage, cfg.K, cfg.mode, cfg.grid, cfg.threads, cfg.smem, b, st);
    return patch_call_for(cfg.storage, cfg.K, PatchCall{PatchCall::LAUNCH, cfg.shape, cfg.ragged, cfg.threads,
                                                        cfg.smem, cfg.grid, false, nullptr, &b, st});
}

// How a side of B blocks splits into patches of at most P blocks: the grid,
// and how many patches are whole (the others are one block shorter). False
// when patches of P and P - 1 blocks cannot make up the side.
static bool split_side(int B, int P, int *grid, int *whole)
{
    *grid = (B + P - 1) / P;
    const int missing = *grid * P - B;
    if (missing > *grid || (P == 1 && missing)) return false;
    *whole = *grid - missing;
    return true;
}

// Modelled SM cycles per sweep of a run in a patch layout: the instructions of
// the warps that share an SM's schedulers at the issue rate the kernels
// reach, or one CTA's latency where those do not fill it, times the waves of
// tiles. Fitted to timings of 16 x 16 to 100 x 200 lattices, 32 to 2,048
// replicas (within 15 %): binary32 100 x 100, 1,024 replicas, shapes 2x5 /
// 2x4 / 2x3 / 2x2 measured 5.5 / 6.9 / 7.0 / 6.2 us per sweep, modelled 5.3 /
// 6.9 / 7.1 / 5.6.
static double patch_cost(int storage, int K, int R, int C, bool ragged, int warps, int occ, int replicas, int sms)
{
    const int NE = 2 * R + 2 * C - 1, words = K / 2;
    // instructions per 2x2 block and pass, per warp, the twist and the wrap
    // spread over their periods; instructions issued per scheduler and cycle
    const double block = storage == COSM_F32 ? 42.0 : storage == COSM_Q16 ? 12.0 + 26.0 * words : 8.0 + 62.0 * words;
    const double rate = storage == COSM_F32 ? 0.57 : storage == COSM_Q16 ? 0.62 : 0.60;
    const double inst = 2.0 * R * C * block + 4.0 * NE + 30.0 + (ragged ? 4.0 * NE : 0.0);
    const double tiles = std::ceil((double)replicas / K), slots = (double)occ * sms;
    const double together = std::max(1.0, std::ceil(std::min(tiles, slots) / sms));
    const double sweep = std::max(420.0 + 2.0 * inst, std::ceil(together * warps / 4.0) * inst / rate);
    return sweep * std::max(1.0, tiles / slots);
}

// The same for 16-bit floats on shared memory, the least over tiles of two,
// four and eight replicas (measured, 2x2 blocks per sweep and tile: 5.1 us for
// 5,000 blocks and 0.64 us for 64 at two replicas, 4.2 us for 2,500 at four,
// 8.2 us for 2,500 at eight). Binary32 and fixed point are faster in registers
// wherever a shape fits; 16-bit floats, whose widening, wraps and rounding
// outweigh the loads and stores saved, only up to about 100 x 100.
static double shared_cost_16(int blocks, int replicas, int sms)
{
    const double per[3] = {1.9, 3.4, 6.6}, latency[3] = {1200.0, 1000.0, 1000.0};
    double best = 1e300;
    for (int k = 0; k < 3; ++k) {
        const int K = 2 << k;
        if ((size_t)blocks * 8 * K > 220 * 1024) continue;  // the tile does not fit
        best = std::min(best, (per[k] * blocks + latency[k]) * std::max(1.0, std::ceil((double)replicas / K) / sms));
    }
    return best;
}

// Modelled costs within 10 % count as a tie between a tile and one of twice
// its width, which goes to the narrower one where narrow ties are asked for.
static double tie_weight(bool narrow_ties, int K) { return narrow_ties ? 1.0 + 0.1 * __builtin_ctz((unsigned)K) : 1.0; }

// Layout of a 2D lattice with its phases in registers (cosm_patch.cuh):
// among the shapes and tile widths that fit, the one whose modelled time per
// replica and sweep is lowest. Binary32 tiles hold two replicas, 16-bit ones
// four or two. Returns false when no shape fits (the lattice then keeps its
// phases in shared memory).
static bool choose_patch(cosm_handle *h, int replicas, int forceK, bool narrow_ties)
{
    const cosm_params &p = h->prm;
    const int BR = h->Q / h->Wd, BC = h->Wd, only = env_int("COSM_PATCH", -2);
    if (only == -1) return false;  // test hook: the shared-memory passes
    const int Ks[2] = {p.storage == COSM_F32 ? 2 : 4, 2};
    const bool f16 = p.storage == COSM_F16 || p.storage == COSM_BF16;
    double best = f16 && only < 0 ? shared_cost_16(h->Q, replicas, h->num_sms) : 1e300;
    for (int k = 0; k < (p.storage == COSM_F32 ? 1 : 2); ++k) {
        const int K = Ks[k];
        if (forceK && K != forceK) continue;
        const size_t smem = sweep_smem_bytes(p.storage, K, h->g.n, p.n_bisectors, MODE_LATTICE2D_);
        for (int s = 0; s < kPatchShapes; ++s) {
            if (only >= 0 && s != only) continue;
            if (!patch_built(f16, K, kPatchR[s], kPatchC[s])) continue;
            const int R = kPatchR[s], C = kPatchC[s], NE = 2 * R + 2 * C - 1;
            int gr, gc, fr, fc;
            if (!split_side(BR, R, &gr, &fr) || !split_side(BC, C, &gc, &fc)) continue;
            // the published sites take the place of the tile
            if ((int64_t)gr * gc * NE > h->g.n || gr * gc > 1024) continue;
            const bool ragged = fr != gr || fc != gc;
            const int T = (gr * gc + 31) / 32 * 32;
            const int occ = patch_occupancy(p.storage, K, s, ragged, T, smem);
            if (occ < 1) continue;
            const double cost = patch_cost(p.storage, K, R, C, ragged, T / 32, occ, replicas, h->num_sms) *
                                tie_weight(narrow_ties, K);
            if (cost < best) {
                best = cost;
                h->shape = s;
                h->ragged = ragged;
                h->K = K;
                h->threads = T;
                h->occupancy = occ;
                h->smem = smem;
                h->pgr = gr;
                h->pgc = gc;
                h->pfr = fr;
                h->pfc = fc;
            }
        }
    }
    return h->shape >= 0;
}

// Weight words of the chosen shape (InstView::pwt), from the block weight
// bits: word k of a patch holds bits 32 k .. of its own blocks' nibbles, then
// its shifted blocks'. In the float forms a pair across the torus seam takes
// the negated step, so its weight bit is flipped (fixed point swaps the
// roles instead).
static int ensure_patch_weights(cosm_handle *h)
{
    DevBuf<uint32_t> &buf = h->d_pwt[h->shape];
    if (buf.p) return COSM_OK;
    const int R = kPatchR[h->shape], C = kPatchC[h->shape], T = h->pgr * h->pgc, words = (8 * R * C + 31) / 32;
    const int BR = h->Q / h->Wd, BC = h->Wd;
    const bool flip = h->prm.storage != COSM_Q16;
    std::vector<uint32_t> wt((size_t)words * T, 0u);
    for (int pr = 0; pr < h->pgr; ++pr) {
        for (int pc = 0; pc < h->pgc; ++pc) {
            const int r0 = pr * R - std::max(0, pr - h->pfr), nr = pr < h->pfr ? R : R - 1;
            const int c0 = pc * C - std::max(0, pc - h->pfc), nc = pc < h->pfc ? C : C - 1;
            for (int i = 0; i < nr; ++i) {
                for (int j = 0; j < nc; ++j) {
                    const int f = (r0 + i) * h->Wd + c0 + j;
                    uint32_t odd = h->nib[(size_t)h->Q + f];
                    if (flip && c0 + j == BC - 1) odd ^= 3u;
                    if (flip && r0 + i == BR - 1) odd ^= 12u;
                    const int b0 = 4 * (i * C + j), b1 = 4 * (R * C + i * C + j);
                    const size_t t = (size_t)pr * h->pgc + pc;
                    wt[(size_t)(b0 / 32) * T + t] |= (uint32_t)h->nib[(size_t)f] << (b0 % 32);
                    wt[(size_t)(b1 / 32) * T + t] |= odd << (b1 % 32);
                }
            }
        }
    }
    int rc = buf.ensure(wt.size());
    if (rc) return rc;
    if (cudaMemcpy(buf.p, wt.data(), wt.size() * 4, cudaMemcpyHostToDevice) != cudaSuccess || settle()) {
        buf.release();
        return fail(COSM_ERR_CUDA, "copying the patch weights to the device failed");
    }
    return COSM_OK;
}

// Format of the record tables of an edge-list instance with tiles of K
// replicas, -1 where it takes the plain records: the simultaneous update,
// staged or split records (test hooks), thread counts that are not whole
// warps, and float weights of 64 and more, whose bits do not fit.
static int record_format(const cosm_handle *h, int K)
{
    const cosm_params &p = h->prm;
    if (h->mode != MODE_GENERAL_ || std::getenv("COSM_STAGE") || std::getenv("COSM_SPLIT_W") ||
        env_int("COSM_THREADS", 0) % 32)
        return -1;
    const int E = K * (p.storage == COSM_F32 ? 4 : 2);
    const bool each = p.storage == COSM_F32 && wrap_period(p.alpha0_deg, p.dwt_ratio, p.dwt_period, p.flags, h->mode,
                                                           p.storage, h->wbound) == 0;
    if (h->wmax == 1 && h->g.n <= (1 << 15) && !each) return EDGES_SIGN;
    const int more = each ? EDGES_EACH : 0;
    // one word (half the record traffic of a weighted graph) where it holds
    if (E >= 8 && h->g.n <= (1 << 14) && h->wmax <= (E == 8 ? 3 : 7)) return EDGES_PACK | more;
    if (p.storage != COSM_Q16 && h->wmax > 63) return -1;
    return EDGES_WEIGHT | more;
}

// Modelled SM cycles per sweep of a run of edge-list tiles of K replicas with T
// threads (record tables): what the CTAs that share an SM issue and move
// through shared memory, plus part of one CTA's latency per sweep (which more
// CTAs hide), times the waves of tiles. Fitted to random 3-regular graphs of
// 20,000 vertices, G(n, m) graphs of 2,000 and 10,000 and 3D lattices of 1,728
// and 21,952, 32 to 2,048 replicas: within 20 %, e.g. G(9973, 24931) with
// weights to 3 at two replicas per tile and 256 / 512 / 1,024 threads 22.3 /
// 24.1 / 33.7 us per sweep of 1,024 replicas, modelled 23.4 / 24.9 / 33.
static double edges_cost(const cosm_handle *h, int K, int format, int T, int occ, int replicas)
{
    const int st = h->prm.storage, W = T / 32, E = K * (st == COSM_F32 ? 4 : 2);
    const double words = K / 2.0, colours = h->C;
    // instructions and shared-memory wavefronts of a row of 32 edges (the
    // colours', the twist's and the wrap's are counted apart below)
    double inst = st == COSM_F32 ? 12.0 + 9.0 * std::max(1.0, words)
                                 : st == COSM_Q16 ? 14.0 + 6.5 * words : 12.0 + 19.0 * words;
    if ((format & ~EDGES_EACH) != EDGES_SIGN) inst += 2.0;
    if (format >= 0 && (format & EDGES_EACH)) inst += 6.0 * std::max(1.0, words);
    const double waves = (E == 4 ? 5.2 : E == 8 ? 9.0 : 17.8) + ((format & ~EDGES_EACH) == EDGES_WEIGHT ? 2.6 : 1.5);
    double rows = 0.0, steps = 0.0;  // rows of all colours, and of the busiest warp
    for (int c = 0; c < h->C; ++c) {
        const int r = (h->off[c + 1] - h->off[c] + 31) / 32;
        rows += r;
        steps += (r + W - 1) / W;
    }
    // the twist and the wrap after the colours, every second sweep or so, and a field pass
    const double slots = h->g.n / 32.0, passes = 0.5 + (h->fields ? 1.0 : 0.0);
    const double tiles = std::ceil((double)replicas / K), room = (double)occ * h->num_sms;
    const double r = std::max(1.0, std::ceil(std::min(tiles, room) / h->num_sms));
    const double rate = std::min(2.4, 0.15 * r * W);  // instructions per SM and cycle
    const double issue = (rows * inst + W * colours * 40.0 + slots * passes * (6.0 + 6.0 * std::max(1.0, words))) / rate;
    const double move = (rows * waves + slots * passes * E / 2.0) / 0.8;
    const double latency = colours * 250.0 + steps * (E >= 16 ? 70.0 : 110.0) + slots / W * passes * 60.0;
    return (r * std::max(issue, move) + 0.6 * latency / r) * std::max(1.0, tiles / room);
}

// Tile width and threads of an edge-list instance on record tables. False
// when no width and thread count take them.
static bool choose_edges(cosm_handle *h, int replicas, int forceK, int forceT, bool narrow_ties)
{
    const cosm_params &p = h->prm;
    const int Ts[8] = {64, 128, 192, 256, 384, 512, 768, 1024};
    double best = 1e300;
    for (int K = p.storage == COSM_F32 ? 1 : 2; K <= (p.storage == COSM_F32 ? 4 : 8); K *= 2) {
        if (forceK && K != forceK) continue;
        const int format = record_format(h, K);
        if (format < 0) return false;
        const size_t smem = sweep_smem_bytes(p.storage, K, h->g.n, p.n_bisectors, h->mode);
        for (int k = 0; k < (forceT ? 1 : 8); ++k) {
            const int T = forceT ? forceT : Ts[k];
            const int occ = edges_occupancy(p.storage, K, format, T, smem);
            if (occ < 1) continue;
            const double cost = edges_cost(h, K, format, T, occ, replicas) * tie_weight(narrow_ties, K);
            if (cost < best) {
                best = cost;
                h->K = K;
                h->threads = T;
                h->occupancy = occ;
                h->smem = smem;
                h->format = format;
            }
        }
    }
    return best < 1e300;
}

// Order of one colour's edges e0 .. e1 - 1 in the rows of a table. A phase
// access of 4, 8 or 16 bytes per lane takes one wavefront per 32, 16 or 8
// lanes when their slots are distinct modulo R = 128 / E, so the edges are
// dealt in groups of R with distinct source residues and, as far as they go
// round, distinct destination residues: each source residue gives an edge
// whose destination residue is still free, both rotated from group to group;
// places left over take the fullest cells. Edges of one colour share no
// vertex, so the order changes no result. Extra wavefronts of 7,500 random
// edges: 7 / 19 / 41 % for R = 8 / 16 / 32 (161 / 206 / 251 % unarranged), at
// 16 ns an edge.
static void arrange_rows(const uint32_t *ij, int e0, int e1, int R, std::vector<int32_t> &out)
{
    const int cnt = e1 - e0;
    out.resize((size_t)cnt);
    if (cnt <= R || std::getenv("COSM_SRC_ORDER")) {
        for (int k = 0; k < cnt; ++k) out[(size_t)k] = e0 + k;
        return;
    }
    std::vector<int32_t> head((size_t)R * R, -1), next((size_t)cnt);
    uint32_t mask[32] = {0};  // destination residues a source residue still has
    int rows[32] = {0}, cols[32] = {0};
    for (int k = cnt - 1; k >= 0; --k) {
        const int a = (int)(ij[e0 + k] & 0xFFFFu) % R, b = (int)(ij[e0 + k] >> 16) % R;
        next[(size_t)k] = head[(size_t)(a * R + b)];
        head[(size_t)(a * R + b)] = k;
        mask[a] |= 1u << b;
        ++rows[a];
        ++cols[b];
    }
    int done = 0;
    auto take = [&](int a, int b) {
        int32_t &hd = head[(size_t)(a * R + b)];
        out[(size_t)done++] = e0 + hd;
        hd = next[(size_t)hd];
        if (hd < 0) mask[a] &= ~(1u << b);
        --rows[a];
        --cols[b];
    };
    const uint32_t full = R == 32 ? 0xFFFFFFFFu : (1u << R) - 1;
    for (int g = 0; done < cnt; ++g) {
        uint32_t used = 0;
        const int stop = std::min(cnt, done + R);
        for (int i = 0; i < R && done < stop; ++i) {
            const int a = (i + g) % R, s = (a + g) % R;
            const uint32_t open = mask[a] & ~used;
            if (!open) continue;
            const uint32_t turned = ((open >> s) | (s ? open << (R - s) : 0u)) & full;
            const int b = (__builtin_ctz(turned) + s) % R;
            used |= 1u << b;
            take(a, b);
        }
        while (done < stop) {
            int a = 0, b = -1;
            for (int i = 1; i < R; ++i)
                if (rows[i] > rows[a]) a = i;
            for (uint32_t m = mask[a]; m; m &= m - 1) {
                const int q = __builtin_ctz(m);
                if (b < 0 || cols[q] > cols[b]) b = q;
            }
            take(a, b);
        }
    }
}

// Builds the record table of the current layout (cosm_edges.h).
static int ensure_records(cosm_handle *h)
{
    for (const auto &t : h->tables) {
        if (t->K == h->K && t->threads == h->threads && t->format == h->format) {
            h->table = t.get();
            return COSM_OK;
        }
    }
    if (h->threads < 32 || h->threads % 32) return fail(COSM_ERR_INVALID_ARG, "record tables need whole warps");
    const int fmt = h->format & ~EDGES_EACH, W = h->threads / 32, RW = fmt == EDGES_WEIGHT ? 2 : 1;
    const uint32_t E = (uint32_t)(h->K * (h->prm.storage == COSM_F32 ? 4 : 2));
    const bool q16 = h->prm.storage == COSM_Q16;
    int nc = 0;
    for (int c = 0; c < h->C; ++c) nc += h->off[c + 1] > h->off[c];  // an empty colour needs no barrier
    std::vector<uint32_t> counts((size_t)W * (nc + 1), 0u);
    std::vector<int32_t> starts((size_t)W + 1, 0), at((size_t)W);
    for (int c = 0, k = 0; c < h->C; ++c) {
        const int ec = h->off[c + 1] - h->off[c], rows = (ec + 31) / 32;
        if (!rows) continue;
        for (int w = 0; w < W; ++w) {
            const int mine = rows / W + (w < rows % W);
            counts[(size_t)w * (nc + 1) + k] = (uint32_t)mine | (ec % 32 && (rows - 1) % W == w ? kPartial : 0u);
            starts[(size_t)w + 1] += mine * 32 * RW;
        }
        ++k;
    }
    for (int w = 0; w < W; ++w) {
        counts[(size_t)w * (nc + 1) + nc] = counts[(size_t)w * (nc + 1)];
        starts[(size_t)w + 1] += starts[(size_t)w] + kRowsAhead * 32 * RW;
    }
    std::vector<uint32_t> rec((size_t)starts[(size_t)W], kNoEdge);
    std::copy(starts.begin(), starts.end() - 1, at.begin());
    std::vector<int32_t> order;
    for (int c = 0; c < h->C; ++c) {
        const int ec = h->off[c + 1] - h->off[c];
        arrange_rows(h->h_ij.data(), h->off[c], h->off[c + 1], (int)(128 / E), order);
        for (int k = 0; k < ec; ++k) {
            const int e = order[(size_t)k], lane = k % 32, w = k / 32 % W;
            uint32_t *r = rec.data() + at[(size_t)w] + lane * RW;
            const uint32_t si = h->h_ij[(size_t)e] & 0xFFFFu, sj = h->h_ij[(size_t)e] >> 16;
            const int wt = h->h_wv[(size_t)e];
            if (fmt == EDGES_SIGN) {
                r[0] = (wt < 0 ? 1u : 0u) | (si << 1) | (sj << 16);
            } else if (fmt == EDGES_PACK) {
                r[0] = (uint32_t)(wt + (int)E / 2) | si * E | (sj << 18);
            } else {
                uint32_t bits = (uint32_t)wt << 18;
                if (!q16) {
                    const float f = (float)wt;
                    std::memcpy(&bits, &f, 4);
                }
                r[0] = si * E;
                r[1] = sj * E | bits;
            }
            if (lane == 31 || k + 1 == ec) at[(size_t)w] += 32 * RW;
        }
    }
    for (int w = 0; w < W; ++w)
        std::copy_n(rec.begin() + starts[(size_t)w],
                    std::min(kRowsAhead * 32 * RW, at[(size_t)w] - starts[(size_t)w]), rec.begin() + at[(size_t)w]);
    std::unique_ptr<RecordTable> t(new RecordTable());
    h->tables.reserve(h->tables.size() + 1);
    t->K = h->K;
    t->threads = h->threads;
    t->format = h->format;
    t->n_colours = nc;
    int rc;
    if ((rc = t->rec.ensure(rec.size())) || (rc = t->counts.ensure(counts.size())) ||
        (rc = t->starts.ensure((size_t)W))) {
        t->release();
        return rc;
    }
    if (cudaMemcpy(t->rec.p, rec.data(), rec.size() * 4, cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemcpy(t->counts.p, counts.data(), counts.size() * 4, cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemcpy(t->starts.p, starts.data(), (size_t)W * 4, cudaMemcpyHostToDevice) != cudaSuccess || settle()) {
        t->release();
        return fail(COSM_ERR_CUDA, "copying the record table to the device failed");
    }
    h->table = t.get();
    h->tables.push_back(std::move(t));
    return COSM_OK;
}

int cosm::ensure_tables(cosm_handle *h)
{
    try {
        if (h->shape >= 0) return ensure_patch_weights(h);
        if (h->format >= 0) return ensure_records(h);
    } catch (const std::bad_alloc &) {
        return fail(COSM_ERR_NOMEM, "host allocation failed");
    }
    return COSM_OK;
}

// Replicas per CTA (K) and threads per CTA: maximise resident replicas per
// SM (COSM_K / COSM_THREADS override for experiments).
int cosm::choose_layout(cosm_handle *h, int replicas, bool narrow_ties, int only_K)
{
    const cosm_params &p = h->prm;
    const int mode = h->mode;
    const int P = p.n_bisectors;
    int max_ec = 0;
    for (int c = 0; c < h->C; ++c) max_ec = std::max(max_ec, h->off[c + 1] - h->off[c]);
    const int Ks_f32[3] = {1, 2, 4}, Ks_f16[3] = {2, 4, 8};
    const int *Ks = p.storage == COSM_F32 ? Ks_f32 : Ks_f16;
    int forceK = env_int("COSM_K", only_K), forceT = at_least_a_warp(env_int("COSM_THREADS", 0));
    int bestK = 0, bestT = 0, bestOcc = 0;
    // 2D lattices keep their phases in registers where a patch shape fits
    // (forced threads and the cross-check switches take the passes on shared
    // memory); else
    // binary32 lattice tiles of two replicas on an even number of block
    // columns take two adjacent 2x2 blocks per thread in the even pass
    // (COSM_SCALAR_F32 and COSM_SINGLE_BLOCKS keep the other passes
    // available as cross-checks)
    h->shape = -1;
    if (mode == MODE_LATTICE2D_ && !forceT && !std::getenv("COSM_SCALAR_F32") && !std::getenv("COSM_SINGLE_BLOCKS") &&
        choose_patch(h, replicas, forceK, narrow_ties)) {
        h->block_pairs = false;
        h->staged = false;
        const size_t esz = p.storage == COSM_F32 ? 4 : 2;
        h->tile_stride = (int64_t)(((size_t)h->g.n * h->K * esz + 15) / 16 * 16 / esz);
        h->format = -1;
        return COSM_OK;
    }
    if (mode == MODE_GENERAL_ && choose_edges(h, replicas, forceK, forceT, narrow_ties)) {
        h->block_pairs = false;
        h->staged = false;
        const size_t esz = p.storage == COSM_F32 ? 4 : 2;
        h->tile_stride = (int64_t)(((size_t)h->g.n * h->K * esz + 15) / 16 * 16 / esz);
        return COSM_OK;
    }
    h->format = -1;
    const bool pairs_ok = mode == MODE_LATTICE2D_ && p.storage == COSM_F32 && h->Wd % 2 == 0 &&
                          !std::getenv("COSM_SCALAR_F32") && !std::getenv("COSM_SINGLE_BLOCKS");
    long bestScore = -1;
    for (int k = 0; k < 3; ++k) {
        const int K = Ks[k];
        if (forceK && K != forceK) continue;
        const size_t smem = sweep_smem_bytes(p.storage, K, h->g.n, P, mode);
        if (smem > 227 * 1024) continue;
        // thread counts to try: edge-list kernels half a colour class's edges
        // (at most 512, or 1,024 for tiles of two or four replicas and for
        // fixed-point tiles of eight); lattice kernels the 2x2 blocks of a
        // sublattice, up to 512 or, for tiles of at most 4 replicas, 1024
        // threads
        int cand[2] = {0, 0};
        if (forceT) {
            cand[0] = forceT;
        } else if (mode == MODE_LATTICE2D_) {
            for (int c = 0; c < (K <= 4 ? 2 : 1); ++c) {
                int T = std::min(c ? 1024 : 512, std::max(64, (h->Q + 31) / 32 * 32));
                // a multiple of the block-row width fixes each thread's column
                if (h->Wd <= T && (T / h->Wd) * h->Wd >= T / 2) T = (T / h->Wd) * h->Wd;
                cand[c] = T;
            }
            if (cand[1] == cand[0]) cand[1] = 0;
        } else {
            cand[0] = std::min(512, std::max(64, ((max_ec + 1) / 2 + 31) / 32 * 32));
            // tiles of two or four replicas (and fixed-point tiles of eight)
            // may also take 1,024 threads
            if (mode == MODE_GENERAL_ && (K == 2 || K == 4 || p.storage == COSM_Q16))
                cand[1] = std::min(1024, std::max(64, ((max_ec + 1) / 2 + 31) / 32 * 32));
            if (cand[1] == cand[0]) cand[1] = 0;
        }
        for (int c = 0; c < 2 && cand[c]; ++c) {
            int T = cand[c];
            int occ = sweep_occupancy(p.storage, K, mode, T, smem);
            while (occ == 0 && T > 64 && !forceT) {
                T /= 2;
                occ = sweep_occupancy(p.storage, K, mode, T, smem);
            }
            if (occ == 0) continue;
            const long tiles = (replicas + K - 1) / K;
            // resident replicas per SM, capped by what the run can fill; on a
            // tie a larger tile amortises per-edge work when the run fills
            // every CTA slot, a smaller one spreads a small run over more
            // SMs; then more resident threads hide more latency
            const long resident = std::min<long>((long)occ * K, std::max<long>(1, tiles * K / h->num_sms));
            const bool full = tiles >= (long)occ * h->num_sms;
            const long score = resident * 100000 + ((full && !narrow_ties) ? K : -K) * 4096 + (long)occ * T;
            if (score > bestScore) {
                bestScore = score;
                bestK = K;
                bestT = T;
                bestOcc = occ;
            }
        }
    }
    if (!bestK) return fail(COSM_ERR_TOO_LARGE, "no replica tile fits in shared memory");
    h->K = bestK;
    h->threads = bestT;
    h->block_pairs = pairs_ok && bestK == 2;
    h->occupancy = bestOcc;
    h->smem = sweep_smem_bytes(p.storage, bestK, h->g.n, P, mode);
    // binary32 edge lists may stage each colour's records in shared memory
    // (two buffers after the tile) where that keeps the tile's occupancy.
    // Measured slower than the global loads in every case tried (the records
    // stay in L1 / L2, and the copies cost more than their latency), so it is
    // taken only when the environment variable COSM_STAGE is set.
    h->staged = false;
    if (mode == MODE_GENERAL_ && p.storage == COSM_F32 && h->C >= 1 && std::getenv("COSM_STAGE")) {
        const size_t sb = 2 * (size_t)(stage_ij_bytes(max_ec) + stage_w_bytes(max_ec));
        if (h->smem + sb <= 227 * 1024 && sweep_occupancy(p.storage, bestK, mode, bestT, h->smem + sb) >= bestOcc) {
            h->staged = true;
            h->smem += sb;
        }
    }
    const size_t esz = p.storage == COSM_F32 ? 4 : 2;
    h->tile_stride = (int64_t)(((size_t)h->g.n * bestK * esz + 15) / 16 * 16 / esz);
    return COSM_OK;
}

int cosm::ensure_run_buffers(cosm_handle *h, int replicas)
{
    const size_t esz = h->prm.storage == COSM_F32 ? 4 : 2;
    const int64_t tiles = (replicas + h->K - 1) / h->K;
    int rc;
    if ((rc = h->d_state.ensure((size_t)tiles * (size_t)h->tile_stride * esz)) ||
        (rc = h->d_cut.ensure((size_t)replicas)) || (rc = h->d_bestp.ensure((size_t)replicas)) ||
        (rc = h->d_energy.ensure((size_t)replicas)) || (rc = h->d_bisB.ensure((size_t)replicas)) ||
        (rc = h->d_ready.ensure((size_t)tiles)))
        return rc;
    if (h->prm.track_period > 0 &&
        (rc = h->d_bits.ensure((size_t)replicas * (size_t)((h->g.n + 31) / 32))))
        return rc;
    return COSM_OK;
}

size_t cosm::device_bytes(const cosm_handle *h)
{
    const auto sum = [](const auto &...b) { return (size_t(0) + ... + (b.cap * sizeof(*b.p))); };
    size_t bytes = sum(h->d_ij, h->d_w, h->d_orig, h->d_slot, h->d_off, h->d_wnib, h->d_h, h->d_hlist, h->d_state, h->d_cut,
                       h->d_bestp, h->d_alpha, h->d_segs, h->d_segoff, h->d_ready, h->d_err, h->d_best, h->d_spins,
                       h->d_energy, h->d_bisB, h->d_trace, h->d_bits, h->d_qbuf, h->d_delta, h->d_items, h->d_stage);
    for (const auto &b : h->d_pwt) bytes += sum(b);
    for (const auto &t : h->tables) bytes += sum(t->rec, t->counts, t->starts);
    return bytes;
}

int32_t cosm::wrap_period(double alpha0_deg, double dwt_ratio, int dwt_period, int flags, int mode, int storage,
                          int64_t wbound)
{
    if (storage != COSM_F32 || (mode != MODE_LATTICE2D_ && mode != MODE_GENERAL_)) return 1;
    const double a0 = std::fabs(alpha0_deg) / 360.0;
    const bool dwt = !(flags & COSM_NO_DWT) && dwt_period > 0;
    const bool lattice = mode == MODE_LATTICE2D_;
    const double limit = lattice ? 0.999 : 1.999;
    int32_t best = lattice ? 1 : 0, best_dwt = 0;
    for (int P = 1; P <= (lattice ? 4 : 12); ++P) {
        const double twists = dwt ? std::ceil((double)P / dwt_period) : 0.0;
        if (0.5 + (double)wbound * P * a0 + twists * std::fabs(dwt_ratio) * a0 >= limit) break;
        best = P;
        if (dwt && P % dwt_period == 0) best_dwt = P;
    }
    // edge lists wrap in the twist's pass: a multiple of the twist period
    // needs no pass of its own
    return (!lattice && best_dwt) ? best_dwt : best;
}

int64_t cosm::vertex_weight_bound(int32_t n, int64_t m, const int32_t *src, const int32_t *dst, const int32_t *w,
                                  const int32_t *h)
{
    std::vector<int64_t> sum((size_t)n, 0);
    for (int64_t e = 0; e < m; ++e) {
        const int64_t a = std::abs((int64_t)w[e]);
        sum[(size_t)src[e]] += a;
        sum[(size_t)dst[e]] += a;
    }
    int64_t b = 0;
    for (int32_t v = 0; v < n; ++v) b = std::max(b, sum[(size_t)v] + (h ? std::abs((int64_t)h[v]) : 0));
    return b;
}

int64_t cosm::colour_weight_bound(const int32_t *off, int C, const int8_t *w, const int32_t *h, int32_t n)
{
    int64_t b = 0;
    for (int c = 0; c < C; ++c) {
        int32_t mx = 0;
        for (int32_t k = off[c]; k < off[c + 1]; ++k) mx = std::max(mx, (int32_t)std::abs((int32_t)w[k]));
        b += mx;
    }
    int32_t mh = 0;
    if (h)
        for (int32_t v = 0; v < n; ++v) mh = std::max(mh, std::abs(h[v]));
    return b + mh;
}

InstView cosm::inst_view(cosm_handle *h)
{
    InstView v;
    std::memset(&v, 0, sizeof(v));
    v.n = h->g.n;
    v.C = h->C;
    v.off = h->d_off.p;
    v.ij = h->d_ij.p;
    v.w = h->d_w.p;
    v.orig_of = h->d_orig.p;
    v.slot_of = h->d_slot.p;
    v.wnib = h->d_wnib.p;
    v.Q = h->Q;
    v.Wd = h->Wd;
    if (h->format >= 0 && h->table) {
        v.rec = h->table->rec.p;
        v.counts = h->table->counts.p;
        v.starts = h->table->starts.p;
        v.n_colours = h->table->n_colours;
    }
    if (h->shape >= 0) {
        v.pwt = h->d_pwt[h->shape].p;
        v.pgr = h->pgr;
        v.pgc = h->pgc;
        v.pfr = h->pfr;
        v.pfc = h->pfc;
    }
    v.seed = h->seed;
    v.replicas = h->replicas;
    v.dwt_period = (h->prm.flags & COSM_NO_DWT) ? 0 : h->prm.dwt_period;
    v.window = (float)(h->prm.window_deg / 360.0);
    v.flags = h->prm.flags;
    v.P = h->prm.n_bisectors;
    v.mode = h->mode;
    v.K = h->K;
    v.qwin = (uint32_t)std::min(2147483648.0, std::floor(h->prm.window_deg / 360.0 * 4294967296.0 + 0.5));
    v.state = h->d_state.p;
    v.state_tile_stride = h->tile_stride;
    v.cut = h->d_cut.p;
    v.bestp = h->d_bestp.p;
    v.hv = h->fields ? h->d_h.p : nullptr;
    v.hlist = h->d_hlist.p;
    v.n_fields = h->n_fields;
    v.W = h->W;
    v.energy = h->d_energy.p;
    v.bisB = h->d_bisB.p;
    v.words = (h->g.n + 31) / 32;
    // the scalar lattice passes (binary32 and 16-bit storage) stay available
    // as a cross-check
    v.paired = std::getenv("COSM_SCALAR_F32") ? 0 : (h->block_pairs ? 2 : 1);
    v.wrap_p = wrap_period(h->prm.alpha0_deg, h->prm.dwt_ratio, h->prm.dwt_period, h->prm.flags, h->mode,
                           h->prm.storage, h->wbound);
    v.check = h->d_err.p;
    if (h->staged) {
        int max_ec = 0;
        for (int c = 0; c < h->C; ++c) max_ec = std::max(max_ec, h->off[c + 1] - h->off[c]);
        v.stage_ij = stage_ij_bytes(max_ec);
        v.stage_w = stage_w_bytes(max_ec);
    }
    return v;
}

static KernelArgs base_args(cosm_handle *h)
{
    KernelArgs a;
    std::memset(&a, 0, sizeof(a));
    a.v = inst_view(h);
    a.ready = h->d_ready.p;
    a.err = h->d_err.p;
    a.wait_limit_ns = h->wait_limit_ns ? h->wait_limit_ns
                                       : (uint64_t)env_int("COSM_WAIT_LIMIT_S", 20) * 1000000000ull;
    return a;
}

static int upload_segments(cosm_handle *h, cudaStream_t st)
{
    if (h->segs_uploaded) return COSM_OK;
    int rc;
    if ((rc = h->d_segs.ensure(h->h_segs.size())) || (rc = h->d_segoff.ensure(h->h_segoff.size())))
        return rc;
    CK(cudaMemcpyAsync(h->d_segs.p, h->h_segs.data(), h->h_segs.size() * sizeof(Segment),
                       cudaMemcpyHostToDevice, st));
    CK(cudaMemcpyAsync(h->d_segoff.p, h->h_segoff.data(), h->h_segoff.size() * 4,
                       cudaMemcpyHostToDevice, st));
    h->segs_uploaded = true;
    return COSM_OK;
}

// Work schedule for sweeps s0..s1 of an S-sweep trial (L = s1 - s0 + 1
// sweeps) of `tiles` tiles on at most G resident CTAs. With tiles <= G every
// CTA runs one tile's whole range. Otherwise the wrap-around rule of
// McNaughton (1959) gives every CTA an equal share of tiles * L sweeps: a
// tile split between CTA b and b+1 runs its head first on b and its tail
// last on b+1 (the share exceeds L, so the two never overlap), and b+1 waits
// for the head's published state before the tail. A range that starts at
// sweep 1 draws the initial phases, a later one loads the stored state; the
// range that ends at sweep S reads out; every range stores its state.
static void build_schedule(cosm_handle *h, int64_t tiles, int64_t s0, int64_t s1, int64_t S, int64_t G)
{
    if (h->sched_tiles == tiles && h->sched_S == S && h->sched_G == G && h->sched_s0 == s0 && h->sched_s1 == s1)
        return;
    h->h_segs.clear();
    h->h_segoff.assign(1, 0);
    h->segs_uploaded = false;
    const int64_t L = s1 - s0 + 1;
    const int32_t first = s0 == 1 ? SEG_INIT : SEG_LOAD;
    const int32_t last = SEG_STORE | (s1 == S ? SEG_READOUT : 0);
    if (tiles <= G) {
        for (int64_t t = 0; t < tiles; ++t) {
            h->h_segs.push_back(Segment{(int32_t)t, first | last, s0, s1});
            h->h_segoff.push_back((int32_t)h->h_segs.size());
        }
    } else {
        const __int128 TL = (__int128)tiles * L;
        for (int64_t b = 0; b < G; ++b) {
            const int64_t lo = (int64_t)(TL * b / G), hi = (int64_t)(TL * (b + 1) / G);
            std::vector<Segment> pieces;
            for (int64_t j = lo / L; j <= (hi - 1) / L && j < tiles; ++j) {
                const int64_t a0 = std::max<int64_t>(lo, j * L) - j * L;
                const int64_t z = std::min<int64_t>(hi, (j + 1) * L) - j * L;
                if (z <= a0) continue;
                Segment sg{(int32_t)j, 0, s0 + a0, s0 + z - 1};
                sg.flags = (a0 == 0) ? first : (SEG_LOAD | SEG_WAIT);
                sg.flags |= (z == L) ? last : (SEG_STORE | SEG_SIGNAL);
                pieces.push_back(sg);
            }
            // execution order: head of the tile continuing on b+1 first, the
            // tail of the tile started on b-1 last
            std::vector<Segment> ordered;
            if (!pieces.empty() && pieces.back().s_begin == s0 && pieces.back().s_end < s1) {
                ordered.push_back(pieces.back());
                pieces.pop_back();
            }
            Segment tail{};
            bool has_tail = false;
            if (!pieces.empty() && pieces.front().s_begin > s0) {
                tail = pieces.front();
                has_tail = true;
                pieces.erase(pieces.begin());
            }
            for (auto &sg : pieces) ordered.push_back(sg);
            if (has_tail) ordered.push_back(tail);
            for (auto &sg : ordered) h->h_segs.push_back(sg);
            h->h_segoff.push_back((int32_t)h->h_segs.size());
        }
    }
    h->sched_tiles = tiles;
    h->sched_S = S;
    h->sched_G = G;
    h->sched_s0 = s0;
    h->sched_s1 = s1;
}

int cosm::upload_alpha(cosm_handle *h, int64_t S, cudaStream_t st)
{
    const double a0 = h->prm.alpha0_deg / 360.0, ratio = h->prm.dwt_ratio;
    if (h->alpha_S == S && h->alpha_a0 == a0 && h->alpha_ratio == ratio) return COSM_OK;
    std::vector<float2> tab((size_t)S);
    const bool q16 = h->prm.storage == COSM_Q16;
    for (int64_t s = 1; s <= S; ++s) {
        // linear ramp alpha_0 -> 0 (Table IX), FP64 rounded once to FP32, or
        // for fixed-point phases rounded to the nearest 2^-16-turn quantum
        const double a = (S <= 1) ? a0 : a0 * (double)(S - s) / (double)(S - 1);
        tab[(size_t)(s - 1)] = q16 ? make_float2((float)std::floor(a * 65536.0 + 0.5),
                                                 (float)std::floor(ratio * a * 65536.0 + 0.5))
                                   : make_float2((float)a, (float)(ratio * a));
    }
    int rc = h->d_alpha.ensure((size_t)S);
    if (rc) return rc;
    CK(cudaMemcpyAsync(h->d_alpha.p, tab.data(), tab.size() * sizeof(float2), cudaMemcpyHostToDevice, st));
    CK(cudaStreamSynchronize(st));  // the host table is released here
    h->alpha_S = S;
    h->alpha_a0 = a0;
    h->alpha_ratio = ratio;
    return COSM_OK;
}

// Optimal-bisector readout of every replica from the stored state, one CTA
// of 1024 threads per replica at a time, one CTA per SM.
int cosm::launch_opt_readout(cosm_handle *h, bool keep_better, cudaStream_t st)
{
    const int n = h->g.n;
    const int grid = std::max(1, std::min(h->replicas, h->num_sms));
    int rc;
    if ((rc = h->d_qbuf.ensure((size_t)grid * n)) || (rc = h->d_delta.ensure((size_t)grid * n)) ||
        (rc = h->d_items.ensure((size_t)grid * 2 * n)))
        return rc;
    OptArgs o;
    std::memset(&o, 0, sizeof(o));
    o.v = inst_view(h);
    if (keep_better && h->prm.track_period > 0) o.v.bits = h->d_bits.p;
    o.qbuf = h->d_qbuf.p;
    o.delta = h->d_delta.p;
    o.items = h->d_items.p;
    o.keep_better = keep_better ? 1 : 0;
    o.storage = h->prm.storage;
    if (opt_readout_launch(o, grid, st))
        return fail(COSM_ERR_CUDA, std::string("optimal-bisector launch: ") + cudaGetErrorString(cudaGetLastError()));
    return COSM_OK;
}

int cosm::launch_finalize(cosm_handle *h, cudaStream_t st)
{
    FinalArgs f;
    f.n = h->g.n;
    f.replicas = h->replicas;
    f.K = h->K;
    f.storage = h->prm.storage;
    f.P = h->prm.n_bisectors;
    f.W = h->W;
    f.state = h->d_state.p;
    f.state_tile_stride = h->tile_stride;
    f.orig_of = h->d_orig.p;
    f.cut = h->d_cut.p;
    f.bestp = h->d_bestp.p;
    f.energy = h->d_energy.p;
    f.bisB = h->d_bisB.p;
    f.bits = h->bits_valid ? h->d_bits.p : nullptr;
    f.words = (h->g.n + 31) / 32;
    f.best = h->d_best.p;
    f.spins = h->d_spins.p;
    f.target = h->target;
    if (finalize_launch(f, st)) return fail(COSM_ERR_CUDA, std::string("finalize launch: ") +
                                                          cudaGetErrorString(cudaGetLastError()));
    return COSM_OK;
}

// The layout, tables and buffers of `replicas` replicas. Where no layout fits
// or its tables cannot be built the handle keeps the layout it had, with the
// state and results that are stored in it; a new layout ends them.
static int prepare_replicas(cosm_handle *h, int32_t replicas)
{
    const auto forget = [h] { h->have_state = h->have_result = h->have_trace = h->bits_valid = false; };
    int rc;
    if (!h->K || replicas != h->replicas) {
        const TileLayout before = *h;
        if ((rc = choose_layout(h, replicas)) || (rc = ensure_tables(h))) {
            static_cast<TileLayout &>(*h) = before;
            return rc;
        }
        h->replicas = replicas;
        forget();
    }
    if ((rc = ensure_run_buffers(h, replicas))) forget();
    return rc;
}

// Sweeps s0..s1 of an S-sweep trial of every replica (cosm_run: 1..S).
static int run_range(cosm_handle *h, int64_t sweeps, int64_t s0, int64_t s1, int32_t replicas, uint64_t seed,
                     int64_t target_cut, cudaStream_t st)
{
    NvtxRange range("cosm_run");
    if (!h) return fail(COSM_ERR_INVALID_ARG, "NULL handle");
    if (sweeps < 1 || sweeps >= ((int64_t)1 << 31)) return fail(COSM_ERR_INVALID_ARG, "sweeps must be in [1, 2^31)");
    if (replicas < 1 || replicas >= (1 << 24)) return fail(COSM_ERR_INVALID_ARG, "replicas must be in [1, 2^24)");
    if (s0 < 1 || s1 < s0 || s1 > sweeps) return fail(COSM_ERR_INVALID_ARG, "need 1 <= s_from <= s_to <= sweeps");
    int rc;
    if (s0 > 1) {
        // a continued trial keeps its replicas, seed and layout
        if (!h->have_state || h->sweep_idx != s0 - 1)
            return fail(COSM_ERR_STATE, "the state is at sweep " + std::to_string(h->sweep_idx) +
                                            ", not " + std::to_string(s0 - 1));
        if (replicas != h->replicas || seed != h->seed)
            return fail(COSM_ERR_INVALID_ARG, "a continued trial keeps its replica count and seed");
        if (h->stream && h->stream != st) CK(cudaStreamSynchronize(h->stream));
    }
    if ((rc = prepare_replicas(h, replicas))) return rc;
    h->seed = seed;
    h->target = target_cut;
    if ((rc = upload_alpha(h, sweeps, st))) return rc;
    const int64_t tiles = (replicas + h->K - 1) / h->K;
    int64_t cap = (int64_t)h->occupancy * h->num_sms;
    const int cap_env = env_int("COSM_GRID_CAP", 0);  // test hook: fewer resident CTAs
    if (cap_env > 0) cap = std::min<int64_t>(cap, cap_env);
    build_schedule(h, tiles, s0, s1, sweeps, cap);
    if (h->fault == COSM_FAULT_DROP_SIGNAL) {
        // injected fault: the heads of split tiles do not publish their state,
        // so the tails' bounded waits give up (COSM_ERR_TIMEOUT at cosm_sync)
        for (Segment &sg : h->h_segs) sg.flags &= ~SEG_SIGNAL;
        h->segs_uploaded = false;
        rc = upload_segments(h, st);
        h->sched_tiles = -1;  // the next run rebuilds the true schedule
        h->fault = 0;
        if (rc) return rc;
    } else if ((rc = upload_segments(h, st))) {
        return rc;
    }
    const bool waits = tiles > cap;
    if (waits) CK(cudaMemsetAsync(h->d_ready.p, 0, (size_t)tiles * 4, st));
    CK(cudaMemsetAsync(h->d_err.p, 0, 4, st));
    const int track = h->prm.track_period;
    const int32_t n_trace = track > 0 ? (int32_t)((sweeps + track - 1) / track) : 0;
    if (track > 0 && (rc = h->d_trace.ensure((size_t)replicas * (size_t)n_trace))) return rc;
    KernelArgs a = base_args(h);
    a.v.alpha_tab = h->d_alpha.p;
    a.v.alpha_base = 1;
    a.v.S = sweeps;
    if (track > 0) {
        a.v.track = track;
        a.v.n_trace = n_trace;
        a.v.trace = h->d_trace.p;
        a.v.bits = h->d_bits.p;
    }
    a.segs = h->d_segs.p;
    a.seg_off = h->d_segoff.p;
    LaunchCfg cfg{h->mode, h->prm.storage, h->K, h->threads, (int)(h->h_segoff.size() - 1), h->smem, waits,
                  h->shape, h->ragged, h->format};
    h->grid = cfg.grid;
    if (kernel_launch(cfg, a, st))
        return fail(COSM_ERR_CUDA, std::string("sweep launch: ") + cudaGetErrorString(cudaGetLastError()));
    h->launches = 1;
    h->stream = st;
    h->have_state = true;
    h->sweep_idx = s1;
    if (s1 < sweeps) {
        // mid-trial: no readout yet
        h->have_result = false;
        h->have_trace = false;
        h->bits_valid = false;
        return COSM_OK;
    }
    h->launches = 2;
    if (h->prm.flags & COSM_OPT_BISECTOR) {
        if ((rc = launch_opt_readout(h, track > 0, st))) return rc;
        h->launches = 3;
    }
    h->bits_valid = track > 0;
    h->n_trace = n_trace;
    h->have_trace = track > 0;
    if ((rc = launch_finalize(h, st))) return rc;
    h->have_result = true;
    return COSM_OK;
}

extern "C" int cosm_run(cosm_handle *h, int64_t sweeps, int32_t replicas, uint64_t seed, int64_t target_cut,
                        void *stream)
{
    return run_range(h, sweeps, 1, sweeps, replicas, seed, target_cut, reinterpret_cast<cudaStream_t>(stream));
}

extern "C" int cosm_run_range(cosm_handle *h, int64_t sweeps, int64_t s_from, int64_t s_to, int32_t replicas,
                              uint64_t seed, int64_t target_cut, void *stream)
{
    return run_range(h, sweeps, s_from, s_to, replicas, seed, target_cut, reinterpret_cast<cudaStream_t>(stream));
}

extern "C" int cosm_get_success(cosm_handle *h, int64_t *count)
{
    if (!h || !count) return fail(COSM_ERR_INVALID_ARG, "NULL argument");
    if (!h->have_result) return fail(COSM_ERR_STATE, "no run or readout yet");
    int rc = cosm_sync(h);
    if (rc) return rc;
    CK(cudaMemcpy(count, h->d_best.p + 3, 8, cudaMemcpyDeviceToHost));
    return COSM_OK;
}

extern "C" int cosm_set_wait_limit(cosm_handle *h, double seconds)
{
    if (!h || !(seconds > 0.0) || seconds > 3600.0)
        return fail(COSM_ERR_INVALID_ARG, "the wait limit must be in (0, 3600] seconds");
    h->wait_limit_ns = (uint64_t)(seconds * 1e9);
    return COSM_OK;
}

extern "C" int cosm_inject_fault(cosm_handle *h, int32_t kind)
{
    if (!h || (kind != 0 && kind != COSM_FAULT_DROP_SIGNAL)) return fail(COSM_ERR_INVALID_ARG, "unknown fault");
    h->fault = kind;
    return COSM_OK;
}

extern "C" int cosm_sync(cosm_handle *h)
{
    if (!h) return fail(COSM_ERR_INVALID_ARG, "NULL handle");
    CK(cudaStreamSynchronize(h->stream));
    int err = 0;
    CK(cudaMemcpy(&err, h->d_err.p, 4, cudaMemcpyDeviceToHost));
    if (err & 2) return fail(COSM_ERR_CHECK, "a device-side index check of the checked build failed");
    if (err) return fail(COSM_ERR_TIMEOUT, "a bounded wait between work segments gave up");
    return COSM_OK;
}

extern "C" int cosm_get_best(cosm_handle *h, int64_t *cut, int64_t *energy, int32_t *replica, int8_t *spins)
{
    if (!h) return fail(COSM_ERR_INVALID_ARG, "NULL handle");
    if (!h->have_result) return fail(COSM_ERR_STATE, "no run or readout yet");
    int rc = cosm_sync(h);
    if (rc) return rc;
    int64_t best[3];
    CK(cudaMemcpy(best, h->d_best.p, sizeof(best), cudaMemcpyDeviceToHost));
    if (cut) *cut = best[0];
    if (energy) *energy = best[1];
    if (replica) *replica = (int32_t)best[2];
    if (spins) CK(cudaMemcpy(spins, h->d_spins.p, (size_t)h->g.n, cudaMemcpyDefault));
    return COSM_OK;
}

extern "C" int cosm_get_replica_energies(cosm_handle *h, int64_t *energies)
{
    if (!h || !energies) return fail(COSM_ERR_INVALID_ARG, "NULL argument");
    if (!h->have_result) return fail(COSM_ERR_STATE, "no run or readout yet");
    int rc = cosm_sync(h);
    if (rc) return rc;
    CK(cudaMemcpy(energies, h->d_energy.p, (size_t)h->replicas * 8, cudaMemcpyDefault));
    return COSM_OK;
}

extern "C" int cosm_get_replica_bisectors(cosm_handle *h, uint32_t *B)
{
    if (!h || !B) return fail(COSM_ERR_INVALID_ARG, "NULL argument");
    if (!h->have_result) return fail(COSM_ERR_STATE, "no run or readout yet");
    int rc = cosm_sync(h);
    if (rc) return rc;
    CK(cudaMemcpy(B, h->d_bisB.p, (size_t)h->replicas * 4, cudaMemcpyDefault));
    return COSM_OK;
}

extern "C" int cosm_get_trace(cosm_handle *h, int64_t *trace, int64_t count)
{
    if (!h || !trace) return fail(COSM_ERR_INVALID_ARG, "NULL argument");
    if (!h->have_trace) return fail(COSM_ERR_STATE, "the last run had no tracking");
    if (count != (int64_t)h->replicas * h->n_trace)
        return fail(COSM_ERR_INVALID_ARG, "count must be replicas x ceil(sweeps / track_period) = " +
                                              std::to_string((int64_t)h->replicas * h->n_trace));
    int rc = cosm_sync(h);
    if (rc) return rc;
    CK(cudaMemcpy(trace, h->d_trace.p, (size_t)count * 8, cudaMemcpyDefault));
    return COSM_OK;
}

extern "C" int cosm_get_replica_cuts(cosm_handle *h, int64_t *cuts, int32_t *best_p)
{
    if (!h) return fail(COSM_ERR_INVALID_ARG, "NULL handle");
    if (!h->have_result) return fail(COSM_ERR_STATE, "no run or readout yet");
    int rc = cosm_sync(h);
    if (rc) return rc;
    if (cuts) CK(cudaMemcpy(cuts, h->d_cut.p, (size_t)h->replicas * 8, cudaMemcpyDefault));
    if (best_p) CK(cudaMemcpy(best_p, h->d_bestp.p, (size_t)h->replicas * 4, cudaMemcpyDefault));
    return COSM_OK;
}

// Moves the state between the device's tile layout and rows [replica][vertex]
// of the caller (host or device), a few tiles at a time through a staging
// buffer of at most 64 MB: kind >= 0 exports (StateKind), -1 imports.
static int state_rows(cosm_handle *h, int kind, void *rows)
{
    const size_t esz = kind == STATE_TURNS ? 8 : (h->prm.storage == COSM_F32 ? 4 : 2);
    const size_t row = (size_t)h->g.n * esz;
    const int64_t tiles = (h->replicas + h->K - 1) / h->K;
    int64_t step = std::max<int64_t>(1, std::min<int64_t>(tiles, (int64_t)(((size_t)64 << 20) / (row * h->K))));
    int rc;
    while ((rc = h->d_stage.ensure((size_t)step * h->K * row)) && step > 1) step = (step + 1) / 2;
    if (rc) return rc;
    for (int64_t t0 = 0; t0 < tiles; t0 += step) {
        const int64_t r0 = t0 * h->K, r1 = std::min<int64_t>(h->replicas, (t0 + step) * h->K);
        unsigned char *part = static_cast<unsigned char *>(rows) + (size_t)r0 * row;
        StateArgs a{h->d_state.p, h->tile_stride, h->d_orig.p, h->d_stage.p, h->prm.storage, h->K, h->g.n,
                    h->replicas, (int32_t)t0, (int32_t)std::min<int64_t>(step, tiles - t0)};
        if (kind < 0) CK(cudaMemcpy(h->d_stage.p, part, (size_t)(r1 - r0) * row, cudaMemcpyDefault));
        if (kind < 0 ? state_import_launch(a, nullptr) : state_export_launch(a, kind, nullptr))
            return fail(COSM_ERR_CUDA, std::string("state launch: ") + cudaGetErrorString(cudaGetLastError()));
        if (kind >= 0) CK(cudaMemcpy(part, h->d_stage.p, (size_t)(r1 - r0) * row, cudaMemcpyDefault));
    }
    return settle();
}

extern "C" int cosm_get_state(cosm_handle *h, double *phases)
{
    if (!h || !phases) return fail(COSM_ERR_INVALID_ARG, "NULL argument");
    if (!h->have_state) return fail(COSM_ERR_STATE, "no state yet");
    int rc = cosm_sync(h);
    if (rc) return rc;
    return state_rows(h, STATE_TURNS, phases);
}

extern "C" int cosm_set_state(cosm_handle *h, const double *phases, int32_t replicas, uint64_t seed)
{
    if (!h || !phases) return fail(COSM_ERR_INVALID_ARG, "NULL argument");
    if (replicas < 1 || replicas >= (1 << 24)) return fail(COSM_ERR_INVALID_ARG, "bad replica count");
    int rc;
    if (h->stream) CK(cudaStreamSynchronize(h->stream));
    std::vector<double> in((size_t)replicas * h->g.n);
    CK(cudaMemcpy(in.data(), phases, in.size() * 8, cudaMemcpyDefault));
    for (double x : in)
        if (!(x >= 0.0 && x < 1.0)) return fail(COSM_ERR_INVALID_ARG, "phases must be in [0, 1)");
    if ((rc = prepare_replicas(h, replicas))) return rc;
    h->seed = seed;
    const int64_t tiles = (replicas + h->K - 1) / h->K;
    const size_t esz = h->prm.storage == COSM_F32 ? 4 : 2;
    std::vector<unsigned char> raw((size_t)tiles * (size_t)h->tile_stride * esz, 0);
    for (int32_t r = 0; r < replicas; ++r) {
        const size_t base = (size_t)(r / h->K) * (size_t)h->tile_stride;
        for (int32_t v = 0; v < h->g.n; ++v) {
            const double x = in[(size_t)r * h->g.n + v] + 0.0;  // -0 becomes +0
            const double g = x >= 0.5 ? x - 1.0 : x;
            const size_t idx = base + (size_t)h->slot_of[(size_t)v] * h->K + (size_t)(r % h->K);
            if (esz == 4) {
                const float f = (float)g;
                std::memcpy(raw.data() + idx * 4, &f, 4);
            } else if (h->prm.storage == COSM_BF16) {
                const __nv_bfloat16 bv = __float2bfloat16_rn((float)g);
                std::memcpy(raw.data() + idx * 2, &bv, 2);
            } else if (h->prm.storage == COSM_F16) {
                const __half hv = __float2half_rn((float)g);
                std::memcpy(raw.data() + idx * 2, &hv, 2);
            } else {
                const uint16_t q = (uint16_t)((uint32_t)std::floor(x * 65536.0 + 0.5) & 0xFFFFu);
                std::memcpy(raw.data() + idx * 2, &q, 2);
            }
        }
    }
    CK(cudaMemcpy(h->d_state.p, raw.data(), raw.size(), cudaMemcpyHostToDevice));
    if ((rc = settle())) return rc;
    h->have_state = true;
    h->sweep_idx = 0;
    h->have_result = false;
    h->have_trace = false;
    h->bits_valid = false;
    return COSM_OK;
}

extern "C" int cosm_export_state(cosm_handle *h, void *phases, int32_t storage, int64_t *sweep_idx)
{
    if (!h || !phases) return fail(COSM_ERR_INVALID_ARG, "NULL argument");
    if (storage != h->prm.storage) return fail(COSM_ERR_INVALID_ARG, "storage differs from the handle's");
    if (!h->have_state) return fail(COSM_ERR_STATE, "no state yet");
    int rc = cosm_sync(h);
    if (rc) return rc;
    if ((rc = state_rows(h, STATE_RAW, phases))) return rc;
    if (sweep_idx) *sweep_idx = h->sweep_idx;
    return COSM_OK;
}

extern "C" int cosm_import_state(cosm_handle *h, const void *phases, int32_t storage, int32_t replicas,
                                 uint64_t seed, int64_t sweep_idx)
{
    if (!h || !phases) return fail(COSM_ERR_INVALID_ARG, "NULL argument");
    if (storage != h->prm.storage) return fail(COSM_ERR_INVALID_ARG, "storage differs from the handle's");
    if (replicas < 1 || replicas >= (1 << 24)) return fail(COSM_ERR_INVALID_ARG, "bad replica count");
    if (sweep_idx < 0 || sweep_idx >= ((int64_t)1 << 31)) return fail(COSM_ERR_INVALID_ARG, "bad sweep index");
    int rc;
    if (h->stream) CK(cudaStreamSynchronize(h->stream));
    if ((rc = prepare_replicas(h, replicas))) return rc;
    h->seed = seed;
    if ((rc = state_rows(h, -1, const_cast<void *>(phases)))) return rc;
    h->have_state = true;
    h->sweep_idx = sweep_idx;
    h->have_result = false;
    h->have_trace = false;
    h->bits_valid = false;
    return COSM_OK;
}

// One launch over all tiles of the current state with per-tile segments of
// the given flags and sweep range.
static int launch_on_state(cosm_handle *h, int32_t flags, int64_t s0, int64_t s1, const float2 *tab,
                           int64_t base, cudaStream_t st)
{
    const int64_t tiles = (h->replicas + h->K - 1) / h->K;
    h->h_segs.clear();
    h->h_segoff.assign(1, 0);
    for (int64_t t = 0; t < tiles; ++t) {
        h->h_segs.push_back(Segment{(int32_t)t, flags, s0, s1});
        h->h_segoff.push_back((int32_t)h->h_segs.size());
    }
    h->sched_tiles = -1;  // invalidate the cached run schedule
    h->segs_uploaded = false;
    int rc = upload_segments(h, st);
    if (rc) return rc;
    CK(cudaMemsetAsync(h->d_err.p, 0, 4, st));
    KernelArgs a = base_args(h);
    a.v.alpha_tab = tab;
    a.v.alpha_base = base;
    a.v.S = s1;
    a.segs = h->d_segs.p;
    a.seg_off = h->d_segoff.p;
    LaunchCfg cfg{h->mode, h->prm.storage, h->K, h->threads, (int)tiles, h->smem, false, h->shape, h->ragged, h->format};
    h->grid = cfg.grid;
    if (kernel_launch(cfg, a, st))
        return fail(COSM_ERR_CUDA, std::string("sweep launch: ") + cudaGetErrorString(cudaGetLastError()));
    h->stream = st;
    return COSM_OK;
}

extern "C" int cosm_step(cosm_handle *h, int64_t sweep, float alpha, void *stream)
{
    NvtxRange range("cosm_step");
    if (!h) return fail(COSM_ERR_INVALID_ARG, "NULL handle");
    if (!h->have_state) return fail(COSM_ERR_STATE, "no state yet");
    if (sweep < 1 || sweep >= ((int64_t)1 << 31)) return fail(COSM_ERR_INVALID_ARG, "bad sweep index");
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    int rc;
    DevBuf<float2> tab;  // one-entry step table for this sweep
    if ((rc = tab.ensure(1))) return rc;
    const float2 v = h->prm.storage == COSM_Q16
                         ? make_float2((float)std::floor((double)alpha * 65536.0 + 0.5),
                                       (float)std::floor(h->prm.dwt_ratio * (double)alpha * 65536.0 + 0.5))
                         : make_float2(alpha, (float)(h->prm.dwt_ratio * (double)alpha));
    if (h->stream) CK(cudaStreamSynchronize(h->stream));
    if (cudaMemcpyAsync(tab.p, &v, sizeof(v), cudaMemcpyHostToDevice, st) != cudaSuccess) {
        tab.release();
        return fail(COSM_ERR_CUDA, "alpha upload failed");
    }
    rc = launch_on_state(h, SEG_LOAD | SEG_STORE, sweep, sweep, tab.p, sweep, st);
    if (!rc) rc = cudaStreamSynchronize(st) == cudaSuccess ? COSM_OK : fail(COSM_ERR_CUDA, "step failed");
    tab.release();
    h->sweep_idx = sweep;
    h->have_result = false;
    h->have_trace = false;
    h->bits_valid = false;
    h->launches = 1;
    return rc;
}

extern "C" int cosm_readout(cosm_handle *h, void *stream)
{
    NvtxRange range("cosm_readout");
    if (!h) return fail(COSM_ERR_INVALID_ARG, "NULL handle");
    if (!h->have_state) return fail(COSM_ERR_STATE, "no state yet");
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    int rc = launch_on_state(h, SEG_LOAD | SEG_READOUT, 1, 0, h->d_alpha.p, 1, st);
    if (rc) return rc;
    h->launches = 2;
    if (h->prm.flags & COSM_OPT_BISECTOR) {
        if ((rc = launch_opt_readout(h, false, st))) return rc;
        h->launches = 3;
    }
    h->bits_valid = false;
    h->have_trace = false;
    if ((rc = launch_finalize(h, st))) return rc;
    h->have_result = true;
    return COSM_OK;
}

extern "C" int cosm_layout(cosm_handle *h, int32_t out[8])
{
    if (!h || !out) return fail(COSM_ERR_INVALID_ARG, "NULL argument");
    out[0] = h->K;
    out[1] = h->threads;
    out[2] = (int32_t)h->smem;
    out[3] = h->occupancy;
    out[4] = h->mode == MODE_LATTICE2D_ ? 2 : (h->lattice ? 1 : 0);
    out[5] = h->grid;
    out[6] = h->launches;
    out[7] = h->C;
    return COSM_OK;
}

extern "C" int cosm_layout_form(cosm_handle *h, int32_t out[4])
{
    if (!h || !out) return fail(COSM_ERR_INVALID_ARG, "NULL argument");
    out[0] = h->shape;
    out[1] = h->shape >= 0 && h->ragged;
    out[2] = h->format;
    out[3] = 0;
    return COSM_OK;
}

extern "C" int cosm_solve(const cosm_graph_desc *g, const cosm_params *p, int64_t sweeps, int32_t replicas,
                          uint64_t seed, int64_t *best_cut, int64_t *energy, int8_t *spins,
                          int64_t *replica_cuts)
{
    cosm_handle *h = nullptr;
    int rc = cosm_create(g, p, &h);
    if (rc) return rc;
    rc = cosm_run(h, sweeps, replicas, seed, INT64_MIN, nullptr);
    if (!rc) rc = cosm_get_best(h, best_cut, energy, nullptr, spins);
    if (!rc && replica_cuts) rc = cosm_get_replica_cuts(h, replica_cuts, nullptr);
    cosm_destroy(h);
    return rc;
}

// ====================================================================== batch
// Many instances of uneven size run together. Each instance is a handle as
// above; its replica tiles form units (instance, tile) = one whole trial of
// K replicas. Units of one (storage, K, kernel mode) class share a
// persistent launch whose CTAs drain a queue ordered by decreasing cost
// (longest processing time first); class launches are forked on separate
// streams so a class's tail overlaps the next class's start, and the whole
// run -- counter resets, class kernels, per-instance finalisation -- is
// captured once into a CUDA graph and replayed while the layout is unchanged.

struct BatchClass {
    int storage, K, mode;
    int shape;          // patch shape of lattices kept in registers (-1: none)
    bool ragged;
    int format;         // record-table format of edge lists (-1: none)
    int threads;        // threads per CTA
    size_t smem;        // largest tile of the class
    int grid;           // CTAs (resident capacity, capped by units)
    int32_t unit0, units;
};

// What an instance's layout in a batch was chosen for, and its CTAs per SM: a
// run with the same ones keeps the layout (choosing it asks the driver for the
// occupancy of up to 24 kernel configurations).
struct BatchChoice {
    int32_t replicas = 0, fill = 0, policy = -1, threads = -1, occupancy = 0;
};

struct cosm_batch {
    std::vector<cosm_handle *> hs;
    std::vector<BatchChoice> chosen;  // per instance; empty after a run that failed
    std::vector<BatchClass> classes;
    std::vector<BatchUnit> h_units;
    DevBuf<BatchUnit> d_units;
    DevBuf<InstView> d_insts;
    DevBuf<BatchFinal> d_fin;
    DevBuf<int32_t> d_counters;
    std::vector<cudaStream_t> side;  // one per class (created on demand)
    std::vector<cudaEvent_t> ev;     // fork + one per class
    cudaStream_t own = nullptr;      // capture stream (the legacy stream cannot capture)
    cudaGraphExec_t exec = nullptr;
    std::vector<int64_t> sig;        // layout signature of the captured graph
    int policy = 0;                  // 0: per-instance rule for a full GPU, 1: smallest tile, 2: per-instance rule,
                                     // 3: rule for a full GPU with ties to the narrower tile
    int threads = 0;                 // 0: per-class rule, else forced
    cudaStream_t last = nullptr;
    bool have_result = false;
    int64_t launches = 0;
    int64_t graph_builds = 0;
};

extern "C" void cosm_batch_destroy(cosm_batch *b)
{
    if (!b) return;
    if (b->own) cudaStreamSynchronize(b->own);
    // instances first: their handles still name the batch's stream
    for (cosm_handle *h : b->hs) {
        h->stream = nullptr;
        h->have_state = false;
        cosm_destroy(h);
    }
    b->hs.clear();
    if (b->exec) cudaGraphExecDestroy(b->exec);
    for (cudaStream_t s : b->side) cudaStreamDestroy(s);
    for (cudaEvent_t e : b->ev) cudaEventDestroy(e);
    if (b->own) cudaStreamDestroy(b->own);
    b->d_units.release(); b->d_insts.release(); b->d_fin.release(); b->d_counters.release();
    delete b;
}

extern "C" int cosm_batch_create(int32_t count, const cosm_graph_desc *graphs, const cosm_params *params,
                                 int32_t shared_params, cosm_batch **out)
{
    NvtxRange range("cosm_batch_create");
    if (!graphs || !params || !out || count < 1 || count > (1 << 20))
        return fail(COSM_ERR_INVALID_ARG, "bad batch arguments");
    *out = nullptr;
    // host-side checks of every instance before any device work
    for (int32_t i = 0; i < count; ++i) {
        const int rc = single_only(&graphs[i], shared_params ? &params[0] : &params[i]);
        if (rc) return fail(rc, "instance " + std::to_string(i) + ": " + g_err);
    }
    cosm_batch *b = new (std::nothrow) cosm_batch();
    if (!b) return fail(COSM_ERR_NOMEM, "host allocation failed");
    // instances are created by host worker threads (validation, colouring
    // and device tables of each run in parallel), each with the caller's
    // device current; the first failing instance is reported
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) {
        delete b;
        return fail(COSM_ERR_CUDA, "cudaGetDevice failed");
    }
    b->hs.assign((size_t)count, nullptr);
    std::vector<int> rcs((size_t)count, COSM_OK);
    std::vector<std::string> msgs((size_t)count);
    const auto work = [&](size_t i) {
        const cosm_params *pi = shared_params ? &params[0] : &params[i];
        if ((rcs[i] = cosm_create(&graphs[i], pi, &b->hs[i]))) msgs[i] = g_err;
    };
    if (count < 4)
        for (size_t i = 0; i < (size_t)count; ++i) work(i);
    else
        side_by_side((size_t)count, dev, work);
    for (int32_t i = 0; i < count; ++i) {
        if (rcs[(size_t)i]) {
            std::string msg = "instance " + std::to_string(i) + ": " + msgs[(size_t)i];
            const int rc = rcs[(size_t)i];
            b->hs.erase(std::remove(b->hs.begin(), b->hs.end(), nullptr), b->hs.end());
            cosm_batch_destroy(b);
            return fail(rc, msg);
        }
    }
    if (cudaStreamCreateWithFlags(&b->own, cudaStreamNonBlocking) != cudaSuccess) {
        cosm_batch_destroy(b);
        return fail(COSM_ERR_CUDA, "stream creation failed");
    }
    *out = b;
    return COSM_OK;
}

// Tile layout of one instance inside a batch. Policy 0: the single-instance
// rule (choose_layout) for `fill` replicas, 0.6 of the number of this
// instance's trials that would be as much work as the whole batch: a batch
// that fills the GPU takes the tiles that keep it busiest, a small one the
// tiles that finish a trial soonest (100 sweeps of 16 tori and graphs of 800
// to 3,000 vertices: 2.2 ms at the whole fill, 1.5 at 0.6, 1.4 at 0.35; 48 of
// up to 20,000: 9.0 / 8.7 / 9.1). Policy 1: the narrowest tile of the storage
// type. Policy 2: the single-instance rule with the instance's own replica
// count. Policy 3: as policy 0 with ties to the narrower tile (more CTAs per
// SM, whose barriers and record loads overlap; modelled costs within 10 % are
// a tie). Kernels without a fitted cost
// (plain records, lattices on shared memory) score policies 0, 1 and 3 as if
// the run filled every CTA slot.
static int batch_instance_layout(cosm_batch *b, cosm_handle *h, int32_t replicas, int32_t fill)
{
    int rc;
    if (b->policy == 2) return choose_layout(h, replicas);
    if ((rc = choose_layout(h, fill, b->policy == 3))) return rc;
    if (h->shape < 0 && h->format < 0 && (rc = choose_layout(h, 1 << 23, b->policy == 3))) return rc;
    // two replicas are the least a lattice in registers has
    const int narrowest = h->prm.storage == COSM_F32 && h->shape < 0 ? 1 : 2;
    if (b->policy == 1 && h->K != narrowest) return choose_layout(h, fill, false, narrowest);
    return COSM_OK;
}

// The device tables of every instance's layout. Missing ones (a first run, or
// another layout) are built by host threads side by side.
static int batch_tables(cosm_batch *b)
{
    std::vector<cosm_handle *> todo;
    for (cosm_handle *h : b->hs) {
        bool there = h->shape < 0 && h->format < 0;
        if (h->shape >= 0) there = h->d_pwt[h->shape].p != nullptr;
        for (size_t k = 0; k < h->tables.size() && h->format >= 0 && !there; ++k) {
            const RecordTable &t = *h->tables[k];
            there = t.K == h->K && t.threads == h->threads && t.format == h->format;
        }
        if (there) {
            if (int rc = ensure_tables(h)) return rc;
        } else {
            todo.push_back(h);
        }
    }
    if (todo.empty()) return COSM_OK;
    int dev = 0;
    CK(cudaGetDevice(&dev));
    std::vector<int> rcs(todo.size(), COSM_OK);
    std::vector<std::string> msgs(todo.size());
    side_by_side(todo.size(), dev, [&](size_t i) {
        if ((rcs[i] = ensure_tables(todo[i]))) msgs[i] = g_err;
    });
    for (size_t i = 0; i < todo.size(); ++i)
        if (rcs[i]) return fail(rcs[i], msgs[i]);
    return COSM_OK;
}

static int batch_layout(cosm_batch *b, const int64_t *sweeps, const int32_t *replicas, const uint64_t *seeds,
                        cudaStream_t st)
{
    const int n = (int)b->hs.size();
    std::vector<InstView> views((size_t)n);
    std::vector<BatchFinal> fins((size_t)n);
    b->chosen.resize((size_t)n);
    double total = 0.0;  // edge updates of the run
    for (int i = 0; i < n; ++i) total += (double)b->hs[(size_t)i]->g.m * (double)replicas[i] * (double)sweeps[i];
    for (int i = 0; i < n; ++i) {
        cosm_handle *h = b->hs[(size_t)i];
        int rc;
        const double share = 0.6 * total / ((double)h->g.m * (double)sweeps[i]);
        const int32_t fill = (int32_t)std::max((double)replicas[i], std::min(share, 8388608.0));
        BatchChoice &was = b->chosen[(size_t)i];
        if (was.replicas != replicas[i] || was.fill != fill || was.policy != b->policy || was.threads != b->threads) {
            was = BatchChoice();
            if ((rc = batch_instance_layout(b, h, replicas[i], fill))) return rc;
            if (b->threads && h->shape < 0) {
                h->threads = at_least_a_warp(b->threads);  // a tuning file may name any count
                if (h->format >= 0) h->threads = (h->threads + 31) / 32 * 32;  // whole warps
                while (h->threads > 64 && kernel_occupancy(h, h->threads, h->smem, true) == 0)
                    h->threads = half_threads(h->threads, h->format >= 0);
            }
            was = BatchChoice{replicas[i], fill, b->policy, b->threads, kernel_occupancy(h, h->threads, h->smem, true)};
        }
        h->replicas = replicas[i];
        h->seed = seeds[i];
        if ((rc = ensure_run_buffers(h, replicas[i]))) return rc;
        if ((rc = upload_alpha(h, sweeps[i], st))) return rc;
    }
    if (int rc = batch_tables(b)) return rc;
    for (int i = 0; i < n; ++i) {
        cosm_handle *h = b->hs[(size_t)i];
        InstView v = inst_view(h);
        v.alpha_tab = h->d_alpha.p;
        v.alpha_base = 1;
        v.S = sweeps[i];
        views[(size_t)i] = v;
        fins[(size_t)i] = BatchFinal{h->W, h->d_spins.p, h->d_best.p, h->prm.storage, 0};
    }
    // classes: instances of one kernel (storage, tile width, mode), thread
    // count and occupancy share a persistent launch (the class's largest
    // tile has the same occupancy as every other, occupancy falling with
    // shared memory); their units form one queue, longest trials first
    b->classes.clear();
    b->h_units.clear();
    struct Key { int storage, K, mode, shape; bool ragged; int format, threads, occ; };
    std::vector<Key> keys;
    std::vector<int> cls((size_t)n);
    for (int i = 0; i < n; ++i) {
        const cosm_handle *h = b->hs[(size_t)i];
        const Key k{h->prm.storage, h->K, h->mode, h->shape, h->shape >= 0 && h->ragged, h->format, h->threads,
                    b->chosen[(size_t)i].occupancy};
        int c = -1;
        for (size_t q = 0; q < keys.size() && c < 0; ++q) {
            const Key &o = keys[q];
            if (o.storage == k.storage && o.K == k.K && o.mode == k.mode && o.shape == k.shape && o.ragged == k.ragged &&
                o.format == k.format && o.threads == k.threads && o.occ == k.occ)
                c = (int)q;
        }
        if (c < 0) {
            keys.push_back(k);
            c = (int)keys.size() - 1;
        }
        cls[(size_t)i] = c;
    }
    int dev_sms = b->hs[0]->num_sms;
    for (size_t c = 0; c < keys.size(); ++c) {
        BatchClass bc{keys[c].storage, keys[c].K, keys[c].mode, keys[c].shape, keys[c].ragged, keys[c].format,
                      keys[c].threads, 0, 0,
                      (int32_t)b->h_units.size(), 0};
        std::vector<std::pair<double, BatchUnit>> us;
        for (int i = 0; i < n; ++i) {
            if (cls[(size_t)i] != (int)c) continue;
            const cosm_handle *h = b->hs[(size_t)i];
            bc.smem = std::max(bc.smem, h->smem);
            const int64_t tiles = (replicas[i] + h->K - 1) / h->K;
            const double cost = (double)h->g.m * (double)h->K * (double)sweeps[i];
            for (int64_t t = 0; t < tiles; ++t)
                us.push_back({cost, BatchUnit{i, (int32_t)t, SEG_INIT | SEG_READOUT | SEG_STORE, 0, 1, sweeps[i]}});
        }
        std::stable_sort(us.begin(), us.end(), [](const auto &x, const auto &y) { return x.first > y.first; });
        for (auto &u : us) b->h_units.push_back(u.second);
        bc.units = (int32_t)us.size();
        int T = bc.threads;
        const auto occ_of = [&](int threads) {
            return bc.shape >= 0    ? patch_occupancy(bc.storage, bc.K, bc.shape, bc.ragged, threads, bc.smem)
                   : bc.format >= 0 ? edges_occupancy(bc.storage, bc.K, bc.format, threads, bc.smem)
                                    : batch_occupancy(bc.storage, bc.K, bc.mode, threads, bc.smem);
        };
        int occ = occ_of(T);
        while (occ == 0 && T > 64 && bc.shape < 0 && bc.format < 0) {  // tables are laid out for T
            T /= 2;
            occ = occ_of(T);
        }
        if (occ == 0) return fail(COSM_ERR_TOO_LARGE, "a batch tile does not fit on an SM");
        bc.threads = T;
        bc.grid = (int)std::min<int64_t>((int64_t)occ * dev_sms, bc.units);
        b->classes.push_back(bc);
    }
    int rc;
    if ((rc = b->d_insts.ensure((size_t)n)) || (rc = b->d_fin.ensure((size_t)n)) ||
        (rc = b->d_units.ensure(b->h_units.size())) || (rc = b->d_counters.ensure(b->classes.size())))
        return rc;
    CK(cudaMemcpyAsync(b->d_insts.p, views.data(), views.size() * sizeof(InstView), cudaMemcpyHostToDevice, st));
    CK(cudaMemcpyAsync(b->d_fin.p, fins.data(), fins.size() * sizeof(BatchFinal), cudaMemcpyHostToDevice, st));
    CK(cudaMemcpyAsync(b->d_units.p, b->h_units.data(), b->h_units.size() * sizeof(BatchUnit),
                       cudaMemcpyHostToDevice, st));
    CK(cudaStreamSynchronize(st));  // host tables are released on return
    return COSM_OK;
}

// Records the class launches and the finaliser on `st` (captured or not).
static int batch_enqueue(cosm_batch *b, cudaStream_t st)
{
    const size_t nc = b->classes.size();
    while (b->side.size() < nc) {
        cudaStream_t s;
        CK(cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking));
        b->side.push_back(s);
    }
    while (b->ev.size() < nc + 1) {
        cudaEvent_t e;
        CK(cudaEventCreateWithFlags(&e, cudaEventDisableTiming));
        b->ev.push_back(e);
    }
    CK(cudaMemsetAsync(b->d_counters.p, 0, nc * 4, st));
    CK(cudaEventRecord(b->ev[0], st));
    for (size_t c = 0; c < nc; ++c) {
        const BatchClass &bc = b->classes[c];
        CK(cudaStreamWaitEvent(b->side[c], b->ev[0], 0));
        BatchArgs a{b->d_insts.p, b->d_units.p + bc.unit0, bc.units, b->d_counters.p + c};
        if (bc.units > 0 && kernel_launch_queue(LaunchCfg{bc.mode, bc.storage, bc.K, bc.threads, bc.grid, bc.smem, false, bc.shape,
                                                       bc.ragged, bc.format}, a, b->side[c]))
            return fail(COSM_ERR_CUDA, std::string("batch launch: ") + cudaGetErrorString(cudaGetLastError()));
        CK(cudaEventRecord(b->ev[c + 1], b->side[c]));
    }
    for (size_t c = 0; c < nc; ++c) CK(cudaStreamWaitEvent(st, b->ev[c + 1], 0));
    if (batch_finalize_launch((int)b->hs.size(), b->d_insts.p, b->d_fin.p, st))
        return fail(COSM_ERR_CUDA, std::string("batch finalize: ") + cudaGetErrorString(cudaGetLastError()));
    return COSM_OK;
}

// Lays a run out and launches it on the batch's stream, after earlier work on
// the caller's and before later.
static int batch_launch_run(cosm_batch *b, const int64_t *sweeps, const int32_t *replicas, const uint64_t *seeds,
                            cudaStream_t user)
{
    cudaStream_t st = b->own;
    // order the batch after earlier work on the caller's stream
    cudaEvent_t e0;
    CK(cudaEventCreateWithFlags(&e0, cudaEventDisableTiming));
    CK(cudaEventRecord(e0, user));
    CK(cudaStreamWaitEvent(st, e0, 0));
    cudaEventDestroy(e0);
    int rc = batch_layout(b, sweeps, replicas, seeds, st);
    if (rc) return rc;
    std::vector<int64_t> sig;
    sig.push_back((int64_t)(uintptr_t)b->d_insts.p);
    sig.push_back((int64_t)(uintptr_t)b->d_units.p);
    sig.push_back((int64_t)(uintptr_t)b->d_counters.p);
    for (const BatchClass &bc : b->classes) {
        sig.push_back(bc.storage); sig.push_back(bc.K); sig.push_back(bc.mode); sig.push_back(bc.threads);
        sig.push_back(bc.shape); sig.push_back(bc.ragged); sig.push_back(bc.format);
        sig.push_back((int64_t)bc.smem); sig.push_back(bc.grid); sig.push_back(bc.unit0); sig.push_back(bc.units);
    }
    if (!b->exec || sig != b->sig) {
        if (b->exec) {
            cudaGraphExecDestroy(b->exec);
            b->exec = nullptr;
        }
        cudaGraph_t graph = nullptr;
        CK(cudaStreamBeginCapture(st, cudaStreamCaptureModeThreadLocal));
        rc = batch_enqueue(b, st);
        cudaError_t ce = cudaStreamEndCapture(st, &graph);
        if (rc) {
            if (graph) cudaGraphDestroy(graph);
            return rc;
        }
        if (ce != cudaSuccess) return fail(COSM_ERR_CUDA, std::string("graph capture: ") + cudaGetErrorString(ce));
        ce = cudaGraphInstantiate(&b->exec, graph, 0);
        cudaGraphDestroy(graph);
        if (ce != cudaSuccess) return fail(COSM_ERR_CUDA, std::string("graph instantiate: ") + cudaGetErrorString(ce));
        b->sig = sig;
        b->graph_builds++;
    }
    CK(cudaGraphLaunch(b->exec, st));
    cudaEvent_t e1;
    CK(cudaEventCreateWithFlags(&e1, cudaEventDisableTiming));
    CK(cudaEventRecord(e1, st));
    CK(cudaStreamWaitEvent(user, e1, 0));
    cudaEventDestroy(e1);
    for (cosm_handle *h : b->hs) {
        h->stream = st;
        h->have_state = true;
        h->have_result = true;
    }
    b->last = st;
    b->have_result = true;
    b->launches = (int64_t)b->classes.size() + 1;
    return COSM_OK;
}

extern "C" int cosm_batch_run(cosm_batch *b, const int64_t *sweeps, const int32_t *replicas,
                              const uint64_t *seeds, void *stream)
{
    NvtxRange range("cosm_batch_run");
    if (!b || !sweeps || !replicas || !seeds) return fail(COSM_ERR_INVALID_ARG, "NULL argument");
    for (size_t i = 0; i < b->hs.size(); ++i)
        if (sweeps[i] < 1 || sweeps[i] >= ((int64_t)1 << 31) || replicas[i] < 1 || replicas[i] >= (1 << 24))
            return fail(COSM_ERR_INVALID_ARG, "instance " + std::to_string(i) + ": bad sweeps or replicas");
    const int rc = batch_launch_run(b, sweeps, replicas, seeds, reinterpret_cast<cudaStream_t>(stream));
    if (rc) {
        // some instances may have a new layout: the last run's states and results
        // end here
        for (cosm_handle *h : b->hs) h->have_state = h->have_result = false;
        b->have_result = false;
        b->chosen.clear();
    }
    return rc;
}

extern "C" int cosm_batch_sync(cosm_batch *b)
{
    if (!b) return fail(COSM_ERR_INVALID_ARG, "NULL batch");
    CK(cudaStreamSynchronize(b->own));
    return COSM_OK;
}

extern "C" int cosm_batch_get_best(cosm_batch *b, int32_t i, int64_t *cut, int64_t *energy, int32_t *replica,
                                   int8_t *spins)
{
    if (!b || i < 0 || i >= (int32_t)b->hs.size()) return fail(COSM_ERR_INVALID_ARG, "bad instance index");
    if (!b->have_result) return fail(COSM_ERR_STATE, "no batch run yet");
    return cosm_get_best(b->hs[(size_t)i], cut, energy, replica, spins);
}

extern "C" int cosm_batch_get_replica_cuts(cosm_batch *b, int32_t i, int64_t *cuts, int32_t *best_p)
{
    if (!b || i < 0 || i >= (int32_t)b->hs.size()) return fail(COSM_ERR_INVALID_ARG, "bad instance index");
    if (!b->have_result) return fail(COSM_ERR_STATE, "no batch run yet");
    return cosm_get_replica_cuts(b->hs[(size_t)i], cuts, best_p);
}

extern "C" int cosm_batch_get_state(cosm_batch *b, int32_t i, double *phases)
{
    if (!b || i < 0 || i >= (int32_t)b->hs.size()) return fail(COSM_ERR_INVALID_ARG, "bad instance index");
    return cosm_get_state(b->hs[(size_t)i], phases);
}

// Autotuner: times short runs of the whole batch (probe_sweeps sweeps per
// instance, the caller's replica counts) for each tile policy and thread
// count and keeps the fastest. With COSM_TUNE_CACHE set, choices are read
// from / appended to that text file, keyed by the batch's shape.
extern "C" int cosm_batch_tune(cosm_batch *b, const int32_t *replicas, int64_t probe_sweeps, void *stream)
{
    NvtxRange range("cosm_batch_tune");
    if (!b || !replicas || probe_sweeps < 1) return fail(COSM_ERR_INVALID_ARG, "bad tuning arguments");
    const size_t n = b->hs.size();
    uint64_t key = 1469598103934665603ull;  // FNV-1a over the batch's shape
    auto mix = [&](uint64_t x) {
        for (int k = 0; k < 8; ++k) { key ^= (x >> (8 * k)) & 0xFF; key *= 1099511628211ull; }
    };
    for (size_t i = 0; i < n; ++i) {
        const cosm_handle *h = b->hs[i];
        mix((uint64_t)h->g.n); mix((uint64_t)h->g.m); mix((uint64_t)h->C); mix((uint64_t)h->mode);
        mix((uint64_t)h->prm.storage); mix((uint64_t)replicas[i]);
        // what decides an instance's kernel and record format besides
        mix((uint64_t)h->wmax); mix((uint64_t)h->prm.n_bisectors);
        mix((uint64_t)wrap_period(h->prm.alpha0_deg, h->prm.dwt_ratio, h->prm.dwt_period, h->prm.flags, h->mode,
                                  h->prm.storage, h->wbound));
    }
    mix(2);  // the policies' meaning: an entry chosen under another one is not taken
    const char *cache = std::getenv("COSM_TUNE_CACHE");
    if (cache) {
        FILE *f = std::fopen(cache, "r");
        if (f) {
            unsigned long long k;
            int pol, thr;
            while (std::fscanf(f, "%llx %d %d", &k, &pol, &thr) == 3)
                if (k == key) {
                    b->policy = pol;
                    b->threads = thr;
                    std::fclose(f);
                    return COSM_OK;
                }
            std::fclose(f);
        }
    }
    std::vector<int64_t> sw(n, probe_sweeps);
    std::vector<uint64_t> seeds(n, 12345);
    float best_ms = 1e30f;
    int best_pol = 0, best_thr = 0;
    cudaEvent_t e0, e1;
    CK(cudaEventCreate(&e0));
    CK(cudaEventCreate(&e1));
    // policies with the rule's thread counts, then the default policy with
    // forced thread counts
    const int cfgs[8][2] = {{0, 0}, {1, 0}, {2, 0}, {3, 0}, {0, 128}, {0, 256}, {0, 512}, {3, 256}};
    for (const auto &cf : cfgs) {
        const int pol = cf[0], thr = cf[1];
        b->policy = pol;
        b->threads = thr;
        int rc = cosm_batch_run(b, sw.data(), replicas, seeds.data(), stream);  // warm-up + graph build
        if (rc) continue;
        CK(cudaEventRecord(e0, b->own));
        rc = cosm_batch_run(b, sw.data(), replicas, seeds.data(), stream);
        CK(cudaEventRecord(e1, b->own));
        CK(cudaEventSynchronize(e1));
        if (rc) continue;
        float ms = 0.f;
        cudaEventElapsedTime(&ms, e0, e1);
        if (ms < best_ms) {
            best_ms = ms;
            best_pol = pol;
            best_thr = thr;
        }
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    b->policy = best_pol;
    b->threads = best_thr;
    if (cache) {
        FILE *f = std::fopen(cache, "a");
        if (f) {
            std::fprintf(f, "%llx %d %d\n", (unsigned long long)key, best_pol, best_thr);
            std::fclose(f);
        }
    }
    return COSM_OK;
}

extern "C" int cosm_batch_layout(cosm_batch *b, int32_t i, int32_t out[8])
{
    if (!b || i < 0 || i >= (int32_t)b->hs.size()) return fail(COSM_ERR_INVALID_ARG, "bad instance index");
    if (!b->have_result) return fail(COSM_ERR_STATE, "no batch run yet");
    return cosm_layout(b->hs[(size_t)i], out);
}

extern "C" int cosm_batch_info(cosm_batch *b, int64_t out[8])
{
    if (!b || !out) return fail(COSM_ERR_INVALID_ARG, "NULL argument");
    out[0] = (int64_t)b->hs.size();
    out[1] = (int64_t)b->classes.size();
    out[2] = (int64_t)b->h_units.size();
    out[3] = b->launches;
    out[4] = b->graph_builds;
    out[5] = b->policy;
    out[6] = b->threads;
    int64_t ctas = 0;
    for (const BatchClass &bc : b->classes) ctas += bc.grid;
    out[7] = ctas;
    return COSM_OK;
}
