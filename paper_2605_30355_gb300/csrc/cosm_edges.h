// Host-side interface of the edge-list kernels on record tables
// (cosm_edges.cuh).
#pragma once

#include <stddef.h>
#include <stdint.h>

#include "cosm_internal.h"

namespace cosm {

// Record formats of an edge list (InstView::rec). With E bytes per slot:
//  EDGES_SIGN    one word: [w = -1] | slot(i) << 1 | slot(j) << 16; +-1 weights on at most 2^15 slots
//  EDGES_PACK    one word: w + 4 (E = 8) or w + 8 (E = 16) | byte offset of x_i | slot(j) << 18; at most
//                2^14 slots, |w| <= 3 or 7
//  EDGES_WEIGHT  two words: byte offset of x_i; byte offset of x_j | weight << 18 (fixed point), or | the top
//                14 bits of the weight as binary32 (float forms; exact for |w| < 64)
// EDGES_EACH: every binary32 update is wrapped (not with EDGES_SIGN).
enum EdgeFormat { EDGES_SIGN = 0, EDGES_PACK = 1, EDGES_WEIGHT = 2, EDGES_EACH = 4 };
constexpr uint32_t kNoEdge = 0xFFFFFFFFu;  // first word of an empty place

// A colour's edges come in rows of 32, one per lane; row k W + w is the k-th
// row of warp w (of W). Each warp has its rows of all non-empty colours one
// after the other in the record table (from word starts[w] on, followed by a
// copy of its first kRowsAhead rows, so that a fetch past the sweep's end
// finds the next sweep's first rows), and counts[w (n_colours + 1) + c] rows
// of colour c, the first count once more at the end. kPartial marks a count
// whose last row has empty places.
constexpr int kRowsAhead = 4;
constexpr uint32_t kPartial = 0x80000000u;

struct EdgesCall {
    enum What { OCCUPANCY, LAUNCH } what;
    int K;
    int format;
    int threads;
    size_t smem;
    int grid;
    bool cooperative;
    const KernelArgs *run;   // segment lists (single instance), or
    const BatchArgs *queue;  // a queue of units
    void *stream;
};
int edges_call_f32(const EdgesCall &c);
int edges_call_f16(const EdgesCall &c);
int edges_call_bf16(const EdgesCall &c);
int edges_call_q16(const EdgesCall &c);

}  // namespace cosm
