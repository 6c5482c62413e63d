// Host-side interface of the lattice kernels that keep phases in registers
// (cosm_patch.cuh): the patch shapes and the calls the runtime makes.
#pragma once

#include <stddef.h>
#include <stdint.h>

#include "cosm_internal.h"

namespace cosm {

// Shapes (index, block rows, block columns), largest first. A patch of R x C
// 2x2 blocks holds 4 R C sites.
#define COSM_PATCH_SHAPES(X) X(0, 2, 5) X(1, 2, 4) X(2, 2, 3) X(3, 2, 2) X(4, 1, 2) X(5, 1, 1)
constexpr int kPatchShapes = 6;
constexpr int kPatchR[kPatchShapes] = {2, 2, 2, 2, 1, 1};
constexpr int kPatchC[kPatchShapes] = {5, 4, 3, 2, 2, 1};

// Threads per CTA a shape's kernel is compiled for: the register file's 65,536
// registers divided by what the shape needs (its phases plus about 45).
constexpr int patch_max_threads(int R, int C, int site_bytes)
{
    const int regs = R * C * site_bytes + 45;
    return regs > 96 ? 512 : regs > 80 ? 640 : regs > 64 ? 768 : 1024;
}

// Four 16-bit floats per site spill above 2 x 2 blocks: no such kernel.
constexpr bool patch_built(bool float16, int K, int R, int C) { return !(float16 && K == 4 && R * C > 4); }

struct PatchCall {
    enum What { OCCUPANCY, LAUNCH } what;
    int shape;
    int ragged;
    int threads;
    size_t smem;
    int grid;
    bool cooperative;
    const KernelArgs *run;   // segment lists (single instance), or
    const BatchArgs *queue;  // a queue of units
    void *stream;
};

// One translation unit per storage form.
int patch_call_f32_k2(const PatchCall &c);
int patch_call_f16_k2(const PatchCall &c);
int patch_call_f16_k4(const PatchCall &c);
int patch_call_bf16_k2(const PatchCall &c);
int patch_call_bf16_k4(const PatchCall &c);
int patch_call_q16_k2(const PatchCall &c);
int patch_call_q16_k4(const PatchCall &c);

}  // namespace cosm
