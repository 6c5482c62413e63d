// Register-resident lattice kernels: __nv_bfloat16 phases, 2 replicas per tile.
#include "cosm_patch.cuh"

int cosm::patch_call_bf16_k2(const PatchCall &c) { return patch_dispatch<__nv_bfloat16, 2>(c); }
