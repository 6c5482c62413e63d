// Register-resident lattice kernels: __nv_bfloat16 phases, 4 replicas per tile.
#include "cosm_patch.cuh"

int cosm::patch_call_bf16_k4(const PatchCall &c) { return patch_dispatch<__nv_bfloat16, 4>(c); }
