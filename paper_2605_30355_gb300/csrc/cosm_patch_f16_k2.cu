// Register-resident lattice kernels: __half phases, 2 replicas per tile.
#include "cosm_patch.cuh"

int cosm::patch_call_f16_k2(const PatchCall &c) { return patch_dispatch<__half, 2>(c); }
