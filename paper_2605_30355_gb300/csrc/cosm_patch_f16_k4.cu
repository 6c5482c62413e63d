// Register-resident lattice kernels: __half phases, 4 replicas per tile.
#include "cosm_patch.cuh"

int cosm::patch_call_f16_k4(const PatchCall &c) { return patch_dispatch<__half, 4>(c); }
