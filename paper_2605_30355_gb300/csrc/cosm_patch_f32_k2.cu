// Register-resident lattice kernels: float phases, 2 replicas per tile.
#include "cosm_patch.cuh"

int cosm::patch_call_f32_k2(const PatchCall &c) { return patch_dispatch<float, 2>(c); }
