// Register-resident lattice kernels: uint16_t phases, 2 replicas per tile.
#include "cosm_patch.cuh"

int cosm::patch_call_q16_k2(const PatchCall &c) { return patch_dispatch<uint16_t, 2>(c); }
