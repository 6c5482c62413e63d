// Register-resident lattice kernels: uint16_t phases, 4 replicas per tile.
#include "cosm_patch.cuh"

int cosm::patch_call_q16_k4(const PatchCall &c) { return patch_dispatch<uint16_t, 4>(c); }
