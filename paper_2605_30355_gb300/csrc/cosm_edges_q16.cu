// Edge-list kernels on record tables: uint16_t phases.
#include "cosm_edges.cuh"

int cosm::edges_call_q16(const EdgesCall &c) { return edges_dispatch<uint16_t, 2, 4, 8>(c); }
