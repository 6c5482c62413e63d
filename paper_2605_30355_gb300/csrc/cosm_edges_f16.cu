// Edge-list kernels on record tables: __half phases.
#include "cosm_edges.cuh"

int cosm::edges_call_f16(const EdgesCall &c) { return edges_dispatch<__half, 2, 4, 8>(c); }
