// Edge-list kernels on record tables: float phases.
#include "cosm_edges.cuh"

int cosm::edges_call_f32(const EdgesCall &c) { return edges_dispatch<float, 1, 2, 4>(c); }
