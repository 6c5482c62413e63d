// Edge-list kernels on record tables: __nv_bfloat16 phases.
#include "cosm_edges.cuh"

int cosm::edges_call_bf16(const EdgesCall &c) { return edges_dispatch<__nv_bfloat16, 2, 4, 8>(c); }
