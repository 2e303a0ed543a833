// Read-out kernel instantiations for lattice D3Q15 with __nv_bfloat16 population storage.
#include "read.cuh"
LBM_DEFINE_READ_ENTRY(d3q15_bf16, lbm::D3Q15, __nv_bfloat16, false)
