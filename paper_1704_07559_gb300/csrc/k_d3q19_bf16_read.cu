// Read-out kernel instantiations for lattice D3Q19 with __nv_bfloat16 population storage.
#include "read.cuh"
LBM_DEFINE_READ_ENTRY(d3q19_bf16, lbm::D3Q19, __nv_bfloat16, false)
