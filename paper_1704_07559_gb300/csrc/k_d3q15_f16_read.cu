// Read-out kernel instantiations for lattice D3Q15 with __half population storage.
#include "read.cuh"
LBM_DEFINE_READ_ENTRY(d3q15_f16, lbm::D3Q15, __half, false)
