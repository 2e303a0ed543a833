// Read-out kernel instantiations for lattice D3Q15 with float population storage.
#include "read.cuh"
LBM_DEFINE_READ_ENTRY(d3q15_f32, lbm::D3Q15, float, true)
