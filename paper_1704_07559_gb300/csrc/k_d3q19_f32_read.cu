// Read-out kernel instantiations for lattice D3Q19 with float population storage.
#include "read.cuh"
LBM_DEFINE_READ_ENTRY(d3q19_f32, lbm::D3Q19, float, true)
