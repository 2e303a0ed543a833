// Read-out kernel instantiations for lattice D2Q9 with float population storage.
#include "read.cuh"
LBM_DEFINE_READ_ENTRY(d2q9_f32, lbm::D2Q9, float, true)
