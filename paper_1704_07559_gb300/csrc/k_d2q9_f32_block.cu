// Several steps per launch in shared-memory tiles: D2Q9 with float population storage.
#include "step_block.cuh"

namespace lbm {

// Not for the lagged closure, whose stored tau the margins would each advance
bool block_d2q9_f32_pays(const StepArgs<float>& a, int closure, int force) {
    int dev = 0, sms = 0;
    if (closure == CL_SMAG_LAGGED || cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return false;
    return block_pays(a, closure, force, sms);
}

// BLOCK_STEPS steps from a's source to its destination
cudaError_t block_d2q9_f32(const StepArgs<float>& a, int closure, int formula, int force, cudaStream_t s) {
    switch (closure) {
        case CL_NEWTON: return launch_block_c<CL_NEWTON>(a, formula, force, s);
        case CL_SMAG: return launch_block_c<CL_SMAG>(a, formula, force, s);
        case CL_POWERLAW: return launch_block_c<CL_POWERLAW>(a, formula, force, s);
        case CL_SMAG_DEV: return launch_block_c<CL_SMAG_DEV>(a, formula, force, s);
        default: return cudaErrorNotSupported;
    }
}

}  // namespace lbm
