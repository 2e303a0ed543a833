// Several steps per launch in shared-memory tiles: D2Q9 with float population storage.
#include "step_block.cuh"

namespace lbm {

// BLOCK_STEPS steps from a's source to its destination.  Not for the lagged closure, whose stored tau the
// margins would each advance, nor for the power law, n != 1, above 2^19 nodes
// (step_block.cuh).
cudaError_t block_d2q9_f32(const StepArgs<float>& a, int closure, int formula, int force, cudaStream_t s) {
    switch (closure) {
        case CL_NEWTON: return launch_block_c<CL_NEWTON>(a, formula, force, s);
        case CL_SMAG: return launch_block_c<CL_SMAG>(a, formula, force, s);
        case CL_POWERLAW:
            if (a.pl_nm1 != 0.0f && (long long)a.nx * a.ny > (1LL << 19)) return cudaErrorNotSupported;
            return launch_block_c<CL_POWERLAW>(a, formula, force, s);
        case CL_SMAG_DEV: return launch_block_c<CL_SMAG_DEV>(a, formula, force, s);
        default: return cudaErrorNotSupported;
    }
}

}  // namespace lbm
