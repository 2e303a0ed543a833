// Several steps per launch in shared-memory tiles: D2Q9 with float population storage.
#include "step_block.cuh"

namespace lbm {

static cudaError_t dispatch(const StepArgs<float>& a, int rows, int closure, int formula, int force, bool prepare,
                            cudaStream_t s) {
    switch (closure) {
        case CL_NEWTON: return launch_block_c<CL_NEWTON>(a, rows, formula, force, prepare, s);
        case CL_SMAG: return launch_block_c<CL_SMAG>(a, rows, formula, force, prepare, s);
        case CL_POWERLAW: return launch_block_c<CL_POWERLAW>(a, rows, formula, force, prepare, s);
        case CL_SMAG_DEV: return launch_block_c<CL_SMAG_DEV>(a, rows, formula, force, prepare, s);
        default: return cudaErrorNotSupported;  // the lagged closure's stored tau the margins would each advance
    }
}

int block_d2q9_f32_rows(const StepArgs<float>& a, int closure, int formula, int force) {
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return 0;
    if (!block_pays(a, closure, force, sms)) return 0;
    const long long tiles = (a.nx + BW - 1LL) / BW * ((a.ny + 19LL) / 20);
    const int rows = tiles >= sms ? 20 : 16;
    return dispatch(a, rows, closure, formula, force, true, nullptr) == cudaSuccess ? rows : 0;
}

cudaError_t block_d2q9_f32(const StepArgs<float>& a, int rows, int closure, int formula, int force, cudaStream_t s) {
    return dispatch(a, rows, closure, formula, force, false, s);
}

}  // namespace lbm
