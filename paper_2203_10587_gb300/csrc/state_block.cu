// Block-per-state schedule (state_block.cuh): launches without generator masks or phase shifters.
#include <cuda_runtime.h>

#include "state_block.cuh"

namespace exago {

int state_allow_smem() {
    int e = launch_state_x<0>(0, DevNet{}, EvalReq{}, 0, nullptr, true);
    return e != 0 ? e : launch_state_gm(0, DevNet{}, EvalReq{}, 0, nullptr, true);
}

int launch_eval_state(const DevNet &N, const EvalReq &R, int nt, size_t smem, void *stream) {
    if (R.B <= 0) return 0;
    cudaStream_t st = (cudaStream_t)stream;
    if (R.gen_mask || R.tab || N.Gtf) return launch_state_gm(nt, N, R, smem, st, false);
    return launch_state_x<0>(nt, N, R, smem, st, false);
}

}  // namespace exago
