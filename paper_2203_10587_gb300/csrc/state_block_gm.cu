// Block-per-state schedule (state_block.cuh): launches with generator masks, a gathered batch
// (whose states may carry them) or phase shifters.  Compiled beside state_block.cu.
#include <cuda_runtime.h>

#include "state_block.cuh"

namespace exago {

int launch_state_gm(int nt, const DevNet &N, const EvalReq &R, size_t smem, cudaStream_t st, bool set_smem) {
    return launch_state_x<W_GM | W_PS>(nt, N, R, smem, st, set_smem);
}

}  // namespace exago
