// Block-per-state schedule of the polar AC-OPF model evaluation (ExaGO, arXiv 2203.10587,
// Sec. III, eqs. (7)-(10)) for grids whose branch-end records fit one block's shared memory: a
// block evaluates one state, its branches, then, after a barrier, its buses.
//
// What bounds it: for few states the latency of one branch item and one bus item (a warp's FP64
// instruction holds its pipe for 64 cycles, about 110 of them a branch).  The persistent schedule
// adds to that a counter reset in front of the launch, tickets, a release and an acquire through
// L2 between the two items and records read back from L2; here the records never leave the SM and
// the launch is one kernel.  Measured (us, all outputs; persistent, then this): 30 buses x 1 state
// 20.5, 14.4; 118 x 304 33.2, 22.5; 200 x 152 36.7, 24.6; 300 x 304 67.5, 47.2.  Of one 30-bus
// state's 14.4 us, 4.2 are a launch that computes the objective alone; the rest is one warp's
// chain through a branch item and a bus item (warming L1 for the bus item beforehand changed
// nothing).  The items are the persistent schedule's own, so results are bitwise equal.
#pragma once

#include <cuda_runtime.h>

#include "eval_items.cuh"

namespace exago {

template <int WANT, int NT>
__global__ void __launch_bounds__(NT, 512 / NT) k_state(const DevNet N, const EvalReq R) {
    extern __shared__ __align__(16) double s_state[];
    __shared__ double s_part[OBJ_LANES];
    static_assert(OBJ_LANES % NT == 0, "objective lanes");
    const int b = blockIdx.x;
    double *recs = s_state, *stage = s_state + (size_t)NCOMP * N.nslot;
    if (WANT & (W_G | W_J | W_H))
        for (int l = threadIdx.x; l < N.nl; l += NT) branch_item<WANT>(N, R, b, l, recs);
    if (R.f)
        for (int q = 0; q < OBJ_LANES / NT; q++) obj_lanes<(WANT & W_GM) != 0, NT>(N, R, b, q, s_part);
    __syncthreads();
    if (R.f && threadIdx.x >= NT - 32) obj_tree_warp<true>(R, b, s_part);
    for (int i0 = 0; i0 < N.nb; i0 += NT) {
        if (WANT & (W_G | W_J | W_H))
            bus_tile<WANT, BlockGroup, true>(N, R, b, i0, recs, stage, R.stage_cap);
        if (i0 + (int)threadIdx.x < N.nb && R.grad)
            grad_bus<(WANT & W_GM) != 0>(N, R, b, i0 + threadIdx.x);
    }
}

// Launches (or, set_smem, opts in to kStateMaxBytes of shared memory) the variant for the
// requested outputs plus X = 0 or W_GM | W_PS.
template <int NT, int X>
static int launch_state_nt(const DevNet &N, const EvalReq &R, size_t smem, cudaStream_t st, bool set_smem) {
    auto go = [&](auto kern) -> int {
        if (set_smem)
            return (int)cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kStateMaxBytes);
        kern<<<R.B, NT, smem, st>>>(N, R);
        return (int)cudaGetLastError();
    };
    const int want = (R.gh ? W_G : 0) | (R.jval ? W_J : 0) | (R.hval ? W_H : 0);
    int e = 0;
    for (int w = 0; w < 8 && e == 0; w++) {
        if (!set_smem && w != want) continue;
        switch (w) {
            case 0: e = go(k_state<X, NT>); break;
            case 1: e = go(k_state<1 | X, NT>); break;
            case 2: e = go(k_state<2 | X, NT>); break;
            case 3: e = go(k_state<3 | X, NT>); break;
            case 4: e = go(k_state<4 | X, NT>); break;
            case 5: e = go(k_state<5 | X, NT>); break;
            case 6: e = go(k_state<6 | X, NT>); break;
            default: e = go(k_state<7 | X, NT>); break;
        }
    }
    return e;
}

template <int X>
static int launch_state_x(int nt, const DevNet &N, const EvalReq &R, size_t smem, cudaStream_t st, bool set_smem) {
    int e = 0;
    if (set_smem || nt == 64) e = launch_state_nt<64, X>(N, R, smem, st, set_smem);
    if (e == 0 && (set_smem || nt == 256)) e = launch_state_nt<256, X>(N, R, smem, st, set_smem);
    return e;
}

int launch_state_gm(int nt, const DevNet &N, const EvalReq &R, size_t smem, cudaStream_t st, bool set_smem);

}  // namespace exago
