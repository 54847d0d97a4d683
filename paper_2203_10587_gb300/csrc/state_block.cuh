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

// One end of branch l (lanes 2 m and 2 m + 1 of a warp hold the two ends of one branch): the end's part
// of branch_item, with the fold of the two Hessian blocks done by both lanes from each other's values.
// The same operations on the same values, so the same bits; about 70 of a branch's 110 FP64
// instructions a lane.  All 32 lanes call it (valid: the lane has a branch).
template <int WANT>
__device__ __forceinline__ void branch_end_item(const DevNet &N, const EvalReq &R, int b, int l, int end,
                                                bool valid, double *scr) {
    constexpr bool WG = WANT & W_G, WJ = WANT & W_J, WH = WANT & W_H;
    const int nb = N.nb, nl = N.nl;
    bool on = false;
    int u = 0, v = 0;
    double *rec = nullptr, *Jrow = nullptr, *h = nullptr;
    if (valid) {
        const int s = __ldg(N.br_slot + end * nl + l);
        u = __ldg((end ? N.t : N.f) + l);
        v = __ldg((end ? N.f : N.t) + l);
        valid = EXAGO_DCHECK(N, s >= 0 && s < N.chk_nslot && u >= 0 && u < nb && v >= 0 && v < nb);
        rec = scr + (size_t)s * NCOMP;
        if (WJ) Jrow = st_jval(N, R, b) + N.nnzJg + 4 * (size_t)(end * nl + l);
        if (WG && R.gh) h = st_gh(N, R, b) + 2 * nb + end * nl + l;
        const uint8_t *mk = st_mask(N, R, b);
        on = valid && (mk == nullptr || mk[l] != 0);
        if (valid && !on) {   // out of service: every value of this end is zero
            if (WG || WJ) { put2(rec, SC_PA, 0.0, 0.0); put2(rec, SC_PV, 0.0, 0.0); put2(rec, SC_QU, 0.0, 0.0); }
            if (WH) { put2(rec, SC_HAA, 0.0, 0.0); put2(rec, SC_HUU, 0.0, 0.0); }
            if (h) *h = 0.0;
            if (WJ)
                for (int k = 0; k < 4; k++) Jrow[k] = 0.0;
        }
    }
    EndHess hs{};
    double Vu = 0.0, Vv = 0.0, VV = 0.0;
    if (on) {
        const double *xb = st_x(N, R, b);
        const double au = __ldg(xb + u), av = __ldg(xb + v);
        Vu = __ldg(xb + nb + u);
        Vv = __ldg(xb + nb + v);
        const double G = __ldg(N.Gft + l), Bm = __ldg(N.Bft + l);
        const double Gss = __ldg((end ? N.Gtt : N.Gff) + l), Bss = __ldg((end ? N.Btt : N.Bff) + l);
        const double Gss2 = __ldg((end ? N.Gtt2 : N.Gff2) + l), Bss2 = __ldg((end ? N.Btt2 : N.Bff2) + l);
        double s, c, Af, Cf, At, Ct;
        branch_sincos(end ? av - au : au - av, &s, &c);   // Va_f - Va_t
        angle_terms<(WANT & W_PS) != 0>(N, l, G, Bm, s, c, &Af, &Cf, &At, &Ct);
        const double A = end ? At : Af, C = end ? Ct : Cf;
        VV = Vu * Vv;
        Mul<false> mul;
        const End e = end_terms<true>(Gss, Bss, Gss2, Bss2, A, C, Vu, Vv, Vu * Vu, VV, mul);
        if (h) *h = fma(e.P, e.P, e.Q * e.Q);
        if (WG || WJ) {
            put2(rec, SC_PA, e.pa, e.pu); put2(rec, SC_PV, e.pv, e.qa); put2(rec, SC_QU, e.qu, e.qv);
        }
        if (WJ) store_hrow(Jrow, e, u < v);
        if (WH) {
            const double *lb = st_lam(N, R, b);
            hs = end_hess(e, Gss2, Bss2, A, C, __ldg(N.Kft + l), Vu, Vv, __ldg(lb + u), __ldg(lb + nb + u),
                          __ldg(lb + 2 * nb + end * nl + l), mul);
        }
    }
    if (WH) {
        EndHess ho;   // the other end's
        ho.W1 = __shfl_xor_sync(0xffffffffu, hs.W1, 1);
        ho.W2 = __shfl_xor_sync(0xffffffffu, hs.W2, 1);
        ho.tK = __shfl_xor_sync(0xffffffffu, hs.tK, 1);
        ho.hau = 0.0;
        ho.huu = 0.0;
        ho.huv = __shfl_xor_sync(0xffffffffu, hs.huv, 1);
        if (on) {   // this end as the "from" end of branch_hess
            const BranchHess f = branch_hess(hs, ho, Vu, Vv, 0.0, Vv * Vv, VV);
            put2(rec, SC_HAA, f.haa, f.xf);
            put2(rec, SC_HUU, f.mff, f.mft);
        }
    }
}

// For few states (a block per SM at most): 512 threads a state.  PAIR (up to 64 branches, a warp for
// each of the SM's four FP64 pipes): two threads a branch; with more branches the 28% of FP64 work that
// both ends repeat costs more than the shorter chain saves (118 buses: 18.4 us against 16.4).  The bus
// phase is two independent kinds of items on different threads: a bus sums its diagonal terms and
// finishes with bus_tail; a slot (branch end) writes its neighbour's row entries; in bus_item one
// thread does a bus's slots one after another.  What bounds it: the chain through the two items, at 64
// cycles an FP64 instruction.  Against k_state (us): 30 buses x 1 14.4, 12.3; 200 buses (260 branches)
// x 100 24.6, 22.6; 300 x 152 32.8, 29.4.
template <int WANT, bool PAIR>
__global__ void __launch_bounds__(512, 1) k_state_few(const DevNet N, const EvalReq R) {
    extern __shared__ __align__(16) double s_state[];
    __shared__ double s_part[OBJ_LANES];
    constexpr bool GM = (WANT & W_GM) != 0, WJ = WANT & W_J, WH = WANT & W_H;
    const int b = blockIdx.x, tid = threadIdx.x;
    double *recs = s_state;
    if (WANT & (W_G | W_J | W_H)) {
        if (PAIR) {
            for (int i = tid; (i & ~31) < 2 * N.nl; i += 512)
                branch_end_item<WANT>(N, R, b, i >> 1, i & 1, i < 2 * N.nl, recs);
        } else {
            for (int l = tid; l < N.nl; l += 512) branch_item<WANT>(N, R, b, l, recs);
        }
    }
    if (R.f && tid < OBJ_LANES) obj_lanes<GM, OBJ_LANES>(N, R, b, 0, s_part);
    __syncthreads();
    if (R.f && tid >= 512 - 32) obj_tree_warp<true>(R, b, s_part);
    TileRows T{};
    if (WJ) T.P = T.Q = st_jval(N, R, b);
    if (WH) T.A = T.M = st_hval(N, R, b);
    const int nslots = (WJ || WH) ? N.nslot : 0;
    for (int it = tid; it < N.nb + nslots; it += 512) {
        if (it < N.nb) {
            const int i = it;
            if (WANT & (W_G | W_J | W_H)) {
                const int s0 = __ldg(N.slot_ptr + i), s1 = __ldg(N.slot_ptr + i + 1);
                if (EXAGO_DCHECK(N, s0 >= 0 && s0 <= s1 && s1 <= N.chk_nslot)) {
                    Rec D{};
                    for (int s = s0; s < s1; s++) {
                        const Rec r = load_rec<WANT, true>(recs + (size_t)s * NCOMP);
                        if (s == s0) D = r;
                        else add_diag<WANT>(D, r);
                    }
                    bus_tail<WANT>(N, R, b, i, D, T.template of<WANT>(N, i));
                }
            }
            if (R.grad) grad_bus<GM>(N, R, b, i);
        } else {
            slot_rows<WANT, true>(N, it - N.nb, recs, T);
        }
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
static int launch_few_x(const DevNet &N, const EvalReq &R, size_t smem, cudaStream_t st, bool set_smem) {
    const int want = (R.gh ? W_G : 0) | (R.jval ? W_J : 0) | (R.hval ? W_H : 0);
    const bool pair = N.nl <= 64;
    int e = 0;
    auto go = [&](auto kern, int w, bool p) {
        if (e != 0) return;
        if (set_smem) {
            e = (int)cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kStateMaxBytes);
        } else if (w == want && p == pair) {
            kern<<<R.B, 512, smem, st>>>(N, R);
            e = (int)cudaGetLastError();
        }
    };
    go(k_state_few<X, false>, 0, pair);
    go(k_state_few<1 | X, false>, 1, false); go(k_state_few<1 | X, true>, 1, true);
    go(k_state_few<2 | X, false>, 2, false); go(k_state_few<2 | X, true>, 2, true);
    go(k_state_few<3 | X, false>, 3, false); go(k_state_few<3 | X, true>, 3, true);
    go(k_state_few<4 | X, false>, 4, false); go(k_state_few<4 | X, true>, 4, true);
    go(k_state_few<5 | X, false>, 5, false); go(k_state_few<5 | X, true>, 5, true);
    go(k_state_few<6 | X, false>, 6, false); go(k_state_few<6 | X, true>, 6, true);
    go(k_state_few<7 | X, false>, 7, false); go(k_state_few<7 | X, true>, 7, true);
    return e;
}

template <int X>
static int launch_state_x(int nt, const DevNet &N, const EvalReq &R, size_t smem, cudaStream_t st, bool set_smem) {
    int e = 0;
    if (set_smem || nt == 512) e = launch_few_x<X>(N, R, smem, st, set_smem);
    if (e == 0 && (set_smem || nt == 64)) e = launch_state_nt<64, X>(N, R, smem, st, set_smem);
    if (e == 0 && (set_smem || nt == 256)) e = launch_state_nt<256, X>(N, R, smem, st, set_smem);
    return e;
}

int launch_state_gm(int nt, const DevNet &N, const EvalReq &R, size_t smem, cudaStream_t st, bool set_smem);

}  // namespace exago
