// Batched numeric block factorisation and solve (blockfact.h).  The columns below k0 go level by
// level of the elimination tree, one thread per (state, target block) or a few (below); the last
// ones, the dense tail, get their updates by those columns here and are then factored as one
// matrix per state (densetail.h), which holds most of the work of a large grid.
//
// Factor, per level: every target (I, J) of the level's columns accumulates its left-looking
// update T_IJ = A_IJ - sum_K F_IK U_KJ (SYM: U_KJ = L_JK') in registers, in the pair order the
// host fixed (ascending K), and stores it (a fill block starts from zero, unread);
// the diagonal target also inverts its column's pivot block D_J = T_JJ, by Gauss-Jordan
// elimination without pivoting, into the diagonal position of L; then every other target is
// scaled by that inverse (L_IJ = T_IJ D_J^-1; LU: U_JI = D_J^-1 T'_JI).  Solve: forward y_J = r_J
// - sum_K F_JK z_K, z_J = D_J^-1 y_J over ascending levels (F = L D is what the factor kept in T),
// then backward x_J = z_J - sum_I U_JI x_I over descending levels, the tail's sweeps between.
// A warp holds 32 consecutive states of one target, so every value load is one coalesced
// 256-byte access and every index load is uniform across the warp.
#include <cuda_runtime.h>

#include "blockfact.h"
#include "densetail.h"
#include "internal.h"

namespace exago {

namespace {

constexpr int kNT = 128;   // states per block

template <int BS>
__device__ __forceinline__ void load_blk(const double *A, int64_t p, int B, int b, double *v) {
    constexpr int BB = BS * BS;
    const double *a = A + (size_t)p * BB * B + b;
#pragma unroll
    for (int e = 0; e < BB; e++) v[e] = __ldg(a + (size_t)e * B);
}

template <int BS>
__device__ __forceinline__ void load_blk_cg(const double *A, int64_t p, int B, int b, double *v) {
    // values written earlier in the same factorisation by other blocks: through L2
    constexpr int BB = BS * BS;
    const double *a = A + (size_t)p * BB * B + b;
#pragma unroll
    for (int e = 0; e < BB; e++) v[e] = __ldcg(a + (size_t)e * B);
}

template <int BS>
__device__ __forceinline__ void store_blk(double *A, int64_t p, int B, int b, const double *v) {
    constexpr int BB = BS * BS;
    double *a = A + (size_t)p * BB * B + b;
#pragma unroll
    for (int e = 0; e < BB; e++) a[(size_t)e * B] = v[e];
}

// acc -= X Y  (X, Y, acc BS x BS row-major), or acc -= X Y' with TY.
template <int BS, bool TY>
__device__ __forceinline__ void sub_mul(double *acc, const double *X, const double *Y) {
#pragma unroll
    for (int i = 0; i < BS; i++)
#pragma unroll
        for (int j = 0; j < BS; j++) {
            double s = acc[i * BS + j];
#pragma unroll
            for (int k = 0; k < BS; k++) s = fma(-X[i * BS + k], TY ? Y[j * BS + k] : Y[k * BS + j], s);
            acc[i * BS + j] = s;
        }
}

// out = X Y
template <int BS>
__device__ __forceinline__ void mul(const double *X, const double *Y, double *out) {
#pragma unroll
    for (int i = 0; i < BS; i++)
#pragma unroll
        for (int j = 0; j < BS; j++) {
            double s = X[i * BS] * Y[j];
#pragma unroll
            for (int k = 1; k < BS; k++) s = fma(X[i * BS + k], Y[k * BS + j], s);
            out[i * BS + j] = s;
        }
}

// Inverse of the pivot block by Gauss-Jordan elimination without pivoting.  neg: pivots below
// zero (for a symmetric block, its negative eigenvalues: the pivots are the D of its LDL');
// bad: pivots with |d| <= tiny * max |entry| (the block is numerically singular).
template <int BS>
__device__ __forceinline__ void invert(const double *D, double *inv, int *neg, int *bad, double tiny) {
    double a[BS][2 * BS];
    double amax = 0.0;
#pragma unroll
    for (int i = 0; i < BS; i++)
#pragma unroll
        for (int j = 0; j < BS; j++) {
            a[i][j] = D[i * BS + j];
            a[i][BS + j] = i == j ? 1.0 : 0.0;
            amax = fmax(amax, fabs(D[i * BS + j]));
        }
    int nneg = 0, nbad = 0;
#pragma unroll
    for (int k = 0; k < BS; k++) {
        const double piv = a[k][k];
        nneg += piv < 0.0;
        nbad += !(fabs(piv) > tiny * amax);
        const double r = 1.0 / piv;
#pragma unroll
        for (int j = 0; j < 2 * BS; j++) a[k][j] *= r;
#pragma unroll
        for (int i = 0; i < BS; i++) {
            if (i == k) continue;
            const double f = a[i][k];
#pragma unroll
            for (int j = 0; j < 2 * BS; j++) a[i][j] = fma(-f, a[k][j], a[i][j]);
        }
    }
#pragma unroll
    for (int i = 0; i < BS; i++)
#pragma unroll
        for (int j = 0; j < BS; j++) inv[i * BS + j] = a[i][BS + j];
    *neg = nneg;
    *bad = nbad;
}

// A column's pivot block D is final: its inverse goes to the diagonal position of L, and its
// negative and near-zero pivots are counted.
template <int BS>
__device__ __forceinline__ void finish_pivot(double *L, int p, int B, int b, const double *D, int *neg,
                                             int *bad, double tiny) {
    double Di[BS * BS];
    int nn, nbad;
    invert<BS>(D, Di, &nn, &nbad, tiny);
    store_blk<BS>(L, p, B, b, Di);
    if (nn) atomicAdd(neg + b, nn);
    if (nbad) atomicAdd(bad + b, nbad);
}

// Update phase of one level: targets [t0, t0 + gridDim.x); the diagonal ones also invert their
// pivot block.
template <int BS, bool SYM>
__global__ void __launch_bounds__(kNT) k_bf_update(const DevSymK S, int B, double *T, double *TU,
                                                   double *L, const double *U, int *neg, int *bad,
                                                   double tiny, int t0) {
    constexpr int BB = BS * BS;
    const int b = blockIdx.y * kNT + threadIdx.x;
    if (b >= B) return;
    const int t = t0 + blockIdx.x;
    const int p = __ldg(S.tgt_blk + t);
    const bool diag = p == __ldg(S.tgt_diag + t);
    const int64_t q0 = __ldg(S.tptr + t), q1 = __ldg(S.tptr + t + 1);
    if (q0 == q1 && !diag) return;   // nothing to subtract: T already holds A_IJ
    double acc[BB], accU[BB];
    if (__ldg(S.tgt_fill + t)) {   // A_IJ = 0, not assembled
#pragma unroll
        for (int e = 0; e < BB; e++) { acc[e] = 0.0; accU[e] = 0.0; }
    } else {
        load_blk_cg<BS>(T, p, B, b, acc);
        if (!SYM && !diag) load_blk_cg<BS>(TU, p, B, b, accU);
    }
    for (int64_t q = q0; q < q1; q++) {
        const int2 pr = __ldg(S.pairs + q);   // (I, K), (J, K)
        if (!EXAGO_DCHECK(S, pr.x >= 0 && pr.x < S.nblk && pr.y >= 0 && pr.y < S.nblk)) continue;
        double X[BB], Y[BB];
        load_blk_cg<BS>(T, pr.x, B, b, X);                      // F_IK
        if (SYM) {
            load_blk_cg<BS>(L, pr.y, B, b, Y);                  // L_JK
            sub_mul<BS, true>(acc, X, Y);
        } else {
            load_blk_cg<BS>(U, pr.y, B, b, Y);                  // U_KJ
            sub_mul<BS, false>(acc, X, Y);
            if (!diag) {
                load_blk_cg<BS>(T, pr.y, B, b, X);              // F_JK
                load_blk_cg<BS>(U, pr.x, B, b, Y);              // U_KI
                sub_mul<BS, false>(accU, X, Y);
            }
        }
    }
    if (q0 != q1) store_blk<BS>(T, p, B, b, acc);
    if (!SYM && !diag) store_blk<BS>(TU, p, B, b, accU);
    if (diag) finish_pivot<BS>(L, p, B, b, acc, neg, bad, tiny);
}

// Scale phase of one level.  (Every target used to invert its column's pivot block for itself: 150
// FP64 instructions beside the 64 of its product; 2,000 buses x 512: 1.2 ms of the factorisation.)
template <int BS, bool SYM>
__global__ void __launch_bounds__(kNT) k_bf_scale(const DevSymK S, int B, const double *T,
                                                  const double *TU, double *L, double *U, int t0) {
    constexpr int BB = BS * BS;
    const int b = blockIdx.y * kNT + threadIdx.x;
    if (b >= B) return;
    const int t = t0 + blockIdx.x;
    const int p = __ldg(S.tgt_blk + t), pd = __ldg(S.tgt_diag + t);
    if (p == pd) return;
    double Di[BB], X[BB], Y[BB];
    load_blk_cg<BS>(L, pd, B, b, Di);
    load_blk_cg<BS>(T, p, B, b, X);
    mul<BS>(X, Di, Y);                                          // L_IJ = T_IJ D_J^-1
    store_blk<BS>(L, p, B, b, Y);
    if (!SYM) {
        load_blk_cg<BS>(TU, p, B, b, X);
        mul<BS>(Di, X, Y);                                      // U_JI = D_J^-1 T'_JI
        store_blk<BS>(U, p, B, b, Y);
    }
}

// ---- small batches: a block's rows on different warps (threads 32 states x BS rows), so that a
// block product is 16 dependent-free multiply-adds a warp in place of 64 (an FP64 instruction holds
// its pipe for 64 cycles whatever the lanes).  Every element's sum is the same, so results do not
// depend on the choice.
constexpr int kRowsBelow = 129;   // states

// acc[j] (row r of target t) less its pairs up to q1; accU likewise for the upper block (LU).
template <int BS, bool SYM>
__device__ __forceinline__ void row_sums(const DevSymK &S, int B, int b, int r, int64_t q0, int64_t q1,
                                         const double *T, const double *L, const double *U, bool upper,
                                         double *acc, double *accU) {
    constexpr int BB = BS * BS;
    auto row = [&](const double *A, int64_t p, double *v) {
#pragma unroll
        for (int k = 0; k < BS; k++) v[k] = __ldcg(A + ((size_t)p * BB + r * BS + k) * B + b);
    };
    for (int64_t q = q0; q < q1; q++) {
        const int2 pr = __ldg(S.pairs + q);
        if (!EXAGO_DCHECK(S, pr.x >= 0 && pr.x < S.nblk && pr.y >= 0 && pr.y < S.nblk)) continue;
        double X[BS], Y[BB];
        row(T, pr.x, X);
        load_blk_cg<BS>(SYM ? L : U, pr.y, B, b, Y);
#pragma unroll
        for (int j = 0; j < BS; j++)
#pragma unroll
            for (int k = 0; k < BS; k++) acc[j] = fma(-X[k], SYM ? Y[j * BS + k] : Y[k * BS + j], acc[j]);
        if (!SYM && upper) {
            row(T, pr.y, X);
            load_blk_cg<BS>(U, pr.x, B, b, Y);
#pragma unroll
            for (int j = 0; j < BS; j++)
#pragma unroll
                for (int k = 0; k < BS; k++) accU[j] = fma(-X[k], Y[k * BS + j], accU[j]);
        }
    }
}

// Row r of target t's own block (zero for a fill block).
template <int BS>
__device__ __forceinline__ void own_row(const DevSymK &S, const double *A, int t, int p, int B, int b, int r,
                                        double *v) {
    const bool fill = __ldg(S.tgt_fill + t);
#pragma unroll
    for (int k = 0; k < BS; k++)
        v[k] = fill ? 0.0 : __ldcg(A + ((size_t)p * BS * BS + r * BS + k) * B + b);
}

template <int BS, bool SYM>
__global__ void __launch_bounds__(32 * BS) k_bf_update_rows(const DevSymK S, int B, double *T, double *TU,
                                                            double *L, const double *U, int *neg,
                                                            int *bad, double tiny, int t0) {
    __shared__ double s_d[BS * BS][32];
    const int lane = threadIdx.x, r = threadIdx.y, b = blockIdx.y * 32 + lane;
    const bool live = b < B;
    const int t = t0 + blockIdx.x, p = __ldg(S.tgt_blk + t);
    const bool diag = p == __ldg(S.tgt_diag + t);
    const int64_t q0 = __ldg(S.tptr + t), q1 = __ldg(S.tptr + t + 1);
    if (q0 == q1 && !diag) return;
    double acc[BS], accU[BS];
    if (live) {
        own_row<BS>(S, T, t, p, B, b, r, acc);
        if (!SYM && !diag) own_row<BS>(S, TU, t, p, B, b, r, accU);
        row_sums<BS, SYM>(S, B, b, r, q0, q1, T, L, U, !diag, acc, accU);
#pragma unroll
        for (int k = 0; k < BS; k++) {
            if (q0 != q1) T[((size_t)p * BS * BS + r * BS + k) * B + b] = acc[k];
            if (!SYM && !diag) TU[((size_t)p * BS * BS + r * BS + k) * B + b] = accU[k];
            if (diag) s_d[r * BS + k][lane] = acc[k];
        }
    }
    if (!diag) return;   // uniform over the block
    __syncthreads();
    if (r != 0 || !live) return;
    double D[BS * BS];
#pragma unroll
    for (int e = 0; e < BS * BS; e++) D[e] = s_d[e][lane];
    finish_pivot<BS>(L, p, B, b, D, neg, bad, tiny);
}

// ---- split variants: the terms of one target (or one column's sweep) divided among kSlices warps of
// a block that holds 32 states; slice w takes every kSlices-th term from the w-th, and the slices'
// partial sums are added in slice order, an entry or two per warp (one warp alone would be at it
// longer than at its terms: an FP64 instruction holds its pipe for 64 cycles).  Used where a level
// has few targets and long sums, so that these are not one thread's latency chain.  The split is
// fixed by the structure alone (never by the batch size), so every state's result is the same
// whatever the batch it belongs to (on one side of BlockSym::tail_most).
constexpr int kSlices = 8;

template <int BS, bool SYM>
__global__ void __launch_bounds__(32 * kSlices) k_bf_update_split(const DevSymK S, int B, double *T,
                                                                  double *TU, double *L,
                                                                  const double *U, int *neg, int *bad,
                                                                  double tiny, int t0) {
    constexpr int BB = BS * BS, NP = SYM ? BB : 2 * BB;   // partial sums: lower (and upper)
    __shared__ double part[kSlices][NP][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int b = blockIdx.y * 32 + lane;
    const bool live = b < B;
    const int t = t0 + blockIdx.x;
    const int p = __ldg(S.tgt_blk + t);
    const bool diag = p == __ldg(S.tgt_diag + t);
    const int64_t q0 = __ldg(S.tptr + t), q1 = __ldg(S.tptr + t + 1);
    if (q0 == q1 && !diag) return;   // uniform over the block
    double acc[BB], accU[BB];
#pragma unroll
    for (int e = 0; e < BB; e++) { acc[e] = 0.0; accU[e] = 0.0; }
    if (live)
        for (int64_t q = q0 + w; q < q1; q += kSlices) {
            const int2 pr = __ldg(S.pairs + q);
            if (!EXAGO_DCHECK(S, pr.x >= 0 && pr.x < S.nblk && pr.y >= 0 && pr.y < S.nblk)) continue;
            double X[BB], Y[BB];
            load_blk_cg<BS>(T, pr.x, B, b, X);
            if (SYM) {
                load_blk_cg<BS>(L, pr.y, B, b, Y);
                sub_mul<BS, true>(acc, X, Y);
            } else {
                load_blk_cg<BS>(U, pr.y, B, b, Y);
                sub_mul<BS, false>(acc, X, Y);
                if (!diag) {
                    load_blk_cg<BS>(T, pr.y, B, b, X);
                    load_blk_cg<BS>(U, pr.x, B, b, Y);
                    sub_mul<BS, false>(accU, X, Y);
                }
            }
        }
#pragma unroll
    for (int e = 0; e < BB; e++) {
        part[w][e][lane] = acc[e];
        if (!SYM) part[w][(NP - BB) + e][lane] = accU[e];
    }
    __syncthreads();
    for (int e = w; e < NP; e += kSlices) {
        double s = part[0][e][lane];
#pragma unroll
        for (int v = 1; v < kSlices; v++) s += part[v][e][lane];
        part[0][e][lane] = s;   // entry e is this warp's alone
    }
    __syncthreads();
    if (w != 0 || !live) return;
    if (__ldg(S.tgt_fill + t)) {
#pragma unroll
        for (int e = 0; e < BB; e++) { acc[e] = 0.0; accU[e] = 0.0; }
    } else {
        load_blk_cg<BS>(T, p, B, b, acc);
        if (!SYM && !diag) load_blk_cg<BS>(TU, p, B, b, accU);
    }
#pragma unroll
    for (int e = 0; e < BB; e++) {
        acc[e] += part[0][e][lane];
        if (!SYM) accU[e] += part[0][(NP - BB) + e][lane];
    }
    if (q0 != q1) store_blk<BS>(T, p, B, b, acc);
    if (!SYM && !diag) store_blk<BS>(TU, p, B, b, accU);
    if (diag) finish_pivot<BS>(L, p, B, b, acc, neg, bad, tiny);
}

// Forward sweep of one level's columns, split: y_J = r_J + (the slices' sums of -F_JK z_K);
// z_J = D_J^-1 y_J.
template <int BS>
__global__ void __launch_bounds__(32 * kSlices) k_bf_forward_split(const DevSymK S, int B,
                                                                   const double *T,
                                                                   const double *L, double *x,
                                                                   int c0) {
    __shared__ double part[kSlices][BS][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int b = blockIdx.y * 32 + lane;
    const bool live = b < B;
    const int J = __ldg(S.lvl_cols + c0 + blockIdx.x);
    double y[BS];
#pragma unroll
    for (int i = 0; i < BS; i++) y[i] = 0.0;
    const int64_t r0 = __ldg(S.rowptr + J), r1 = __ldg(S.rowptr + J + 1);
    if (live)
        for (int64_t r = r0 + w; r < r1; r += kSlices) {
            const int K = __ldg(S.rowcol + r), p = __ldg(S.rowblk + r);
            if (!EXAGO_DCHECK(S, K >= 0 && K < S.nb && p >= 0 && p < S.nblk)) continue;
            double F[BS * BS], z[BS];
            load_blk<BS>(T, p, B, b, F);
#pragma unroll
            for (int i = 0; i < BS; i++) z[i] = __ldcg(x + ((size_t)K * BS + i) * B + b);
#pragma unroll
            for (int i = 0; i < BS; i++)
#pragma unroll
                for (int k = 0; k < BS; k++) y[i] = fma(-F[i * BS + k], z[k], y[i]);
        }
#pragma unroll
    for (int i = 0; i < BS; i++) part[w][i][lane] = y[i];
    __syncthreads();
    if (w < BS && live) {
        double s = part[0][w][lane];
#pragma unroll
        for (int v = 1; v < kSlices; v++) s += part[v][w][lane];
        part[0][w][lane] = __ldcg(x + ((size_t)J * BS + w) * B + b) + s;
    }
    __syncthreads();
    if (w != 0 || !live) return;
#pragma unroll
    for (int i = 0; i < BS; i++) y[i] = part[0][i][lane];
    double Di[BS * BS];
    load_blk<BS>(L, __ldg(S.colptr + J), B, b, Di);
#pragma unroll
    for (int i = 0; i < BS; i++) {
        double s = Di[i * BS] * y[0];
#pragma unroll
        for (int k = 1; k < BS; k++) s = fma(Di[i * BS + k], y[k], s);
        x[((size_t)J * BS + i) * B + b] = s;
    }
}

// Backward sweep of one level's columns, split: x_J = z_J + (the slices' sums of -U_JI x_I).
template <int BS, bool SYM>
__global__ void __launch_bounds__(32 * kSlices) k_bf_backward_split(const DevSymK S, int B,
                                                                    const double *L,
                                                                    const double *U, double *x,
                                                                    int c0) {
    __shared__ double part[kSlices][BS][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int b = blockIdx.y * 32 + lane;
    const bool live = b < B;
    const int J = __ldg(S.lvl_cols + c0 + blockIdx.x);
    double v[BS];
#pragma unroll
    for (int i = 0; i < BS; i++) v[i] = 0.0;
    const int64_t p0 = __ldg(S.colptr + J), p1 = __ldg(S.colptr + J + 1);
    if (live)
        for (int64_t p = p0 + 1 + w; p < p1; p += kSlices) {
            const int I = __ldg(S.rowidx + p);
            if (!EXAGO_DCHECK(S, I >= 0 && I < S.nb)) continue;
            double M[BS * BS], xi[BS];
            load_blk<BS>(SYM ? L : U, p, B, b, M);
#pragma unroll
            for (int i = 0; i < BS; i++) xi[i] = __ldcg(x + ((size_t)I * BS + i) * B + b);
#pragma unroll
            for (int i = 0; i < BS; i++)
#pragma unroll
                for (int k = 0; k < BS; k++)
                    v[i] = fma(-(SYM ? M[k * BS + i] : M[i * BS + k]), xi[k], v[i]);
        }
#pragma unroll
    for (int i = 0; i < BS; i++) part[w][i][lane] = v[i];
    __syncthreads();
    if (w >= BS || !live) return;
    double s = part[0][w][lane];
#pragma unroll
    for (int u = 1; u < kSlices; u++) s += part[u][w][lane];
    x[((size_t)J * BS + w) * B + b] = __ldcg(x + ((size_t)J * BS + w) * B + b) + s;
}

// Forward sweep of one level's columns: y_J = r_J - sum_K F_JK z_K; z_J = D_J^-1 y_J.
template <int BS>
__global__ void __launch_bounds__(kNT) k_bf_forward(const DevSymK S, int B, const double *T,
                                                    const double *L, double *x, int c0) {
    const int b = blockIdx.y * kNT + threadIdx.x;
    if (b >= B) return;
    const int J = __ldg(S.lvl_cols + c0 + blockIdx.x);
    double y[BS];
#pragma unroll
    for (int i = 0; i < BS; i++) y[i] = __ldcg(x + ((size_t)J * BS + i) * B + b);
    const int64_t r0 = __ldg(S.rowptr + J), r1 = __ldg(S.rowptr + J + 1);
    for (int64_t r = r0; r < r1; r++) {
        const int K = __ldg(S.rowcol + r), p = __ldg(S.rowblk + r);
        if (!EXAGO_DCHECK(S, K >= 0 && K < S.nb && p >= 0 && p < S.nblk)) continue;
        double F[BS * BS], z[BS];
        load_blk<BS>(T, p, B, b, F);
#pragma unroll
        for (int i = 0; i < BS; i++) z[i] = __ldcg(x + ((size_t)K * BS + i) * B + b);
#pragma unroll
        for (int i = 0; i < BS; i++)
#pragma unroll
            for (int k = 0; k < BS; k++) y[i] = fma(-F[i * BS + k], z[k], y[i]);
    }
    double Di[BS * BS];
    load_blk<BS>(L, __ldg(S.colptr + J), B, b, Di);
#pragma unroll
    for (int i = 0; i < BS; i++) {
        double s = Di[i * BS] * y[0];
#pragma unroll
        for (int k = 1; k < BS; k++) s = fma(Di[i * BS + k], y[k], s);
        x[((size_t)J * BS + i) * B + b] = s;
    }
}

// Backward sweep of one level's columns: x_J = z_J - sum_{I in colstruct(J)} U_JI x_I
// (SYM: U_JI = L_IJ').
template <int BS, bool SYM>
__global__ void __launch_bounds__(kNT) k_bf_backward(const DevSymK S, int B, const double *L,
                                                     const double *U, double *x, int c0) {
    const int b = blockIdx.y * kNT + threadIdx.x;
    if (b >= B) return;
    const int J = __ldg(S.lvl_cols + c0 + blockIdx.x);
    double v[BS];
#pragma unroll
    for (int i = 0; i < BS; i++) v[i] = __ldcg(x + ((size_t)J * BS + i) * B + b);
    const int64_t p0 = __ldg(S.colptr + J), p1 = __ldg(S.colptr + J + 1);
    for (int64_t p = p0 + 1; p < p1; p++) {
        const int I = __ldg(S.rowidx + p);
        if (!EXAGO_DCHECK(S, I >= 0 && I < S.nb)) continue;
        double M[BS * BS], xi[BS];
        load_blk<BS>(SYM ? L : U, p, B, b, M);
#pragma unroll
        for (int i = 0; i < BS; i++) xi[i] = __ldcg(x + ((size_t)I * BS + i) * B + b);
#pragma unroll
        for (int i = 0; i < BS; i++)
#pragma unroll
            for (int k = 0; k < BS; k++)
                v[i] = fma(-(SYM ? M[k * BS + i] : M[i * BS + k]), xi[k], v[i]);
    }
#pragma unroll
    for (int i = 0; i < BS; i++) x[((size_t)J * BS + i) * B + b] = v[i];
}

// (i, j), j <= i, of e = i (i + 1) / 2 + j.
__device__ __forceinline__ void lower_pair(int e, int *pi, int *pj) {
    int i = (int)((sqrtf(8.0f * (float)e + 1.0f) - 1.0f) * 0.5f);
    while (i * (i + 1) / 2 > e) i--;
    while ((i + 1) * (i + 2) / 2 <= e) i++;
    *pi = i;
    *pj = e - i * (i + 1) / 2;
}

// BS values v[0], v[step], .. to consecutive, aligned doubles.
template <int BS>
__device__ __forceinline__ void store_col(double *p, const double *v, int step) {
    if constexpr (BS == 4)
        asm volatile("st.global.v4.f64 [%0], {%1, %2, %3, %4};" ::"l"(p), "d"(v[0]), "d"(v[step]),
                     "d"(v[2 * step]), "d"(v[3 * step])
                     : "memory");
    else
        *reinterpret_cast<double2 *>(p) = make_double2(v[0], v[step]);
}

// The tail's panels from the assembled blocks: T_IJ = A_IJ - sum over the columns K < k0 of
// F_IK U_KJ, one thread per (state, lower block of the tail), written where densetail.h keeps it
// (LU: the upper block, transposed, into V; inside a 64-column panel's own square also in place).
template <int BS, bool SYM>
__global__ void __launch_bounds__(kNT) k_bf_tail(const DevSymK S, int B, const double *T,
                                                 const double *TU, const double *L,
                                                 const double *U, double *D, double *V,
                                                 size_t dstride) {
    constexpr int BB = BS * BS;
    const int b = blockIdx.y * kNT + threadIdx.x;
    if (b >= B) return;
    const int e = blockIdx.x;
    int i, j;
    lower_pair(e, &i, &j);
    double acc[BB], accU[BB];
#pragma unroll
    for (int k = 0; k < BB; k++) { acc[k] = 0.0; accU[k] = 0.0; }
    const int t = __ldg(S.tail_tgt + e);
    if (t >= 0) {
        const int p = __ldg(S.tgt_blk + t);
        if (!__ldg(S.tgt_fill + t)) {
            load_blk_cg<BS>(T, p, B, b, acc);
            if (!SYM) load_blk_cg<BS>(TU, p, B, b, accU);
        }
        for (int64_t q = __ldg(S.tptr + t), q1 = __ldg(S.tail_q1 + t); q < q1; q++) {
            const int2 pr = __ldg(S.pairs + q);
            if (!EXAGO_DCHECK(S, pr.x >= 0 && pr.x < S.nblk && pr.y >= 0 && pr.y < S.nblk)) continue;
            double X[BB], Y[BB];
            load_blk_cg<BS>(T, pr.x, B, b, X);
            load_blk_cg<BS>(SYM ? L : U, pr.y, B, b, Y);
            sub_mul<BS, SYM>(acc, X, Y);
            if (!SYM && i != j) {
                load_blk_cg<BS>(T, pr.y, B, b, X);
                load_blk_cg<BS>(U, pr.x, B, b, Y);
                sub_mul<BS, false>(accU, X, Y);
            }
        }
    }
    const int n = S.tail_n, r0 = BS * i, c0 = BS * j;
    double *Db = D + (size_t)b * dstride, *Vb = SYM ? nullptr : V + (size_t)b * dstride;
    // a block's column is BS consecutive rows, aligned (r0 and the panels' heights are multiples of
    // BS): one store of a whole 16- or 32-byte piece, since the lanes' states lie apart
#pragma unroll
    for (int c = 0; c < BS; c++) {
        store_col<BS>(Db + tail_pos(n, r0, c0 + c), acc + c, BS);
        if (SYM || i == j) continue;
        if ((r0 >> 6) == (c0 >> 6))   // row c of U_JI's block is column r of the transpose
            store_col<BS>(Db + tail_pos(n, c0, r0 + c), accU + c, BS);
        else
            store_col<BS>(Vb + tail_pos(n, r0, c0 + c), accU + c * BS, 1);
    }
}

// k_bf_tail for small batches (k_bf_update_rows says why).
template <int BS, bool SYM>
__global__ void __launch_bounds__(32 * BS) k_bf_tail_rows(const DevSymK S, int B, const double *T,
                                                          const double *TU, const double *L,
                                                          const double *U, double *D, double *V,
                                                          size_t dstride) {
    const int r = threadIdx.y, b = blockIdx.y * 32 + threadIdx.x;
    if (b >= B) return;
    int i, j;
    lower_pair(blockIdx.x, &i, &j);
    double acc[BS], accU[BS];
#pragma unroll
    for (int k = 0; k < BS; k++) { acc[k] = 0.0; accU[k] = 0.0; }
    const int t = __ldg(S.tail_tgt + blockIdx.x);
    if (t >= 0) {
        const int p = __ldg(S.tgt_blk + t);
        own_row<BS>(S, T, t, p, B, b, r, acc);
        if (!SYM) own_row<BS>(S, TU, t, p, B, b, r, accU);
        row_sums<BS, SYM>(S, B, b, r, __ldg(S.tptr + t), __ldg(S.tail_q1 + t), T, L, U, i != j, acc, accU);
    }
    const int n = S.tail_n, r0 = BS * i, c0 = BS * j;
    double *Db = D + (size_t)b * dstride, *Vb = SYM ? nullptr : V + (size_t)b * dstride;
#pragma unroll
    for (int c = 0; c < BS; c++) Db[tail_pos(n, r0 + r, c0 + c)] = acc[c];
    if (SYM || i == j) return;
    if ((r0 >> 6) == (c0 >> 6)) {
#pragma unroll
        for (int c = 0; c < BS; c++) Db[tail_pos(n, c0 + r, r0 + c)] = accU[c];
    } else {
        store_col<BS>(Vb + tail_pos(n, r0, c0 + r), accU, 1);
    }
}

// Identity in the rows that pad the tail to a multiple of 64: one thread per entry and state.
__global__ void __launch_bounds__(kNT) k_bf_tail_pad(int n, int nreal, double *D, double *V,
                                                     size_t dstride) {
    const int e = blockIdx.x * kNT + threadIdx.x;
    if (e >= (n - nreal) * n) return;
    const int row = nreal + e % (n - nreal), col = e / (n - nreal);
    const size_t b = blockIdx.y;
    if (row >= (col & ~63)) {
        D[b * dstride + tail_pos(n, row, col)] = row == col ? 1.0 : 0.0;
        if (V) V[b * dstride + tail_pos(n, row, col)] = 0.0;
    }
    // LU: the padding columns of a panel's own square, above the padding rows
    if (V && (row >> 6) == (col >> 6) && col < nreal) D[b * dstride + tail_pos(n, col, row)] = 0.0;
}

// Right-hand side of the tail: r_J - sum over K < k0 of F_JK z_K, one block of kSlices warps per (32
// states, column), the slices' sums added in slice order.
template <int BS>
__global__ void __launch_bounds__(32 * kSlices) k_bf_tail_rhs(const DevSymK S, int B, const double *T,
                                                              double *x) {
    __shared__ double part[kSlices][BS][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, b = blockIdx.y * 32 + lane;
    const bool live = b < B;
    const int J = S.k0 + blockIdx.x;
    double y[BS];
#pragma unroll
    for (int i = 0; i < BS; i++) y[i] = 0.0;
    if (live)
        for (int64_t r = __ldg(S.rowptr + J) + w, r1 = __ldg(S.tail_r1 + J); r < r1; r += kSlices) {
            const int K = __ldg(S.rowcol + r), p = __ldg(S.rowblk + r);
            if (!EXAGO_DCHECK(S, K >= 0 && K < S.nb && p >= 0 && p < S.nblk)) continue;
            double F[BS * BS], z[BS];
            load_blk<BS>(T, p, B, b, F);
#pragma unroll
            for (int i = 0; i < BS; i++) z[i] = __ldcg(x + ((size_t)K * BS + i) * B + b);
#pragma unroll
            for (int i = 0; i < BS; i++)
#pragma unroll
                for (int k = 0; k < BS; k++) y[i] = fma(-F[i * BS + k], z[k], y[i]);
        }
#pragma unroll
    for (int i = 0; i < BS; i++) part[w][i][lane] = y[i];
    __syncthreads();
    if (w >= BS || !live) return;
    double s = part[0][w][lane];
#pragma unroll
    for (int v = 1; v < kSlices; v++) s += part[v][w][lane];
    x[((size_t)J * BS + w) * B + b] = __ldcg(x + ((size_t)J * BS + w) * B + b) + s;
}

}  // namespace

// A level is split when it has fewer than kSplitBelow targets (factor) or columns (sweeps) and a sum of
// more than kSplitTerms terms: properties of the structure, not of the batch.  Levels of short sums
// were split too: 200 buses x 37 states spent 200 us in 12 sweep launches of a few terms each.
constexpr int kSplitBelow = 64, kSplitTerms = 2;

template <int BS, bool SYM>
int launch_block_factor(const DevSym &S, int B, double *T, double *TU, double *L, double *U,
                        int *neg, int *bad, double tiny, void *tail, cudaStream_t st) {
    if (B <= 0) return 0;
    const unsigned gy = (unsigned)((B + kNT - 1) / kNT), gy32 = (unsigned)((B + 31) / 32);
    for (int l = 0; l < S.nlevels; l++) {
        const int t0 = S.lvl_tptr[l], nt = S.sp_tgts[l];
        if (nt <= 0) continue;
        const dim3 grid((unsigned)nt, gy);
        if (nt < kSplitBelow && S.sp_pairs[l] > kSplitTerms)
            k_bf_update_split<BS, SYM><<<dim3((unsigned)nt, gy32), 32 * kSlices, 0, st>>>(
                S.k, B, T, TU, L, U, neg, bad, tiny, t0);
        else if (B < kRowsBelow)
            k_bf_update_rows<BS, SYM><<<dim3((unsigned)nt, gy32), dim3(32, BS), 0, st>>>(
                S.k, B, T, TU, L, U, neg, bad, tiny, t0);
        else
            k_bf_update<BS, SYM><<<grid, kNT, 0, st>>>(S.k, B, T, TU, L, U, neg, bad, tiny, t0);
        if (nt > S.sp_cols[l])   // blocks below a diagonal
            k_bf_scale<BS, SYM><<<grid, kNT, 0, st>>>(S.k, B, T, TU, L, U, t0);
    }
    if (S.k.tail_n > 0) {
        const int n = S.k.tail_n, R = S.k.nb - S.k.k0, nreal = R * BS;
        const TailShape ts = tail_shape(n, B, SYM);
        double *D = (double *)((char *)tail + ts.dn);
        double *V = SYM ? nullptr : (double *)((char *)tail + ts.dv);
        const unsigned blocks = (unsigned)(R * (R + 1) / 2);
        if (B < kRowsBelow)
            k_bf_tail_rows<BS, SYM><<<dim3(blocks, gy32), dim3(32, BS), 0, st>>>(
                S.k, B, T, TU, L, U, D, V, ts.dense_doubles);
        else
            k_bf_tail<BS, SYM><<<dim3(blocks, gy), kNT, 0, st>>>(S.k, B, T, TU, L, U, D, V,
                                                                 ts.dense_doubles);
        for (int b0 = 0; n > nreal && b0 < B; b0 += 65535)
            k_bf_tail_pad<<<dim3((unsigned)(((n - nreal) * n + kNT - 1) / kNT),
                                 (unsigned)(B - b0 < 65535 ? B - b0 : 65535)), kNT, 0, st>>>(
                n, nreal, D + b0 * ts.dense_doubles, V ? V + b0 * ts.dense_doubles : nullptr,
                ts.dense_doubles);
        const int e = launch_tail_factor(ts, B, BS, SYM, tail, neg, bad, tiny, S.k.status, st);
        if (e != 0) return e;
    }
    return (int)cudaGetLastError();
}

template <int BS, bool SYM>
int launch_block_solve(const DevSym &S, int B, const double *T, const double *L, const double *U,
                       double *x, const void *tail, cudaStream_t st) {
    if (B <= 0) return 0;
    const unsigned gy = (unsigned)((B + kNT - 1) / kNT), gy32 = (unsigned)((B + 31) / 32);
    for (int l = 0; l < S.nlevels; l++) {
        const int c0 = S.lvl_colptr[l], nc = S.sp_cols[l];
        if (nc <= 0) continue;
        if (nc < kSplitBelow && S.sp_rows[l] > kSplitTerms)
            k_bf_forward_split<BS><<<dim3((unsigned)nc, gy32), 32 * kSlices, 0, st>>>(
                S.k, B, T, L, x, c0);
        else
            k_bf_forward<BS><<<dim3((unsigned)nc, gy), kNT, 0, st>>>(S.k, B, T, L, x, c0);
    }
    if (S.k.tail_n > 0) {
        const int R = S.k.nb - S.k.k0;
        k_bf_tail_rhs<BS><<<dim3((unsigned)R, gy32), 32 * kSlices, 0, st>>>(S.k, B, T, x);
        const int e = launch_tail_solve(tail_shape(S.k.tail_n, B, SYM), B, R * BS, SYM, tail,
                                        x + (size_t)S.k.k0 * BS * B, st);
        if (e != 0) return e;
    }
    for (int l = S.nlevels - 1; l >= 0; l--) {
        const int c0 = S.lvl_colptr[l], nc = S.sp_cols[l];
        if (nc <= 0) continue;
        if (nc < kSplitBelow && S.sp_colblks[l] > kSplitTerms)
            k_bf_backward_split<BS, SYM><<<dim3((unsigned)nc, gy32), 32 * kSlices, 0, st>>>(
                S.k, B, L, U, x, c0);
        else
            k_bf_backward<BS, SYM><<<dim3((unsigned)nc, gy), kNT, 0, st>>>(S.k, B, L, U, x, c0);
    }
    return (int)cudaGetLastError();
}

exago_status grow_workspace(void **ws, size_t *bytes, size_t need, size_t least, const char *what) {
    if (*bytes >= need) return EXAGO_OK;
    size_t room = 0, total = 0;
    if (least < need && cudaMemGetInfo(&room, &total) == cudaSuccess && room + *bytes < need) need = least;
    if (*bytes >= need) return EXAGO_OK;
    if (*ws) {
        cudaError_t e = cudaDeviceSynchronize();
        if (e != cudaSuccess) return set_last_error(EXAGO_ECUDA, cudaGetErrorString(e));
        cudaFree(*ws);
        *ws = nullptr;
        *bytes = 0;
    }
    cudaError_t e = dev_malloc(ws, need);
    if (e != cudaSuccess) {
        *ws = nullptr;
        return set_last_error(e == cudaErrorMemoryAllocation ? EXAGO_ENOMEM : EXAGO_ECUDA, what);
    }
    *bytes = need;
    return EXAGO_OK;
}

void host_ranges(const BlockSym &S, DevSym &D) {
    D.k.nb = S.nb;
    D.k.nlevels = D.nlevels = S.nlevels;
    D.k.nblk = S.nblk;
    D.k.ntgt = (int64_t)S.tgt_blk.size();
    D.k.npairs = (int64_t)S.pairs.size();
    D.lvl_colptr = S.lvl_colptr;
    D.lvl_tptr = S.lvl_tptr;
    D.sp_cols = S.sp_cols;
    D.sp_tgts = S.sp_tgts;
    D.sp_pairs = S.sp_pairs;
    D.sp_rows = S.sp_rows;
    D.sp_colblks = S.sp_colblks;
    D.sparse_blocks = S.colptr[S.k0];
    D.k.k0 = S.k0;
    D.k.tail_n = S.tail_n;
}

int upload_block_sym(const BlockSym &S, DevSym &D, std::vector<void *> &allocs) {
    D = DevSym();
    host_ranges(S, D);
    auto up = [&](const void *src, size_t bytes, const void **dst) -> int {
        *dst = nullptr;
        if (bytes == 0) return 0;
        void *p = nullptr;
        cudaError_t e = dev_malloc(&p, bytes);
        if (e != cudaSuccess) return (int)e;
        allocs.push_back(p);
        e = cudaMemcpy(p, src, bytes, cudaMemcpyHostToDevice);
        *dst = p;
        return (int)e;
    };
    int e = S.tail_n > 0 ? tail_allow_smem() : 0;
#define UPV(field, vec) \
    if (!e) e = up(S.vec.data(), S.vec.size() * sizeof(S.vec[0]), (const void **)&D.k.field)
    UPV(colptr, colptr); UPV(rowidx, rowidx); UPV(rowptr, rowptr); UPV(rowblk, rowblk);
    UPV(rowcol, rowcol); UPV(lvl_cols, lvl_cols); UPV(tgt_blk, tgt_blk); UPV(tgt_diag, tgt_diag);
    UPV(tgt_fill, tgt_fill);
    UPV(tptr, tptr); UPV(pairs, pairs); UPV(tail_tgt, tail_tgt); UPV(tail_q1, tail_q1);
    UPV(tail_r1, tail_r1);
#undef UPV
    return e;
}

template int launch_block_factor<4, true>(const DevSym &, int, double *, double *, double *,
                                          double *, int *, int *, double, void *, cudaStream_t);
template int launch_block_factor<2, false>(const DevSym &, int, double *, double *, double *,
                                           double *, int *, int *, double, void *, cudaStream_t);
template int launch_block_solve<4, true>(const DevSym &, int, const double *, const double *,
                                         const double *, double *, const void *, cudaStream_t);
template int launch_block_solve<2, false>(const DevSym &, int, const double *, const double *,
                                          const double *, double *, const void *, cudaStream_t);

}  // namespace exago
