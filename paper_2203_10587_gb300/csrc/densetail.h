// The dense tail of the batched block factorisation (blockfact.h): the last R columns of the
// elimination order, whose factor is (nearly) full, factored as one dense matrix per state.
// Internal to the library.
//
// On bus graphs a minimum-degree order ends in a clique that holds almost all of the work: on the
// 2,000-bus grid the last 192 columns hold 95% of the block products (1.02 of 1.07 million per
// state) and 179 of the 190 levels.  Those products run here on the tensor cores, in 62-bit fixed point:
//
//   * A panel of 64 scalar columns of F = L D (and of L, or U' for LU) is kept as G = F 2^-c and
//     H = L 2^c, the columns balanced by powers of two (half_exp), G in FP64 and both as 7 "digits"
//     per value: with 2^e above every magnitude of a row's 64 values, each value is X 2^(e-62), X a
//     62-bit integer written in base 512 with digits in [-256, 256], so every digit is exact in
//     bf16.  A value below 2^-9 of its row's largest loses its lowest bits; the error of a product
//     is then 2^-61 of the rows' largest values, relative to sqrt|a_ii a_jj| as that of an FP64
//     elimination is (2^-53 of the terms' sum there).
//   * The product of two such rows is sum over digit pairs (s, t) of 2^(-9(s+t)) D_st, D_st a sum
//     of 64 products of integers of at most 2^16.  The 28 pairs with s + t <= 6 are multiplied by
//     tcgen05.mma into 7 FP32 accumulators in TMEM, one per s + t.  The sums with s + t <= 3 stay
//     within 2^24, so they are exact; the later ones would need digits near their bound in every
//     place to round at all, and their weight is 2^-36 and less.  The dropped pairs weigh 2^-63.
//   * The seven sums are put together in 64-bit integers (unit 2^-61 of the rows' bounds) and one
//     FP64 subtraction takes the 64 products' sum from the target, where the FP64 path
//     rounds 64 times.
//
// GB300's FP64 pipe retires 528 G multiply-adds/s (measured), so the 76 M of one state's tail
// take 75 ms for 512 states on it; their 28 bf16 products take 1-2 ms on the tensor cores.  Put
// together, 2,000 buses x 512 states: KKT step 96.3 to 15.6 ms, power-flow step 37.3 to 8.0 ms;
// 200 buses x 37 states, where the 190 levels' launches went instead: 1,442 to 513 us.  Mean error
// of the step against extended precision, before and after: 5.7e-15 and 5.6e-15 (2,000 buses),
// 3.1e-15 and 3.1e-15 (200); with barrier terms over many decades see half_exp.
//
// Per panel J of 64 columns, for every state:
//   k_dt_update<diag>  T_JJ -= sum_{K<J} F_JK L_JK'
//   k_dt_factor        scalar L D L' (or L D U) of T_JJ in FP64 without pivoting -- the pivots of
//                      the 4 x 4 (2 x 2) pivot blocks in order -- and the inverse of its unit
//                      triangle(s)
//   k_dt_update<rows>  for the 128-row tiles below: T_IJ -= sum_{K<J} F_IK L_JK', then
//                      F_IJ = T_IJ L_JJ^-T by the same digit product with the inverse (all of it
//                      with the columns balanced: G), and the digits of G_IJ and of H_IJ
// and k_dt_solve does both triangular sweeps of the tail.
#pragma once

#include <cuda_runtime.h>

#include <cstddef>
#include <cstdint>

namespace exago {

// Shape and workspace of the dense tail of B states (all offsets in bytes, 256-aligned).
struct TailShape {
    int n = 0;          // scalar size, a multiple of 64 (padded with the identity)
    int P = 0;          // panels of 64 columns
    int chunk = 0;      // states whose digits are held at a time
    size_t dn = 0, dv = 0;          // FP64 panels of F (and of U', LU only)
    size_t dinv = 0;                // reciprocal pivots
    size_t sf = 0, sl = 0;          // digits of F and of L / U', `chunk` states
    size_t ef = 0, el = 0;          // their row exponents
    size_t inv = 0, inve = 0;       // digits and exponents of the current panel's inverse(s)
    size_t bytes = 0;
    size_t dense_doubles = 0, digit_bytes = 0;   // per state: FP64 panels; digits of one operand
};
TailShape tail_shape(int n, int B, bool sym);

// Once per device: the kernels' dynamic shared memory.
int tail_allow_smem();

// Factors the assembled panels (dn, dv of the workspace w) of B states; neg, bad [B] count the
// negative and the near-zero pivots as the block factorisation does.
int launch_tail_factor(const TailShape &S, int B, int BS, bool sym, void *w, int *neg, int *bad,
                       double tiny, int *status, cudaStream_t st);
// Both sweeps on x (batch-interleaved, its first tail row at x0): r -> solution.
int launch_tail_solve(const TailShape &S, int B, int nreal, bool sym, const void *w, double *x0,
                      cudaStream_t st);

// Position of (row, col), row >= 64 (col / 64), in one state's FP64 panels: panel after panel,
// each column-major over its rows 64 J .. n - 1.
__host__ __device__ inline size_t tail_pos(int n, int row, int col) {
    const int J = col >> 6;
    return (size_t)64 * J * n - (size_t)2048 * J * (J - 1) + (size_t)(col & 63) * (n - 64 * J) +
           (row - 64 * J);
}

}  // namespace exago
