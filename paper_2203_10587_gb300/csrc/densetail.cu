// Dense tail of the batched block factorisation (densetail.h says what it computes and why).
#include <cuda_runtime.h>

#include <algorithm>

#include "densetail.h"

namespace exago {

namespace {

constexpr int kDigits = 7;            // base-512 digits of a value
constexpr int kTile = 8192;           // bytes of 64 rows x 64 digits (bf16)
constexpr int kFlag = 1 << 20;        // row exponent of a row that holds an infinity or a NaN
constexpr uint32_t kTmemCols = 512;   // 7 sums x 64 columns, allocated as a power of two
constexpr int kCols = 16;             // columns of a thread that finishes products (and one row)
constexpr int kEpi = 128 * (64 / kCols);   // such threads
constexpr int kUpdThreads = kEpi + 32;
constexpr int kSmemA = kDigits * 2 * kTile, kSmemB = kDigits * kTile;
constexpr int kSmemUpd = kSmemA + kSmemB + 1024;   // + alignment of the tiles to 1 KB
constexpr int kHalfSums = kDigits * 32;   // TMEM columns of the 7 sums of 32 columns
constexpr int kSpin = 1 << 20;        // polls of an mbarrier before a wait gives up
enum : int { ST_TIMEOUT_TAIL = 4 };

__device__ __forceinline__ uint32_t smem_u32(const void *p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}

// ---- balanced columns ----------------------------------------------------------------------------

// Column k of a panel is split as G_ik = F_ik 2^-c and H_jk = L_jk 2^c (LU: U'_jk 2^c), c half the
// exponent of its pivot d_k, here from the pivot's reciprocal (0 where that is zero, subnormal or not
// finite).  The scales cancel in the products.  With F = L D both operands are then about
// L_ik sqrt|d_k|, whose squares sum to the matrix's own diagonal entry at most (but for growth), so
// the split's errors are relative to sqrt|a_ii a_jj| as those of an elimination in FP64 are,
// whatever the scales of the variables.  Unscaled, the largest entries of a row of F and of one of L
// lie in different columns when pivots differ, as barrier terms make them near convergence: with
// barrier terms over 4, 8 and 12 decades the KKT step was 20, 45 and 26 times as far off as an
// elimination in FP64 for 150 buses of 450 branches (7, 4 and 7 for 100 of 260), balanced it is 1.2, 0.7
// and 0.4 (1.3, 1.1, 0.4).  2,000 buses x 512 states take 15.50 ms unscaled, 15.55 balanced.
__device__ __forceinline__ int half_exp(double r) {
    const int f = (__double2hiint(r) >> 20) & 0x7ff;
    return (unsigned)(f - 1) < 2046u ? (1023 - f) >> 1 : 0;
}

// v 2^c, |c| <= 1024, by moving the exponent field (a multiplication takes the FP64 pipe 64 cycles a
// warp); false, and v as it was, where either end is not a normal number.
__device__ __forceinline__ bool scale_normal(double &v, int c) {
    const int hi = __double2hiint(v), f = (hi >> 20) & 0x7ff;
    if (!((hi << 1) | __double2loint(v))) return true;   // zero
    if ((unsigned)(f - 1) >= 2046u || (unsigned)(f + c - 1) >= 2046u) return false;
    v = __hiloint2double(hi + c * (1 << 20), __double2loint(v));
    return true;
}
__device__ __forceinline__ double scale(double v, int c) {
    if (scale_normal(v, c)) return v;
    const int h = c / 2;
    return v * __hiloint2double((1023 + h) << 20, 0) * __hiloint2double((1023 + c - h) << 20, 0);
}

// ---- digits --------------------------------------------------------------------------------------

// Exponent field of |v| (subnormals and zero: 1).
__device__ __forceinline__ int exp_field(double v) {
    const int e = (__double2hiint(v) >> 20) & 0x7ff;
    return e ? e : 1;
}

// v as the integer X with v = X 2^(E - 1084), E the largest exponent field of its row: |X| < 2^62;
// bits below 2^0 are dropped.
__device__ __forceinline__ long long fixed62(double v, int E) {
    const uint32_t hi = (uint32_t)__double2hiint(v);
    const uint64_t frac = ((uint64_t)(hi & 0xfffff) << 32) | (uint32_t)__double2loint(v);
    const int f = (hi >> 20) & 0x7ff;
    const uint64_t m = f ? frac | (1ull << 52) : frac;
    const int sh = E - (f ? f : 1);
    const uint64_t x = sh <= 9 ? m << (9 - sh) : sh < 73 ? m >> (sh - 9) : 0;
    return (int)hi < 0 ? -(long long)x : (long long)x;
}

// The seven digits of eight neighbouring values of one row, packed as bf16 pairs: out[s] holds
// the eight digits of weight 512^(6 - s).  Adding 256 in each of the six lower places makes every
// digit a bit field less 256; a digit as a float (2^23 + field, less 2^23 + 256) is exact in bf16, its
// upper half.
__device__ __forceinline__ void digits8(const double *v, int E, uint4 *out) {
    constexpr unsigned long long kHalf =   // 256 (1 + 512 + .. + 512^5)
        256ull * (1ull + (1ull << 9) + (1ull << 18) + (1ull << 27) + (1ull << 36) + (1ull << 45));
    uint32_t p[kDigits][4];
#pragma unroll
    for (int h = 0; h < 4; h++) {
        uint32_t f[2][kDigits];
#pragma unroll
        for (int e = 0; e < 2; e++) {
            const unsigned long long X = (unsigned long long)fixed62(v[2 * h + e], E) + kHalf;
            const uint32_t lo = (uint32_t)X, hi = (uint32_t)(X >> 32);
            const uint32_t d[kDigits] = {0, hi >> 13, hi >> 4, __funnelshift_r(lo, hi, 27), lo >> 18, lo >> 9, lo};
#pragma unroll
            for (int s = 1; s < kDigits; s++)
                f[e][s] = __float_as_uint(__uint_as_float((d[s] & 511) | 0x4b000000u) - 8388864.0f);
            f[e][0] = __float_as_uint(__uint_as_float(0x4b000000u + (uint32_t)(((int)hi >> 22) + 512)) - 8389120.0f);
        }
#pragma unroll
        for (int s = 0; s < kDigits; s++) p[s][h] = __byte_perm(f[0][s], f[1][s], 0x7632);
    }
#pragma unroll
    for (int s = 0; s < kDigits; s++) out[s] = make_uint4(p[s][0], p[s][1], p[s][2], p[s][3]);
}

// Byte of (row, 8-column group) in a tile of 128-byte rows with the 128-byte swizzle.
__device__ __forceinline__ int tile_at(int row, int grp) {
    return row * 128 + ((grp ^ (row & 7)) << 4);
}

// Row exponent as stored beside the digits.
__device__ __forceinline__ int row_exp(int E) { return E >= 2047 ? kFlag : E - 1022; }

// The digit sums of one target put together: sum_g D_g 512^(12 - g) = W 2^(63 + shift) + less, |W| < 2^62.
// The unit 2^63 is 2^-61 of the rows' bounds; where the sum is too large for it (which digits near
// their bound in every place would need) it is rounded to 64 units.  A fixed unit of 2^-56 made the
// 200-bus KKT step, whose rows' entries range over five decades, 1.7 times as far off as in FP64,
// and a floor in place of the rounding made it 25 times on a power flow.
__device__ __forceinline__ long long join_sums(const float *d, int *shift) {
    const int i5 = __float2int_rn(fmaf(d[6], 1.0f / 512.0f, d[5]));
    const int i4 = __float2int_rn(d[4]), i3 = __float2int_rn(d[3]), i2 = __float2int_rn(d[2]);
    const int i1 = __float2int_rn(d[1]), i0 = __float2int_rn(d[0]);
    const long long hi = (long long)i0 * (1 << 18) + ((long long)i1 * 512 + i2);
    const long long lo = (long long)i3 * (1 << 18) + ((long long)i4 * 512 + i5);
    const bool wide = (unsigned long long)(hi + (1ll << 34)) >> 35;   // |hi| >= 2^34
    *shift = wide ? 6 : 0;
    return wide ? hi * (1 << 21) + ((lo + 32) >> 6) : hi * (1 << 27) + lo;
}

// Exponent field of what one unit of W weighs for rows of exponents ea and eb: 2^(ea + eb - 61).
__device__ __forceinline__ int unit_field(int ea, int eb) { return ea + eb + (1023 - 61); }

// W 2^(f - 1023) as a double, rounded to nearest, on the integer pipe: a conversion instruction
// takes as long on the FP64 pipe as the addition that follows (64 cycles a warp), these twenty
// instructions a third of it.  Zero where it would underflow; NaN for a row's flag or an overflow.
__device__ __forceinline__ double weigh(long long W, int f) {
    const unsigned long long a = (unsigned long long)(W < 0 ? -W : W);
    const int s = __clzll((long long)a);
    const unsigned long long m = a << s;
    const int e = f + 62 - s;   // field of the result, less the leading one's carry
    unsigned long long r = (m >> 11) + ((m >> 10) & 1) + ((unsigned long long)(unsigned)e << 52);
    if (e < 0 || a == 0) r = 0;
    if (e >= 2046) r = 0x7ff8000000000000ull;
    if (W < 0) r |= 1ull << 63;
    return __longlong_as_double((long long)r);
}

// ---- barriers, copies, tensor cores --------------------------------------------------------------

__device__ __forceinline__ void mbar_init(uint64_t *b, int count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(b)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t *b) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(b)) : "memory");
}
__device__ __forceinline__ void mbar_expect(uint64_t *b, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(b)),
                 "r"(bytes)
                 : "memory");
}
// Waits for the phase of the given parity; false (and a timeout code) after kSpin polls, and at
// once when another wait of the block has given up.
__device__ __forceinline__ bool mbar_wait(uint64_t *b, uint32_t parity, int *status, volatile int *dead) {
    for (int i = 0; i < kSpin; i++) {
        uint32_t ok;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(ok)
            : "r"(smem_u32(b)), "r"(parity)
            : "memory");
        if (ok) return true;
        if (*dead) return false;
    }
    *dead = 1;
    if (status) *(volatile int *)status = ST_TIMEOUT_TAIL;
    return false;
}
__device__ __forceinline__ void copy_in(void *dst, const void *src, uint32_t bytes, uint64_t *bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(smem_u32(dst)), "l"(src), "r"(bytes), "r"(smem_u32(bar))
                 : "memory");
}
__device__ __forceinline__ void copy_out(void *dst, const void *src, uint32_t bytes) {
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst),
                 "r"(smem_u32(src)), "r"(bytes)
                 : "memory");
}

// Shared-memory operand: K-major rows of 128 bytes, 128-byte swizzle, 8-row groups 1 KB apart.
__device__ __forceinline__ uint64_t mma_desc(uint32_t addr) {
    return (uint64_t)((addr >> 4) & 0x3fff) | ((uint64_t)1 << 16) | ((uint64_t)(1024 >> 4) << 32) |
           ((uint64_t)1 << 46) | ((uint64_t)2 << 61);
}
// D: FP32, A and B: bf16 K-major, 128 x N.
__host__ __device__ constexpr uint32_t mma_instr(int N) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N / 8) << 17) | ((128u / 16) << 24);
}

template <int N>
__device__ __forceinline__ void mma(uint32_t d, uint64_t a, uint64_t b, bool add) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d),
        "l"(a), "l"(b), "r"(mma_instr(N)), "r"((int)add)
        : "memory");
}

// Digit S of the rows times digits 0 .. 6 - S of 32 columns: these lie one after another in shared
// memory and the sums S .. 6 in TMEM, so they are one operand of 32 (7 - S) columns.  28
// instructions in place of 112 of 32 columns, which one thread could not issue as fast as they ran.
template <int S>
__device__ __forceinline__ void issue_digit(uint32_t tmem, uint64_t a, uint64_t b) {
#pragma unroll
    for (int k = 0; k < 4; k++)
        mma<32 * (kDigits - S)>(tmem + 32 * S, a + ((S * 2 * kTile + 32 * k) >> 4), b + ((32 * k) >> 4),
                                S > 0 || k > 0);
}
// All 28 digit pairs of one 64-deep product with 32 columns, into their 7 sums.
__device__ __forceinline__ void issue_products(uint32_t tmem, uint32_t a0, uint32_t b0) {
    const uint64_t a = mma_desc(a0), b = mma_desc(b0);
    issue_digit<0>(tmem, a, b);
    issue_digit<1>(tmem, a, b);
    issue_digit<2>(tmem, a, b);
    issue_digit<3>(tmem, a, b);
    issue_digit<4>(tmem, a, b);
    issue_digit<5>(tmem, a, b);
    issue_digit<6>(tmem, a, b);
}
__device__ __forceinline__ void commit(uint64_t *bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                     smem_u32(bar))
                 : "memory");
}
// Four columns of this lane's row of the seven sums.  The wait names the loaded registers, so that
// nothing that reads them moves ahead of it.
__device__ __forceinline__ void tmem_sums4(uint32_t addr, float (*v)[4]) {
    uint32_t r[kDigits][4];
#pragma unroll
    for (int g = 0; g < kDigits; g++)
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
                     : "=r"(r[g][0]), "=r"(r[g][1]), "=r"(r[g][2]), "=r"(r[g][3])
                     : "r"(addr + 32 * g)
                     : "memory");
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[0][0]), "+r"(r[0][1]), "+r"(r[0][2]), "+r"(r[0][3]), "+r"(r[1][0]),
                   "+r"(r[1][1]), "+r"(r[1][2]), "+r"(r[1][3]), "+r"(r[2][0]), "+r"(r[2][1]),
                   "+r"(r[2][2]), "+r"(r[2][3]), "+r"(r[3][0]), "+r"(r[3][1])
                 :: "memory");
    asm volatile("" : "+r"(r[3][2]), "+r"(r[3][3]), "+r"(r[4][0]), "+r"(r[4][1]), "+r"(r[4][2]),
                      "+r"(r[4][3]), "+r"(r[5][0]), "+r"(r[5][1]), "+r"(r[5][2]), "+r"(r[5][3]),
                      "+r"(r[6][0]), "+r"(r[6][1]), "+r"(r[6][2]), "+r"(r[6][3]) :: "memory");
#pragma unroll
    for (int g = 0; g < kDigits; g++)
#pragma unroll
        for (int c = 0; c < 4; c++) v[g][c] = __uint_as_float(r[g][c]);
}
__device__ __forceinline__ void epi_sync() { asm volatile("bar.sync 1, %0;" ::"n"(kEpi) : "memory"); }
// The threads of one half of the columns.
__device__ __forceinline__ void half_sync(int half) {
    asm volatile("bar.sync %0, %1;" ::"r"(2 + half), "n"(kEpi / 2) : "memory");
}

// The thread's values, eight places on: the loops below take eight values at a time from the front,
// so that their bodies are in the instruction cache once (unrolled over all columns, half of the
// stalls were for instructions).
__device__ __forceinline__ void rotate8(double *v) {
    double t[8];
#pragma unroll
    for (int i = 0; i < 8; i++) t[i] = v[i];
#pragma unroll
    for (int i = 0; i < kCols - 8; i++) v[i] = v[i + 8];
#pragma unroll
    for (int i = 0; i < 8; i++) v[kCols - 8 + i] = t[i];
}

// acc[0 .. NC) -= (sub) or = the product in TMEM, this thread's row and NC columns from column c0 of
// the half; ea: the row's exponent, eb [32] the columns' (shared memory).
template <int NC>
__device__ __forceinline__ void take_product(uint32_t tmem, int c0, int ea, const int *eb, double *acc,
                                             bool sub) {
#pragma unroll 1
    for (int q = 0; q < NC / 8; q++) {
#pragma unroll
        for (int h = 0; h < 2; h++) {
            float d[kDigits][4];
            tmem_sums4(tmem + c0 + 8 * q + 4 * h, d);
#pragma unroll
            for (int c = 0; c < 4; c++) {
                float v[kDigits];
#pragma unroll
                for (int g = 0; g < kDigits; g++) v[g] = d[g][c];
                int shift;
                const long long W = join_sums(v, &shift);
                const double w = weigh(W, unit_field(ea, eb[c0 + 8 * q + 4 * h + c]) + shift);
                acc[4 * h + c] = sub ? acc[4 * h + c] - w : w;
            }
        }
        if (NC > 8) rotate8(acc);
    }
}

struct UpdateArgs {
    int n, P, J;
    double *D;                        // FP64 panels of the targets
    size_t dstride;                   // doubles per state
    const double *dinv;               // [n] per state
    const char *sa, *sb;              // digits of the row operand and of the column operand
    const int *xa, *xb;               // their row exponents [P][n] per state
    char *oa, *ob;                    // digits written: of F (or, LU's upper side, of U'); of L
    int *ya, *yb;
    const char *inv;                  // digits of the panel's inverse, 7 tiles per state
    const int *inve;                  // [64] per state
    size_t sstride;                   // bytes of one operand's digits per state
    int *status;
};

// Digits of panel K: [digit][row tile K + 1 .. P - 1][8 KB].
__device__ __forceinline__ size_t digit_at(int P, int K, int s, int I) {
    return (size_t)kTile * ((size_t)kDigits * (K * (P - 1) - K * (K - 1) / 2) +
                            (size_t)s * (P - 1 - K) + (I - K - 1));
}

// One tile of 128 rows (DIAG: the panel's own 64) of panel J, one block per (tile, state).
// MODE 0: F and L (SYM); 1: F alone (LU, lower side); 2: U' from U' D' (LU, upper side).  Targets are
// T 2^-c from the start, and what is left in their place is G = F 2^-c (MODE 2: H = U' 2^c).
// What bounds it: the 8,192 targets' integer joins and two FP64-pipe instructions each, beside 2.4
// us of tensor work a 64-deep step; one block per SM (172 KB of digits), 16 warps that finish
// products beside one that issues copies and MMAs.  The columns go in two halves of 32, each with
// its sums in TMEM and 8 warps of its own, so that one half's products run while the other's sums
// are joined: a 64-deep step 6.5 to 8 us (8 with all 64 columns at once), half of it the
// 172 KB from HBM.  DIAG puts the 64 rows into both halves of the lanes, so that every warp has
// half the columns: 8.1 to 5.9 us a step.  2,000 buses x 512 states, all launches: 9.8 to 8.7 ms.
// A wait that gives up sets the status word and the block's flag; the block then runs to its end
// on whatever it holds, so that every barrier is met.
template <bool DIAG, int MODE>
__global__ void __launch_bounds__(kUpdThreads, 1) k_dt_update(const UpdateArgs A) {
    extern __shared__ char raw[];
    __shared__ uint64_t bar_full, bar_mma[2], bar_epi[2], bar_tgt;
    __shared__ uint32_t s_tmem;
    __shared__ volatile int s_dead;
    __shared__ int s_eb[2][64], s_em[64 / kCols][128];
    __shared__ __align__(16) int s_c[64];        // the panel's columns' exponents (half_exp)
    __shared__ __align__(16) double s_hg[64];    // H / G: the pivots' reciprocals, scaled by 2^2c
    char *sA = (char *)(((uintptr_t)raw + 1023) & ~(uintptr_t)1023), *sB = sA + kSmemA;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const size_t st = blockIdx.y;
    const int n = A.n, P = A.P, J = A.J;
    const int I0 = DIAG ? J : J + 1 + 2 * (int)blockIdx.x;   // first 64-row tile
    const int tiles = DIAG ? 1 : min(2, P - I0);
    if (!DIAG && tid < 64) {
        const double r = __ldcg(A.dinv + st * n + 64 * J + tid);
        s_c[tid] = half_exp(r);
        s_hg[tid] = scale(r, 2 * s_c[tid]);
    }
    if (tid == 0) {
        mbar_init(&bar_full, 1);
        for (int h = 0; h < 2; h++) {
            mbar_init(&bar_mma[h], 1);
            mbar_init(&bar_epi[h], kEpi / 2);
        }
        mbar_init(&bar_tgt, kEpi);
        s_dead = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == kEpi / 32) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         smem_u32(&s_tmem)),
                     "r"(kTmemCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = s_tmem;

    if (warp == kEpi / 32) {
        if (lane == 0) {
            const char *sa = A.sa + st * A.sstride, *sb = A.sb + st * A.sstride;
            const uint32_t a0 = smem_u32(sA), b0 = smem_u32(sB);
            const int steps = DIAG ? J : J + 1;   // the last: the targets times the inverse
            bool ok = true;
            for (int K = 0; K < steps && ok; K++) {
                const bool last = K == J;
                // both halves' products of the step before: its operands are no longer read
                if (K > 0) ok = mbar_wait(&bar_mma[1], (K - 1) & 1, A.status, &s_dead);
                if (!ok) break;   // nothing in flight
                mbar_expect(&bar_full, last ? kDigits * kTile : kDigits * kTile * (DIAG ? 3 : tiles + 1));
                for (int s = 0; s < kDigits; s++) {
                    const char *b = last ? A.inv + (st * kDigits + s) * kTile : sb + digit_at(P, K, s, J);
                    if (!last) {
                        const char *a = sa + digit_at(P, K, s, I0);
                        copy_in(sA + s * 2 * kTile, a, kTile * tiles, &bar_full);
                        if (DIAG) copy_in(sA + s * 2 * kTile + kTile, a, kTile, &bar_full);
                    }
                    for (int h = 0; h < 2; h++)
                        copy_in(sB + (h * kDigits + s) * (kTile / 2), b + h * (kTile / 2), kTile / 2, &bar_full);
                }
                // the half's product before has left TMEM; the targets' digits are in shared memory
                if (K > 0) ok = mbar_wait(&bar_epi[0], (K - 1) & 1, A.status, &s_dead);
                if (last) ok = mbar_wait(&bar_tgt, 0, A.status, &s_dead) && ok;
                // this wait also holds a block that gave up until its copies have landed
                volatile int no = 0;
                ok = mbar_wait(&bar_full, K & 1, A.status, ok ? &s_dead : &no) && ok;
                if (!ok) { s_dead = 1; break; }
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                issue_products(tmem, a0, b0);
                commit(&bar_mma[0]);
                if (K > 0) ok = mbar_wait(&bar_epi[1], (K - 1) & 1, A.status, &s_dead);
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                issue_products(tmem + kHalfSums, a0, b0 + kDigits * (kTile / 2));
                commit(&bar_mma[1]);
            }
        }
        __syncwarp();
    } else {
        const int part = warp >> 2, half = part >> 1;     // columns kCols part ..
        // DIAG: lanes 64 .. 127 hold the 64 rows again and take the last 8 of the 16 columns
        const int lane128 = ((warp & 3) << 5) | lane, row = DIAG ? lane128 & 63 : lane128;
        const int c0 = kCols * part + (DIAG ? 8 * (lane128 >> 6) : 0);
        const int grow = 64 * I0 + row;                   // row of the matrix
        const bool live = row < 64 * tiles;
        const uint32_t tw = tmem + ((uint32_t)(warp & 3) << 21) + kHalfSums * half;
        const int ld = n - 64 * J;
        double *Dp = A.D + st * A.dstride + tail_pos(n, 64 * J, 64 * J) + (size_t)c0 * ld +
                     (grow - 64 * J);
        constexpr int NC = DIAG ? 8 : kCols;
        double acc[kCols] = {};
#pragma unroll
        for (int c = 0; c < NC; c++) acc[c] = live ? __ldcg(Dp + (size_t)c * ld) : 0.0;
        if (!DIAG) {   // T 2^-c, while the first operands are copied
            bool normal = true;
#pragma unroll
            for (int c = 0; c < kCols; c++) normal &= scale_normal(acc[c], -s_c[c0 + c]);
            if (!normal) {   // all of them again, one after the other
#pragma unroll 1
                for (int c = 0; c < kCols; c++) {
#pragma unroll
                    for (int i = 1; i < kCols; i++) acc[i - 1] = acc[i];
                    acc[kCols - 1] = scale(__ldcg(Dp + (size_t)c * ld), -s_c[c0 + c]);
                }
            }
        }
        const int *xa = A.xa + st * (size_t)P * n, *xb = A.xb + st * (size_t)P * n;
        // steps K < J: the products of the panels before; J: the targets times the inverse, G_IJ
        // (MODE 2: H_IJ); J + 1: its digits kept for the panels to come; J + 2: H_IJ's (MODE 0)
        const int steps = DIAG ? J : J + (MODE == 0 ? 3 : 2);
        const bool mine = (tid & (kEpi / 2 - 1)) < 32;    // one warp of a half keeps its columns' exponents
        const int col = 32 * half + lane;
#pragma unroll 1
        for (int K = 0; K < steps; K++) {
            int ea = 0;
            if (DIAG || K < J) {
                if (mine) s_eb[K & 1][col] = __ldcg(xb + (size_t)K * n + 64 * J + col) - (DIAG ? 0 : s_c[col]);
                if (live) ea = __ldcg(xa + (size_t)K * n + grow);
                half_sync(half);
            } else {
                if (K == J && mine) s_eb[J & 1][col] = __ldcg(A.inve + st * 64 + col);
                int E = 1;
#pragma unroll
                for (int c = 0; c < kCols; c++) E = max(E, exp_field(acc[c]));
                s_em[part][row] = E;
                epi_sync();
#pragma unroll
                for (int h = 0; h < 64 / kCols; h++) E = max(E, s_em[h][row]);
                ea = row_exp(E);
#pragma unroll 1
                for (int q = 0; q < kCols / 8; q++) {
                    uint4 o[kDigits];
                    digits8(acc, E, o);
#pragma unroll
                    for (int s = 0; s < kDigits; s++)
                        *(uint4 *)(sA + s * 2 * kTile + tile_at(row, kCols / 8 * part + q)) = o[s];
                    rotate8(acc);
                }
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                if (K == J) mbar_arrive(&bar_tgt);
            }
            if (DIAG || K <= J) {
                mbar_wait(&bar_mma[half], K & 1, A.status, &s_dead);
                __syncwarp();
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                take_product<NC>(tw, c0 & 31, ea, s_eb[K & 1] + 32 * half, acc, K < J);
                asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                if (DIAG || K < J) mbar_arrive(&bar_epi[half]);
                if (!DIAG && K == J) {
                    if (MODE == 2)
#pragma unroll
                        for (int c = 0; c < kCols; c++) acc[c] *= s_hg[c0 + c];
                    if (live)
#pragma unroll
                        for (int c = 0; c < kCols; c++) Dp[(size_t)c * ld] = acc[c];
                }
            } else {
                const bool second = K == J + 2;
                int *xo = (second ? A.yb : A.ya) + st * (size_t)P * n + (size_t)J * n + grow;
                if (part == 0 && live) *xo = ea;
                epi_sync();
                if (tid == 0) {
                    char *out = (second ? A.ob : A.oa) + st * A.sstride;
                    for (int s = 0; s < kDigits; s++)
                        copy_out(out + digit_at(P, J, s, I0), sA + s * 2 * kTile, kTile * tiles);
                    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
                    asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
                }
                if (MODE == 0 && !second)
#pragma unroll
                    for (int c = 0; c < kCols; c++) acc[c] *= s_hg[c0 + c];
                epi_sync();
            }
        }
        if (DIAG)
#pragma unroll
            for (int c = 0; c < NC; c++) Dp[(size_t)c * ld] = acc[c];
    }
    __syncthreads();
    if (warp == kEpi / 32)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols));
}

// ---- pivots --------------------------------------------------------------------------------------

constexpr int kFacThreads = 256;
constexpr int kPitch = 65;   // doubles per column in shared memory: rows of a column and columns
                             // of a row both spread over the banks

// Digits of the 64 x 64 unit lower triangular X (shared memory, X[k * kPitch + row] below the diagonal)
// with one exponent per row, as X_jk 2^(c_k - c_j): it takes T 2^-c to G.
__device__ __forceinline__ void panel_digits(const double *X, const int *c, char *out, int *xout) {
    for (int it = threadIdx.x; it < 512; it += kFacThreads) {
        const int row = it >> 3, grp = it & 7;
        double v[8];
        int E = 1;
#pragma unroll
        for (int k = 0; k < 8; k++) {
            const int col = 8 * grp + k;
            v[k] = row > col ? scale(X[col * kPitch + row], c[col] - c[row]) : row == col ? 1.0 : 0.0;
            E = max(E, exp_field(v[k]));
        }
        for (int h = 1; h < 8; h <<= 1) E = max(E, __shfl_xor_sync(0xffffffffu, E, h));
        uint4 o[kDigits];
        digits8(v, E, o);
#pragma unroll
        for (int s = 0; s < kDigits; s++) *(uint4 *)(out + s * kTile + tile_at(row, grp)) = o[s];
        if (grp == 0) xout[row] = row_exp(E);
    }
}

// X = M^-1 for a unit lower triangular M in shared memory: entry (i, k), i > k, at M[k * kPitch + i] or
// (T) at M[i * kPitch + k].  Warp w owns columns w, w + 8, ..; lo / hi: rows lane and lane + 32.
template <bool T>
__device__ __forceinline__ void unit_inverse(const double *M, int warp, int lane, double *lo, double *hi) {
    auto at = [&](int i, int k) { return i > k ? (T ? M[i * kPitch + k] : M[k * kPitch + i]) : 0.0; };
#pragma unroll
    for (int c = 0; c < 8; c++) {
        const int j = warp + 8 * c;
        lo[c] = j == lane ? 1.0 : 0.0;
        hi[c] = j == lane + 32 ? 1.0 : 0.0;
    }
    for (int k = 0; k < 31; k++) {
        const double ml = at(lane, k), mh = at(lane + 32, k);
#pragma unroll
        for (int c = 0; c < 4; c++)
            if (warp + 8 * c <= k) {
                const double x = __shfl_sync(0xffffffffu, lo[c], k);
                lo[c] = fma(-ml, x, lo[c]);
                hi[c] = fma(-mh, x, hi[c]);
            }
    }
    for (int k = 31; k < 63; k++) {
        const double mh = at(lane + 32, k);
#pragma unroll
        for (int c = 0; c < 8; c++)
            if (warp + 8 * c <= k) {
                const double x = __shfl_sync(0xffffffffu, k == 31 ? lo[c] : hi[c], (k - 32) & 31);
                hi[c] = fma(-mh, x, hi[c]);
            }
    }
}

// Magnitude as an integer that compares as it; a NaN counts as zero (as fmax ignores it).
__device__ __forceinline__ unsigned long long mag(double v) {
    const unsigned long long u = (unsigned long long)__double_as_longlong(v) & ~(1ull << 63);
    return u > 0x7ff0000000000000ull ? 0 : u;
}

// L D L' (or L D U) of the panel's 64 x 64 diagonal block without pivoting, one block per state;
// then the inverses of L (and of U'), as digits for the rows below and in FP64, in place of the
// block, for the sweeps.  Warp w holds columns w, w + 8, .. in registers, a lane rows lane and
// lane + 32.  Step k subtracts column k's part from the columns after it; the warp that holds column
// k + 1 does that one first, and its pivot, reciprocal and publication, while the others work.
// Bound by the FP64 pipe (about 5,000 warp instructions of 64 cycles over four pipes) and, for
// few states, by the chain of pivots: 192 us for 512 states (290 before the look-ahead), 76 for 37.
// The pivots are divided, as everywhere else: a step from the hardware's approximation was 3 us
// shorter on 37 states and up to 1 ulp off.
template <bool SYM, int BS>
__global__ void __launch_bounds__(kFacThreads, 4) k_dt_factor(int n, int J, double *D, double *V,
                                                           size_t dstride, double *dinv, char *linv,
                                                           int *line, char *uinv, int *uine,
                                                           int *neg, int *bad, double tiny) {
    extern __shared__ double sm[];
    double *Ls = sm;   // L by columns, Ls[k * kPitch + i], i > k; LU: row k of D U at Ls[j * kPitch + k]
    __shared__ double s_f[2][64], s_d[64], s_r[64];
    __shared__ int s_c[64];   // the columns' exponents (half_exp)
    __shared__ unsigned long long s_max[64];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const size_t st = blockIdx.x;
    const int ld = n - 64 * J;
    double *Dp = D + st * dstride + tail_pos(n, 64 * J, 64 * J);
    double lo[8], hi[8];
#pragma unroll
    for (int c = 0; c < 8; c++) {
        const int j = warp + 8 * c;
        const double *p = Dp + (size_t)j * ld;
        lo[c] = SYM && lane < j ? 0.0 : __ldcg(p + lane);
        hi[c] = SYM && lane + 32 < j ? 0.0 : __ldcg(p + lane + 32);
    }
    // the largest entry of each pivot block, when its turn comes: column j's part
    auto block_max = [&](int c, int j) {
        const int b0 = j / BS * BS;
        const double v = b0 < 32 ? lo[c] : hi[c];
        if ((lane & ~(BS - 1)) == (b0 & 31)) atomicMax(s_max + j, mag(v));
    };
    // column k = warp + 8 c is final: its pivot, and the column for the other warps
    auto publish = [&](int c, int k) {
        const double d = __shfl_sync(0xffffffffu, c < 4 ? lo[c] : hi[c], k & 31);
        const double r = 1.0 / d;
        const double fl = lane > k ? lo[c] : 0.0, fh = lane + 32 > k ? hi[c] : 0.0;
        s_f[k & 1][lane] = fl;
        s_f[k & 1][lane + 32] = fh;
        const double ll = fl * r, lh = fh * r;
        if (lane > k) Ls[k * kPitch + lane] = ll;
        if (lane + 32 > k) Ls[k * kPitch + lane + 32] = lh;
        if (lane == 0) {
            s_d[k] = d;
            s_r[k] = r;
        }
    };
    if (tid < 64) s_max[tid] = 0;
    __syncthreads();
    if (warp < BS) block_max(0, warp);
    if (warp == 0) publish(0, 0);
#pragma unroll
    for (int c = 0; c < 8; c++) {
#pragma unroll 1
        for (int w = 0; w < 8; w++) {
            const int k = 8 * c + w;
            __syncthreads();
            const double fl = SYM ? s_f[k & 1][lane] : lane > k ? Ls[k * kPitch + lane] : 0.0;
            const double fh = SYM ? s_f[k & 1][lane + 32] : lane + 32 > k ? Ls[k * kPitch + lane + 32] : 0.0;
            auto update = [&](int q) {   // column warp + 8 q > k loses column k's part
                const int j = warp + 8 * q;
                double u;   // SYM: F's column times L's row; else L's column times the row of D U
                if (SYM) {
                    u = Ls[k * kPitch + j];
                } else {
                    u = __shfl_sync(0xffffffffu, c < 4 ? lo[q] : hi[q], k & 31);
                    if (lane == 0) Ls[j * kPitch + k] = u;   // D U, scaled at the end
                }
                if (c < 4 && (!SYM || q < 4)) lo[q] = fma(-fl, u, lo[q]);
                hi[q] = fma(-fh, u, hi[q]);
                // column j's block is the next to be eliminated
                if ((k + 1) % BS == 0 && j <= k + BS) block_max(q, j);
            };
            if (w < 7) {
                if (warp == w + 1) {
                    update(c);
                    publish(c, k + 1);
                } else if (warp > w) {
                    update(c);
                }
            } else if (c < 7 && warp == 0) {
                update(c + 1 < 8 ? c + 1 : 7);
                publish(c + 1 < 8 ? c + 1 : 7, k + 1);
            }
#pragma unroll
            for (int q = c + 1; q < 8; q++)
                if (q > c + 1 || w < 7 || warp > 0) update(q);
        }
    }
    __syncthreads();
    if (tid < 64) {
        dinv[st * n + 64 * J + tid] = s_r[tid];
        s_c[tid] = half_exp(s_r[tid]);
        unsigned long long a = 0;
        for (int h = 0; h < BS; h++) a = max(a, s_max[tid / BS * BS + h]);
        const double d = s_d[tid];
        const int nn = __popc(__ballot_sync(0xffffffffu, d < 0.0));
        const int nb = __popc(__ballot_sync(
            0xffffffffu, !(fabs(d) > tiny * __longlong_as_double((long long)a))));
        if (lane == 0 && nn) atomicAdd(neg + st, nn);
        if (lane == 0 && nb) atomicAdd(bad + st, nb);
    }
    if (!SYM) {
        for (int e = tid; e < 64 * 64; e += kFacThreads)
            if ((e >> 6) > (e & 63)) Ls[(e >> 6) * kPitch + (e & 63)] *= s_r[e & 63];
        __syncthreads();
    }
    // the inverses of L and (LU) of U'; each takes L's place in shared memory
    auto finish = [&](double *out, char *digits, int *exps) {
        __syncthreads();
#pragma unroll
        for (int c = 0; c < 8; c++) {
            const int j = warp + 8 * c;
            if (lane > j) Ls[j * kPitch + lane] = lo[c];
            if (lane + 32 > j) Ls[j * kPitch + lane + 32] = hi[c];
            out[(size_t)j * ld + lane] = lo[c];
            out[(size_t)j * ld + lane + 32] = hi[c];
        }
        __syncthreads();
        panel_digits(Ls, s_c, digits + st * kDigits * kTile, exps + st * 64);
    };
    unit_inverse<false>(Ls, warp, lane, lo, hi);
    finish(Dp, linv, line);
    if (!SYM) {
        unit_inverse<true>(Ls, warp, lane, lo, hi);
        finish(V + st * dstride + tail_pos(n, 64 * J, 64 * J), uinv, uine);
    }
}

// ---- sweeps --------------------------------------------------------------------------------------

constexpr int kSolThreads = 256;   // eight warps of eight columns

// The warp's sums of a[0 .. 8): lanes 4 c .. 4 c + 3 receive that of a[c].  Half of the values move to
// the other half of the lanes at each of three steps, so 9 additions in place of 40.
__device__ __forceinline__ double sum8(double *a, int lane) {
#pragma unroll
    for (int h = 4; h >= 1; h >>= 1) {
        const bool up = lane & (4 * h);
#pragma unroll
        for (int c = 0; c < h; c++) {
            const double give = up ? a[c] : a[c + h], keep = up ? a[c + h] : a[c];
            a[c] = keep + __shfl_xor_sync(0xffffffffu, give, 4 * h);
        }
    }
    a[0] += __shfl_xor_sync(0xffffffffu, a[0], 2);
    return a[0] + __shfl_xor_sync(0xffffffffu, a[0], 1);
}

// Both sweeps of one state's tail.  Forward, per panel: z = D^-1 L^-1 r, the rows below lose F z; backward:
// the panel's unknowns lose U's (or D^-1 F's) part, then L^-T (U^-1).  Below the panels' squares D holds
// G = F 2^-c and V H = U' 2^c (half_exp).
template <bool SYM>
__global__ void __launch_bounds__(kSolThreads) k_dt_solve(int n, int nreal, int B, const double *D,
                                                          const double *V, size_t dstride,
                                                          const double *dinv, double *x0) {
    extern __shared__ double sx[];               // [n] the vector, then [4][64] partial sums
    double *part = sx + n;
    __shared__ double zs[64];                    // z 2^c
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const size_t st = blockIdx.x;
    const double *Db = D + st * dstride, *Vb = SYM ? Db : V + st * dstride;
    const double *di = dinv + st * n;
    for (int i = tid; i < n; i += kSolThreads) sx[i] = i < nreal ? x0[(size_t)i * B + st] : 0.0;
    __syncthreads();
    const int P = n / 64, r64 = tid & 63, q4 = tid >> 6;
    for (int J = 0; J < P; J++) {
        const int ld = n - 64 * J, j0 = 64 * J;
        const double *Dp = Db + tail_pos(n, j0, j0);
        double a = 0.0;
#pragma unroll 4
        for (int k = 16 * q4; k < 16 * q4 + 16; k++) a = fma(__ldg(Dp + (size_t)k * ld + r64), sx[j0 + k], a);
        part[q4 * 64 + r64] = a;
        __syncthreads();
        if (tid < 64) {
            const double r = __ldg(di + j0 + tid);
            const double z = ((part[tid] + part[64 + tid]) + (part[128 + tid] + part[192 + tid])) * r;
            sx[j0 + tid] = z;
            zs[tid] = scale(z, half_exp(r));
        }
        __syncthreads();
        // four sums of 16 terms, then one subtraction: shorter chains, and fewer roundings at the
        // size of the target
        for (int i = 64 + tid; i < ld; i += kSolThreads) {
            double a[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll 4
            for (int k = 0; k < 64; k += 4)
#pragma unroll
                for (int h = 0; h < 4; h++)
                    a[h] = fma(__ldg(Dp + (size_t)(k + h) * ld + i), zs[k + h], a[h]);
            sx[j0 + i] -= (a[0] + a[1]) + (a[2] + a[3]);
        }
        __syncthreads();
    }
    for (int J = P - 1; J >= 0; J--) {
        const int ld = n - 64 * J, j0 = 64 * J;
        const double *Vp = Vb + tail_pos(n, j0, j0);
        {   // a warp's eight columns together
            double a[8];
#pragma unroll
            for (int c = 0; c < 8; c++) a[c] = 0.0;
            const double *p = Vp + (size_t)(8 * warp) * ld;
            for (int i = 64 + lane; i < ld; i += 32) {
                const double xi = sx[j0 + i];
#pragma unroll
                for (int c = 0; c < 8; c++) a[c] = fma(__ldg(p + (size_t)c * ld + i), xi, a[c]);
            }
            const double t = sum8(a, lane);
            const int c = 8 * warp + (lane >> 2);
            if ((lane & 3) == 0) {
                const double r = __ldg(di + j0 + c);
                const int e = half_exp(r);
                part[c] = SYM ? fma(-t, scale(r, e), sx[j0 + c]) : sx[j0 + c] - scale(t, -e);
            }
        }
        __syncthreads();
        // x_k = sum_i X[i][k] w_i, X = L^-1 (SYM) or U'^-1: column k of the panel's inverse
        {
            double a[8];
            const double *p = Vp + (size_t)(8 * warp) * ld + lane;
            const double w0 = part[lane], w1 = part[lane + 32];
#pragma unroll
            for (int c = 0; c < 8; c++)
                a[c] = fma(__ldg(p + (size_t)c * ld + 32), w1, __ldg(p + (size_t)c * ld) * w0);
            const double t = sum8(a, lane);
            if ((lane & 3) == 0) sx[j0 + 8 * warp + (lane >> 2)] = t;
        }
        __syncthreads();
    }
    for (int i = tid; i < nreal; i += kSolThreads) x0[(size_t)i * B + st] = sx[i];
}

size_t round256(size_t v) { return (v + 255) / 256 * 256; }

size_t fac_smem() { return 64 * kPitch * sizeof(double); }

}  // namespace

// States whose digits are held at a time: as many as fit 8 GB (at least one).
TailShape tail_shape(int n, int B, bool sym) {
    TailShape s;
    if (n <= 0) return s;
    s.n = n;
    s.P = n / 64;
    s.dense_doubles = (size_t)n * (n + 64) / 2;
    s.digit_bytes = (size_t)kDigits * kTile * s.P * (s.P - 1) / 2;
    const size_t per = 2 * (s.digit_bytes + (size_t)s.P * n * sizeof(int)) + 2 * kDigits * kTile;
    const size_t fit = std::max<size_t>(1, ((size_t)8 << 30) / per);   // then in equal shares
    const size_t parts = ((size_t)B + fit - 1) / fit;
    s.chunk = (int)(((size_t)B + parts - 1) / std::max<size_t>(1, parts));
    const size_t C = (size_t)s.chunk;
    size_t at = 0;
    auto take = [&](size_t bytes) {
        const size_t p = at;
        at += round256(bytes);
        return p;
    };
    s.dn = take(s.dense_doubles * B * sizeof(double));
    s.dv = sym ? 0 : take(s.dense_doubles * B * sizeof(double));
    s.dinv = take((size_t)n * B * sizeof(double));
    s.sf = take(s.digit_bytes * C);
    s.sl = take(s.digit_bytes * C);
    s.ef = take((size_t)s.P * n * C * sizeof(int));
    s.el = take((size_t)s.P * n * C * sizeof(int));
    s.inv = take((size_t)(sym ? 1 : 2) * kDigits * kTile * C);
    s.inve = take((size_t)(sym ? 1 : 2) * 64 * C * sizeof(int));
    s.bytes = at;
    return s;
}

int tail_allow_smem() {
    const cudaFuncAttribute a = cudaFuncAttributeMaxDynamicSharedMemorySize;
    cudaError_t e = cudaFuncSetAttribute(k_dt_update<true, 0>, a, kSmemUpd);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_dt_update<false, 0>, a, kSmemUpd);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_dt_update<false, 1>, a, kSmemUpd);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_dt_update<false, 2>, a, kSmemUpd);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_dt_solve<true>, a, 200 << 10);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_dt_solve<false>, a, 200 << 10);
    return (int)e;
}

int launch_tail_factor(const TailShape &S, int B, int BS, bool sym, void *w, int *neg, int *bad,
                       double tiny, int *status, cudaStream_t st) {
    char *base = (char *)w;
    const int n = S.n, P = S.P;
    for (int b0 = 0; b0 < B; b0 += S.chunk) {
        const int nB = std::min(S.chunk, B - b0);
        double *D = (double *)(base + S.dn) + (size_t)b0 * S.dense_doubles;
        double *V = sym ? nullptr : (double *)(base + S.dv) + (size_t)b0 * S.dense_doubles;
        double *dinv = (double *)(base + S.dinv) + (size_t)b0 * n;
        char *sf = base + S.sf, *sl = base + S.sl;
        int *ef = (int *)(base + S.ef), *el = (int *)(base + S.el);
        char *linv = base + S.inv, *uinv = linv + (size_t)kDigits * kTile * S.chunk;
        int *line = (int *)(base + S.inve), *uine = line + 64 * (size_t)S.chunk;
        for (int J = 0; J < P; J++) {
            UpdateArgs a{n, P, J, D, S.dense_doubles, dinv, sf, sl, ef, el, sf, sl, ef, el,
                         sym ? linv : uinv, sym ? line : uine, S.digit_bytes, status};
            if (J > 0) k_dt_update<true, 0><<<dim3(1, nB), kUpdThreads, kSmemUpd, st>>>(a);
            if (sym)
                k_dt_factor<true, 4><<<nB, kFacThreads, fac_smem(), st>>>(
                    n, J, D, V, S.dense_doubles, dinv, linv, line, uinv, uine, neg + b0, bad + b0, tiny);
            else
                k_dt_factor<false, 2><<<nB, kFacThreads, fac_smem(), st>>>(
                    n, J, D, V, S.dense_doubles, dinv, linv, line, uinv, uine, neg + b0, bad + b0, tiny);
            const dim3 grid((P - J) / 2, nB);   // 128-row tiles of the P - 1 - J below
            if (grid.x == 0) continue;
            if (sym) {
                k_dt_update<false, 0><<<grid, kUpdThreads, kSmemUpd, st>>>(a);
            } else {
                k_dt_update<false, 1><<<grid, kUpdThreads, kSmemUpd, st>>>(a);
                UpdateArgs u = a;
                u.D = V;
                u.sa = sl; u.sb = sf; u.xa = el; u.xb = ef;
                u.oa = sl; u.ya = el;
                u.inv = linv; u.inve = line;
                k_dt_update<false, 2><<<grid, kUpdThreads, kSmemUpd, st>>>(u);
            }
        }
    }
    return (int)cudaGetLastError();
}

int launch_tail_solve(const TailShape &S, int B, int nreal, bool sym, const void *w, double *x0,
                      cudaStream_t st) {
    const char *base = (const char *)w;
    const double *D = (const double *)(base + S.dn), *V = (const double *)(base + S.dv);
    const double *dinv = (const double *)(base + S.dinv);
    const size_t smem = ((size_t)S.n + 256) * sizeof(double);
    if (sym)
        k_dt_solve<true><<<B, kSolThreads, smem, st>>>(S.n, nreal, B, D, V, S.dense_doubles, dinv, x0);
    else
        k_dt_solve<false><<<B, kSolThreads, smem, st>>>(S.n, nreal, B, D, V, S.dense_doubles, dinv, x0);
    return (int)cudaGetLastError();
}

}  // namespace exago
