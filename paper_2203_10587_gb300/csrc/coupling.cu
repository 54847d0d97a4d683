// Coupling (ramp) rows between the states of a batch: the linear constraints that tie the
// subproblems of ExaGO's multi-stage problems together -- consecutive periods (Sec. IV, eq. (15)),
// each contingency to the base case (Sec. V-A, eq. (20)), each scenario to the base scenario
// (Sec. VI-A, eq. (31)), and any tree of them (the general form, Sec. I, eqs. (5)-(6)).  Each state
// b has a parent p(b) in the same batch (-1 for none), and the generators' real power is the
// ramp-limited quantity, one row per (b, k):
//     r[b][k] = Pg_k(x_b) - Pg_k(x_p(b)).
// The rows are linear, so C x is also their Jacobian-vector product, their Jacobian values are the
// constants +1 / -1, and they add nothing to the Lagrangian Hessian.  The transpose product is a
// gather over each state's children, in a fixed order (no atomics):
//     (C^T nu)[b][Pg_k] = [p(b) >= 0] nu[b][k] - sum over children c of b of nu[c][k].
// States with few children are summed by one thread per (state, generator); a state with more than 256
// (the base case of a contingency or scenario batch) by blocks of 4 generators whose 64 rows of threads
// take every 64th child of the list staged in shared memory and then reduce in a fixed tree, one with 9 to 256
// by blocks of 8 generators and 32 rows.
#include <cuda_runtime.h>

#include <algorithm>
#include <new>
#include <string>
#include <vector>

#include "internal.h"

struct exago_coupling {
    int B = 0, nb = 0, ng = 0, n = 0;
    bool on_device = false;
    int device = -1;
    std::vector<int> parent, child_ptr, child_idx, light, some, many;   // states by number of children
    int *d_parent = nullptr, *d_child_ptr = nullptr, *d_child_idx = nullptr;
    int *d_light = nullptr, *d_some = nullptr, *d_many = nullptr;
    void *d_mem = nullptr;
};

namespace {

using exago::set_last_error;

// A state with more children than these is reduced by blocks of kSomeCols or kManyCols generators and
// 256 / that rows of threads for its children (8 batched loads a thread cover 256 children with 32 rows).
constexpr int kSomeChildren = 8, kManyChildren = 256;
constexpr int kSomeCols = 8, kManyCols = 4;
constexpr int kWaveBlocks = 152 * 8;   // such blocks resident at once
constexpr int kMaxGridY = 65535;
// Children of a state staged in shared memory per pass.
constexpr int kStageChildren = 2048;

// Values per thread along a row: every load of a thread is issued before its first store.
constexpr int kUnroll = 4;
constexpr int kRowSpan = 256 * kUnroll;   // values of one row per block

// Block (256 threads) per (state b0 + blockIdx.y, kRowSpan generators): one subtraction per value.
// The state and its parent are uniform over the block.
__global__ void __launch_bounds__(256) k_coupling(const int *__restrict__ parent, int b0, int n,
                                                  int nb, int ng, const double *__restrict__ x,
                                                  double *__restrict__ r) {
    const int b = b0 + blockIdx.y;
    const int p = __ldg(parent + b);
    const double *xb = x + (int64_t)b * n + 2 * nb;
    const double *xp = x + (int64_t)(p < 0 ? b : p) * n + 2 * nb;
    double *rb = r + (int64_t)b * ng;
    const int k0 = blockIdx.x * kRowSpan + threadIdx.x;
    double own[kUnroll], par[kUnroll];
#pragma unroll
    for (int u = 0; u < kUnroll; u++) {
        const int k = k0 + u * 256;
        own[u] = k < ng && p >= 0 ? __ldg(xb + k) : 0.0;
        par[u] = k < ng && p >= 0 ? __ldg(xp + k) : 0.0;
    }
#pragma unroll
    for (int u = 0; u < kUnroll; u++) {
        const int k = k0 + u * 256;
        if (k < ng) rb[k] = p < 0 ? 0.0 : own[u] - par[u];
    }
}

__device__ __forceinline__ void put(double *o, double v, int accumulate) {
    *o = accumulate ? *o + v : v;
}

struct JtvArgs {
    const int *light, *some, *many, *parent, *cptr, *cidx;
    int nsome, nmany, sblocks, mblocks, lblocks, ng, accumulate;   // .blocks: blocks of one state
    const double *nu;
    double *out;
    int64_t ldo;
};

// Block g of COLS generators of state s: its children are staged in shared memory, thread row ty sums
// children ty, ty + ROWS, ... (independent loads), and the partial sums are reduced by a fixed halving tree.
template <int COLS>
__device__ __forceinline__ void sum_children(const JtvArgs &A, int s, int g, int *kids, double *part) {
    constexpr int ROWS = 256 / COLS, PITCH = COLS + 1;
    const int tid = threadIdx.x, tx = tid % COLS, ty = tid / COLS, ng = A.ng, k = g * COLS + tx;
    const int c0 = __ldg(A.cptr + s), c1 = __ldg(A.cptr + s + 1);
    double acc = 0.0;
    for (int base = c0; base < c1; base += kStageChildren) {
        const int cnt = min(kStageChildren, c1 - base);
        __syncthreads();   // the previous pass is done with kids
        for (int j = tid; j < cnt; j += 256) kids[j] = __ldg(A.cidx + base + j);
        __syncthreads();
        if (k < ng) {
#pragma unroll 8
            for (int j = ty; j < cnt; j += ROWS) acc += __ldg(A.nu + (int64_t)kids[j] * ng + k);
        }
    }
    part[ty * PITCH + tx] = acc;
    __syncthreads();
    for (int h = ROWS / 2; h >= 1; h >>= 1) {
        if (ty < h) part[ty * PITCH + tx] += part[(ty + h) * PITCH + tx];
        __syncthreads();
    }
    if (ty == 0 && k < ng) {
        const double own = __ldg(A.parent + s) >= 0 ? __ldg(A.nu + (int64_t)s * ng + k) : 0.0;
        put(A.out + (int64_t)s * A.ldo + k, own - part[tx], A.accumulate);
    }
}

// One launch for all states (256 threads a block): first those with many children, mblocks blocks of
// kManyCols generators each, then those with some, sblocks blocks of kSomeCols, then the light ones,
// lblocks blocks of kRowSpan generators each: the state's own row minus its children's, in ascending order.
// A 512-state star (many): 8 children a thread in one batch of loads; with 8 generators x 32 rows they
// were two, in a launch of its own (15.6 us the two launches).  With a dozen children a state the narrow
// blocks are twice as many for nothing: 900 buses x 4,096 states 55 us with 4 generators a block, 30 with 8;
// so are they where the wide ones fill the chip (a 512-state star of 17,500 generators 65 us, 54 wide).
// WIDE = false: light states alone, without the others' shared memory.
template <bool WIDE>
__global__ void __launch_bounds__(256, 8) k_coupling_jtv(const JtvArgs A) {
    const int tid = threadIdx.x, ng = A.ng;
    unsigned blk = blockIdx.x;   // a grid holds all
    if (WIDE) {
        __shared__ int kids[kStageChildren];
        __shared__ double part[256 + 256 / kManyCols];
        const unsigned many_blocks = A.nmany * A.mblocks, some_blocks = A.nsome * A.sblocks;
        if (blk < many_blocks) {
            sum_children<kManyCols>(A, __ldg(A.many + blk / A.mblocks), blk % A.mblocks, kids, part);
            return;
        }
        blk -= many_blocks;
        if (blk < some_blocks) {
            sum_children<kSomeCols>(A, __ldg(A.some + blk / A.sblocks), blk % A.sblocks, kids, part);
            return;
        }
        blk -= some_blocks;
    }
    const int s = __ldg(A.light + blk / A.lblocks);
    const bool own = __ldg(A.parent + s) >= 0;
    const int c0 = __ldg(A.cptr + s), c1 = __ldg(A.cptr + s + 1);
    const double *ns = A.nu + (int64_t)s * ng;
    double *os = A.out + (int64_t)s * A.ldo;
    const int k0 = (int)(blk % A.lblocks) * kRowSpan + tid;
    double v[kUnroll];
#pragma unroll
    for (int u = 0; u < kUnroll; u++) {
        const int k = k0 + u * 256;
        v[u] = own && k < ng ? __ldg(ns + k) : 0.0;
    }
    for (int c = c0; c < c1; c++) {
        const double *nc = A.nu + (int64_t)__ldg(A.cidx + c) * ng;
#pragma unroll
        for (int u = 0; u < kUnroll; u++) {
            const int k = k0 + u * 256;
            if (k < ng) v[u] -= __ldg(nc + k);
        }
    }
#pragma unroll
    for (int u = 0; u < kUnroll; u++) {
        const int k = k0 + u * 256;
        if (k < ng) put(os + k, v[u], A.accumulate);
    }
}

exago_status check_call(exago_coupling_t c) {
    if (!c) return set_last_error(EXAGO_EINVAL, "coupling is NULL");
    if (!c->on_device)
        return set_last_error(EXAGO_ESTATE, "coupling was built on a net planned without a device");
    int cur = -1;
    cudaError_t e = cudaGetDevice(&cur);
    if (e != cudaSuccess) return set_last_error(EXAGO_ECUDA, cudaGetErrorString(e));
    if (cur != c->device)
        return set_last_error(EXAGO_EINVAL, "make the coupling's device current before the call");
    return EXAGO_OK;
}

// Blocks along a row of ng values: one 256-thread block per kRowSpan values.
unsigned row_blocks(int ng) { return (unsigned)((ng + kRowSpan - 1) / kRowSpan); }

}  // namespace

extern "C" {

exago_status exago_coupling_create(exago_net_t net, int B, const int *parent,
                                   exago_coupling_t *out) {
    if (!out) return set_last_error(EXAGO_EINVAL, "out is NULL");
    *out = nullptr;
    if (!net) return set_last_error(EXAGO_EINVAL, "net is NULL");
    if (B < 0) return set_last_error(EXAGO_EINVAL, "B < 0");
    if (B > 0 && !parent) return set_last_error(EXAGO_EINVAL, "parent is NULL");
    int n = 0, meq = 0, mineq = 0;
    int64_t nnzJ = 0, nnzH = 0;
    exago_status st = exago_net_dims(net, &n, &meq, &mineq, &nnzJ, &nnzH);
    if (st != EXAGO_OK) return st;
    for (int b = 0; b < B; b++) {
        const int p = parent[b];
        if (p < -1 || p >= B || p == b)
            return set_last_error(EXAGO_EINVAL, "parent[" + std::to_string(b) + "] = " +
                                                    std::to_string(p) +
                                                    ": must be -1 or another state of the batch");
    }
    exago_coupling *c = new (std::nothrow) exago_coupling;
    if (!c) return set_last_error(EXAGO_ENOMEM, "host allocation");
    c->B = B;
    c->nb = meq / 2;
    c->n = n;
    c->ng = (n - meq) / 2;   // n = 2 nb + 2 ng, m_eq = 2 nb
    c->parent.assign(parent, parent + B);
    c->child_ptr.assign(B + 1, 0);
    for (int b = 0; b < B; b++)
        if (parent[b] >= 0) c->child_ptr[parent[b] + 1]++;
    for (int b = 0; b < B; b++) c->child_ptr[b + 1] += c->child_ptr[b];
    c->child_idx.resize(c->child_ptr[B]);
    {
        std::vector<int> fill(c->child_ptr.begin(), c->child_ptr.end() - 1);
        for (int b = 0; b < B; b++)   // ascending child order
            if (parent[b] >= 0) c->child_idx[fill[parent[b]]++] = b;
    }
    for (int b = 0; b < B; b++) {
        const int nc = c->child_ptr[b + 1] - c->child_ptr[b];
        (nc > kManyChildren ? c->many : nc > kSomeChildren ? c->some : c->light).push_back(b);
    }

    const exago::HostPlan *plan = nullptr;
    const exago::DevNet *dev = nullptr;
    if (exago::net_internal_view(net, &plan, &dev, &c->device)) {
        c->on_device = true;
        int cur = -1;
        cudaError_t e = cudaGetDevice(&cur);
        if (e != cudaSuccess || cur != c->device) {
            delete c;
            return set_last_error(e != cudaSuccess ? EXAGO_ECUDA : EXAGO_EINVAL,
                                  e != cudaSuccess ? cudaGetErrorString(e)
                                                   : "make the net's device current before the call");
        }
        // one allocation: parent [B], child_ptr [B + 1], child_idx, light, some, many
        const size_t ints = (size_t)B + (B + 1) + c->child_idx.size() + B;
        e = exago::dev_malloc(&c->d_mem, std::max<size_t>(ints, 1) * sizeof(int));
        if (e != cudaSuccess) {
            delete c;
            return set_last_error(EXAGO_ENOMEM, "cudaMalloc (coupling tables)");
        }
        std::vector<int> all;
        all.reserve(ints);
        all.insert(all.end(), c->parent.begin(), c->parent.end());
        all.insert(all.end(), c->child_ptr.begin(), c->child_ptr.end());
        all.insert(all.end(), c->child_idx.begin(), c->child_idx.end());
        all.insert(all.end(), c->light.begin(), c->light.end());
        all.insert(all.end(), c->some.begin(), c->some.end());
        all.insert(all.end(), c->many.begin(), c->many.end());
        if (!all.empty()) {
            e = cudaMemcpy(c->d_mem, all.data(), all.size() * sizeof(int), cudaMemcpyHostToDevice);
            if (e != cudaSuccess) {
                cudaFree(c->d_mem);
                delete c;
                return set_last_error(EXAGO_ECUDA, std::string("cudaMemcpy (coupling tables): ") +
                                                       cudaGetErrorString(e));
            }
        }
        int *p = (int *)c->d_mem;
        c->d_parent = p;
        p += B;
        c->d_child_ptr = p;
        p += B + 1;
        c->d_child_idx = p;
        p += c->child_idx.size();
        c->d_light = p;
        p += c->light.size();
        c->d_some = p;   // those with many follow
        p += c->some.size();
        c->d_many = p;
    }
    *out = c;
    return EXAGO_OK;
}

exago_status exago_coupling_destroy(exago_coupling_t c) {
    if (!c) return EXAGO_OK;
    if (c->d_mem) cudaFree(c->d_mem);
    delete c;
    return EXAGO_OK;
}

exago_status exago_coupling_dims(exago_coupling_t c, int *B, int64_t *rows, int64_t *nnz) {
    if (!c) return set_last_error(EXAGO_EINVAL, "coupling is NULL");
    int64_t coupled = 0;
    for (int p : c->parent) coupled += p >= 0;
    if (B) *B = c->B;
    if (rows) *rows = (int64_t)c->B * c->ng;
    if (nnz) *nnz = 2 * coupled * c->ng;
    return EXAGO_OK;
}

exago_status exago_coupling_jac_pattern(exago_coupling_t c, int64_t *rowptr, int64_t *col,
                                        double *val) {
    if (!c) return set_last_error(EXAGO_EINVAL, "coupling is NULL");
    if (!rowptr || !col) return set_last_error(EXAGO_EINVAL, "rowptr or col is NULL");
    int64_t q = 0;
    rowptr[0] = 0;
    for (int b = 0; b < c->B; b++) {
        const int p = c->parent[b];
        for (int k = 0; k < c->ng; k++) {
            if (p >= 0) {
                const int64_t cb = (int64_t)b * c->n + 2 * c->nb + k;
                const int64_t cp = (int64_t)p * c->n + 2 * c->nb + k;
                const bool self_first = cb < cp;
                col[q] = self_first ? cb : cp;
                col[q + 1] = self_first ? cp : cb;
                if (val) {
                    val[q] = self_first ? 1.0 : -1.0;
                    val[q + 1] = self_first ? -1.0 : 1.0;
                }
                q += 2;
            }
            rowptr[(int64_t)b * c->ng + k + 1] = q;
        }
    }
    return EXAGO_OK;
}

exago_status exago_eval_coupling(exago_coupling_t c, const double *x, double *r, void *stream) {
    exago_status st = check_call(c);
    if (st != EXAGO_OK) return st;
    if (c->B == 0 || c->ng == 0) return EXAGO_OK;
    if (!x || !r) return set_last_error(EXAGO_EINVAL, "x or r is NULL");
    for (int b0 = 0; b0 < c->B; b0 += kMaxGridY) {
        const int nbk = std::min(kMaxGridY, c->B - b0);
        k_coupling<<<dim3(row_blocks(c->ng), nbk), 256, 0, (cudaStream_t)stream>>>(
            c->d_parent, b0, c->n, c->nb, c->ng, x, r);
    }
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess)
        return set_last_error(EXAGO_ECUDA, std::string("coupling launch: ") + cudaGetErrorString(e));
    return EXAGO_OK;
}

exago_status exago_eval_coupling_jtv(exago_coupling_t c, const double *nu, double *out,
                                     int64_t ldo, int accumulate, void *stream) {
    exago_status st = check_call(c);
    if (st != EXAGO_OK) return st;
    if (c->B == 0 || c->ng == 0) return EXAGO_OK;
    if (!nu || !out) return set_last_error(EXAGO_EINVAL, "nu or out is NULL");
    if (ldo < c->ng) return set_last_error(EXAGO_EINVAL, "ldo < ng");
    cudaStream_t s = (cudaStream_t)stream;
    const int nlight = (int)c->light.size();
    int nsome = (int)c->some.size(), nmany = (int)c->many.size();
    const int mb = (c->ng + kManyCols - 1) / kManyCols, sb = (c->ng + kSomeCols - 1) / kSomeCols;
    const int lb = (int)row_blocks(c->ng);
    if ((int64_t)nmany * sb >= kWaveBlocks) {   // the wider blocks fill the chip: all in those
        nsome += nmany;
        nmany = 0;
    }
    // states of one launch, so that its blocks fit the grid (2^31 - 1)
    auto most = [](int blocks) { return std::max(1, (1 << 29) / blocks); };
    for (int m0 = 0, s0 = 0, l0 = 0; m0 < nmany || s0 < nsome || l0 < nlight;) {
        const int nm = std::min(most(mb), nmany - m0), ns = std::min(most(sb), nsome - s0);
        const int nl = std::min(most(lb), nlight - l0);
        const JtvArgs A{c->d_light + l0, c->d_some + s0, c->d_many + m0, c->d_parent, c->d_child_ptr,
                        c->d_child_idx, ns, nm, sb, mb, lb, c->ng, accumulate ? 1 : 0, nu, out, ldo};
        const unsigned blocks = nm * mb + ns * sb + nl * lb;
        if (nm + ns > 0) k_coupling_jtv<true><<<blocks, 256, 0, s>>>(A);
        else k_coupling_jtv<false><<<blocks, 256, 0, s>>>(A);
        m0 += nm;
        s0 += ns;
        l0 += nl;
    }
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess)
        return set_last_error(EXAGO_ECUDA, std::string("coupling transpose launch: ") +
                                               cudaGetErrorString(e));
    return EXAGO_OK;
}

}  // extern "C"
