// Feasibility slacks of the AC-OPF model: load loss and power imbalance (ExaGO, arXiv 2203.10587,
// Sec. III, Fig. 2).  Each slack z_k >= 0 sits at one bus, in the P or the Q balance, with sign
// +1 or -1 and a linear cost: it adds sign z_k to that balance and w cost_k z_k to the objective;
// its Jacobian column is the constant sign in that row and the Hessian gets nothing.  The terms
// are applied to a finished evaluation (exago_eval_* outputs) by one launch, whose blocks do one of
// three things for one state:
//   * objective: one block sums cost_k z_k (four partial sums per thread, then a fixed 256-lane
//     tree) and adds w times the sum to f;
//   * rows: a thread per balance row with slacks adds the row's slacks in ascending slack order (the
//     same additions, in the same order, as the definition);
//   * gradient w cost_k.
// The transpose is a second kernel: sign_k v[row_k], four slacks per thread.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <new>
#include <string>
#include <vector>

#include "int_mul.cuh"
#include "internal.h"

struct exago_slack {
    int nb = 0, nz = 0;
    bool on_device = false;
    int device = -1;
    std::vector<int> bus, row, sign;
    std::vector<double> cost;
    std::vector<int> grow;              // [nz] balance row of each slack: row nb + bus
    std::vector<int> rptr, rlist, used; // CSR of the slacks by balance row; rows that have some
    int *d_int = nullptr;               // rows with slacks and the end (int2); grow and rlist as index << 1 |
                                        // negative
    double *d_cost = nullptr;
    void *d_mem = nullptr;
};

namespace {

using exago::int_mul;
using exago::mul_window;
using exago::set_last_error;

constexpr int kLanes = 256;
constexpr int kMaxGridY = 65535;
constexpr int kPart = 1024;   // gradient entries of one block

// A table entry is an index << 1 | (sign is -1).  The sign is applied to the bits: a multiplication
// by -1 takes the FP64 pipe 64 cycles a warp, which bounded the first version of both kernels.
__device__ __forceinline__ double signed_by(double v, unsigned code) {
    return __hiloint2double(__double2hiint(v) ^ (int)(code << 31), __double2loint(v));
}

// Out of line, so that no FP64 multiplication is issued for every product beside the integer one.
__device__ __noinline__ double fp_mul(double x, double y) { return x * y; }

constexpr int kStates = 4;    // states of one block of rows or gradient: they share its tables

struct SlackArgs {
    const int2 *rows;               // balance rows with slacks: row, first entry (and the end)
    const unsigned *rcode;          // slack << 1 | negative, by row
    int nused, nz, b0, nB, row_blocks, grad_blocks;
    const double *cost, *z, *obj_weight;
    double *gh, *f, *grad_z;
    int64_t ldgh;
};

// For the states b0 + kStates y ..: blocks x < kStates do the objective of one state each (OBJ), then
// row_blocks blocks the rows (ROWS) and the rest the gradient (GRAD) of all of them; an instance for each
// set of outputs, since blocks for absent ones and their registers cost a call of one output over
// 16,384 small states a third of its time (14 buses, rows alone: 9.4 us, 14.7 with them).  One launch in place of
// three, each of which waited for the one before.  Bound by the FP64 pipe (an addition a slack
// for the rows and a multiply-add for the objective: 18 us on 2,000 buses x 512 states, 10,766
// slacks a state), so the gradient's products go to the integer pipe.  69 us in three launches
// with FP64 sign and gradient products, 41 now.
template <bool OBJ, bool ROWS, bool GRAD>
__global__ void __launch_bounds__(kLanes) k_slack_apply(const SlackArgs A) {
    __shared__ double part[OBJ ? kLanes : 1];
    constexpr int S = OBJ || ROWS ? kStates : 1;   // the gradient alone has few blocks otherwise
    const int tid = threadIdx.x, bs = A.b0 + S * blockIdx.y, nz = A.nz;
    const int ns = min(S, A.b0 + A.nB - bs);
    int x = blockIdx.x;
    if (OBJ && x < kStates) {
        if (x >= ns) return;
        const int b = bs + x;
        const double *zb = A.z + (int64_t)b * nz;
        double a0 = 0.0, a1 = 0.0, a2 = 0.0, a3 = 0.0;
        int k = tid;
        for (; k + 3 * kLanes < nz; k += 4 * kLanes) {
            a0 = fma(__ldg(A.cost + k), __ldg(zb + k), a0);
            a1 = fma(__ldg(A.cost + k + kLanes), __ldg(zb + k + kLanes), a1);
            a2 = fma(__ldg(A.cost + k + 2 * kLanes), __ldg(zb + k + 2 * kLanes), a2);
            a3 = fma(__ldg(A.cost + k + 3 * kLanes), __ldg(zb + k + 3 * kLanes), a3);
        }
        for (; k < nz; k += kLanes) a0 = fma(__ldg(A.cost + k), __ldg(zb + k), a0);
        part[tid] = (a0 + a1) + (a2 + a3);
        __syncthreads();
        for (int h = kLanes / 2; h > 0; h >>= 1) {
            if (tid < h) part[tid] += part[tid + h];
            __syncthreads();
        }
        if (tid == 0) A.f[b] = fma(A.obj_weight ? __ldg(A.obj_weight + b) : 1.0, part[0], A.f[b]);
        return;
    }
    if (OBJ) x -= kStates;
    if (ROWS && x < A.row_blocks) {
        const int j = x * kLanes + tid;
        if (j >= A.nused) return;
        const int2 row = __ldg(A.rows + j);
        const int q1 = __ldg(&A.rows[j + 1].y);
        double *g = A.gh + (int64_t)bs * A.ldgh + row.x;
        const double *zb = A.z + (int64_t)bs * nz;
        double v[kStates];
#pragma unroll
        for (int t = 0; t < kStates; t++) v[t] = t < ns ? g[t * A.ldgh] : 0.0;
        for (int q = row.y; q < q1; q += 2) {        // two entries' loads in flight
            const unsigned c0 = __ldg(A.rcode + q), c1 = q + 1 < q1 ? __ldg(A.rcode + q + 1) : 0;
            double t0[kStates], t1[kStates];
#pragma unroll
            for (int t = 0; t < kStates; t++) {
                t0[t] = t < ns ? __ldg(zb + (int64_t)t * nz + (c0 >> 1)) : 0.0;
                t1[t] = t < ns && q + 1 < q1 ? __ldg(zb + (int64_t)t * nz + (c1 >> 1)) : 0.0;
            }
#pragma unroll
            for (int t = 0; t < kStates; t++) v[t] += signed_by(t0[t], c0);
            if (q + 1 < q1)
#pragma unroll
                for (int t = 0; t < kStates; t++) v[t] += signed_by(t1[t], c1);
        }
#pragma unroll
        for (int t = 0; t < kStates; t++)
            if (t < ns) g[t * A.ldgh] = v[t];
        return;
    }
    if (!GRAD) return;
    if (ROWS) x -= A.row_blocks;
#pragma unroll
    for (int u = 0; u < kPart / kLanes; u++) {
        const int k = x * kPart + u * kLanes + tid;
        if (k >= nz) break;
        const double c = __ldg(A.cost + k);
        for (int t = 0; t < ns; t++) {
            const double w = A.obj_weight ? __ldg(A.obj_weight + bs + t) : 1.0;
            // alone, the FP64 pipe is free for the products (integer ones take 1.25 times as long)
            if (!OBJ && !ROWS) A.grad_z[(int64_t)(bs + t) * nz + k] = w * c;
            else A.grad_z[(int64_t)(bs + t) * nz + k] = mul_window(w) && mul_window(c) ? int_mul(w, c)
                                                                                       : fp_mul(w, c);
        }
    }
}

// out[b][k] = sign_k v[b][row_k]: every load of a thread's U slacks before its first store (four, or one
// where a state has no more slacks than a block has threads).
template <int U>
__global__ void __launch_bounds__(256) k_slack_jtv(const unsigned *__restrict__ gcode, int nz, int b0,
                                                   const double *__restrict__ v, int64_t ldv,
                                                   double *__restrict__ out) {
    const int b = b0 + blockIdx.y, k0 = blockIdx.x * (256 * U) + threadIdx.x;
    const double *vb = v + (int64_t)b * ldv;
    double *ob = out + (int64_t)b * nz;
    unsigned c[U];
    double t[U];
#pragma unroll
    for (int u = 0; u < U; u++) c[u] = k0 + u * 256 < nz ? __ldg(gcode + k0 + u * 256) : 0;
#pragma unroll
    for (int u = 0; u < U; u++) t[u] = k0 + u * 256 < nz ? __ldg(vb + (c[u] >> 1)) : 0.0;
#pragma unroll
    for (int u = 0; u < U; u++)
        if (k0 + u * 256 < nz) ob[k0 + u * 256] = signed_by(t[u], c[u]);
}

exago_status check_call(exago_slack_t s, const exago_batch *bt) {
    if (!s) return set_last_error(EXAGO_EINVAL, "slack set is NULL");
    if (!s->on_device)
        return set_last_error(EXAGO_ESTATE, "slack set was built on a net planned without a device");
    if (!bt) return set_last_error(EXAGO_EINVAL, "batch is NULL");
    if (bt->B < 0) return set_last_error(EXAGO_EINVAL, "batch B < 0");
    int cur = -1;
    cudaError_t e = cudaGetDevice(&cur);
    if (e != cudaSuccess) return set_last_error(EXAGO_ECUDA, cudaGetErrorString(e));
    if (cur != s->device)
        return set_last_error(EXAGO_EINVAL, "make the slack set's device current before the call");
    return EXAGO_OK;
}

}  // namespace

extern "C" {

exago_status exago_slack_create(exago_net_t net, int nz, const int *bus, const int *row,
                                const int *sign, const double *cost, exago_slack_t *out) {
    if (!out) return set_last_error(EXAGO_EINVAL, "out is NULL");
    *out = nullptr;
    if (!net) return set_last_error(EXAGO_EINVAL, "net is NULL");
    if (nz < 0) return set_last_error(EXAGO_EINVAL, "nz < 0");
    if (nz > 0 && (!bus || !row || !sign || !cost))
        return set_last_error(EXAGO_EINVAL, "bus, row, sign or cost is NULL");
    int n = 0, meq = 0, mineq = 0;
    int64_t nnzJ = 0, nnzH = 0;
    exago_status st = exago_net_dims(net, &n, &meq, &mineq, &nnzJ, &nnzH);
    if (st != EXAGO_OK) return st;
    const int nb = meq / 2;
    for (int k = 0; k < nz; k++) {
        if (bus[k] < 0 || bus[k] >= nb || (row[k] != 0 && row[k] != 1) ||
            (sign[k] != 1 && sign[k] != -1) || !std::isfinite(cost[k]))
            return set_last_error(EXAGO_EINVAL, "slack " + std::to_string(k) +
                                                    ": bus out of range, row not 0 or 1, sign "
                                                    "not +1 or -1, or cost not finite");
    }
    exago_slack *s = new (std::nothrow) exago_slack;
    if (!s) return set_last_error(EXAGO_ENOMEM, "host allocation");
    s->nb = nb;
    s->nz = nz;
    s->bus.assign(bus, bus + nz);
    s->row.assign(row, row + nz);
    s->sign.assign(sign, sign + nz);
    s->cost.assign(cost, cost + nz);
    s->grow.resize(nz);
    s->rptr.assign(2 * nb + 1, 0);
    for (int k = 0; k < nz; k++) {
        s->grow[k] = row[k] * nb + bus[k];
        s->rptr[s->grow[k] + 1]++;
    }
    for (int r = 0; r < 2 * nb; r++) s->rptr[r + 1] += s->rptr[r];
    s->rlist.resize(nz);
    {
        std::vector<int> fill(s->rptr.begin(), s->rptr.end() - 1);
        for (int k = 0; k < nz; k++) s->rlist[fill[s->grow[k]]++] = k;   // ascending k per row
    }
    for (int r = 0; r < 2 * nb; r++)
        if (s->rptr[r + 1] > s->rptr[r]) s->used.push_back(r);

    const exago::HostPlan *plan = nullptr;
    const exago::DevNet *dev = nullptr;
    if (exago::net_internal_view(net, &plan, &dev, &s->device)) {
        s->on_device = true;
        int cur = -1;
        cudaError_t e = cudaGetDevice(&cur);
        if (e != cudaSuccess || cur != s->device) {
            delete s;
            return set_last_error(e != cudaSuccess ? EXAGO_ECUDA : EXAGO_EINVAL,
                                  e != cudaSuccess ? cudaGetErrorString(e)
                                                   : "make the net's device current before the call");
        }
        std::vector<int> ints;
        for (int r : s->used)
            for (int v : {r, s->rptr[r]}) ints.push_back(v);
        for (int v : {0, nz}) ints.push_back(v);   // the rows' end
        auto code = [&](int index, int k) { return (int)((unsigned)index << 1 | (unsigned)(s->sign[k] < 0)); };
        for (int k = 0; k < nz; k++) ints.push_back(code(s->grow[k], k));
        for (int k : s->rlist) ints.push_back(code(k, k));
        const size_t ibytes = (ints.size() * sizeof(int) + 255) / 256 * 256;
        const size_t bytes = ibytes + std::max<size_t>((size_t)nz, 1) * sizeof(double);
        e = exago::dev_malloc(&s->d_mem, bytes);
        if (e != cudaSuccess) {
            delete s;
            return set_last_error(EXAGO_ENOMEM, "cudaMalloc (slack tables)");
        }
        s->d_int = (int *)s->d_mem;
        s->d_cost = (double *)((char *)s->d_mem + ibytes);
        e = cudaMemcpy(s->d_int, ints.data(), ints.size() * sizeof(int), cudaMemcpyHostToDevice);
        if (e == cudaSuccess && nz > 0)
            e = cudaMemcpy(s->d_cost, s->cost.data(), nz * sizeof(double), cudaMemcpyHostToDevice);
        if (e != cudaSuccess) {
            cudaFree(s->d_mem);
            delete s;
            return set_last_error(EXAGO_ECUDA, std::string("cudaMemcpy (slack tables): ") +
                                                   cudaGetErrorString(e));
        }
    }
    *out = s;
    return EXAGO_OK;
}

exago_status exago_slack_destroy(exago_slack_t s) {
    if (!s) return EXAGO_OK;
    if (s->d_mem) cudaFree(s->d_mem);
    delete s;
    return EXAGO_OK;
}

exago_status exago_slack_pattern(exago_slack_t s, int64_t *rows, double *vals) {
    if (!s) return set_last_error(EXAGO_EINVAL, "slack set is NULL");
    if (s->nz > 0 && (!rows || !vals)) return set_last_error(EXAGO_EINVAL, "rows or vals is NULL");
    for (int k = 0; k < s->nz; k++) {
        rows[k] = s->grow[k];
        vals[k] = s->sign[k];
    }
    return EXAGO_OK;
}

exago_status exago_eval_slack(exago_slack_t s, const exago_batch *bt, const double *z, double *gh,
                              int64_t ldgh, double *f, double *grad_z) {
    exago_status st = check_call(s, bt);
    if (st != EXAGO_OK || bt->B == 0 || s->nz == 0) return st;
    if (!z) return set_last_error(EXAGO_EINVAL, "z is NULL");
    if (gh && ldgh < 2 * s->nb) return set_last_error(EXAGO_EINVAL, "ldgh < 2 nb");
    cudaStream_t stream = (cudaStream_t)bt->stream;
    const int nused = (int)s->used.size();
    SlackArgs A{(const int2 *)s->d_int, (const unsigned *)s->d_int + 2 * (nused + 1) + s->nz, nused,
                s->nz, 0, 0, gh ? (nused + kLanes - 1) / kLanes : 0,
                grad_z ? (s->nz + kPart - 1) / kPart : 0,
                s->d_cost, z, bt->obj_weight, gh, f, grad_z, ldgh};
    auto launch = [&](const SlackArgs &L) {
        for (int b0 = 0; b0 < bt->B && (L.gh || L.f || L.grad_z); b0 += kMaxGridY) {
            SlackArgs C = L;
            C.b0 = b0;
            C.nB = std::min(kMaxGridY, bt->B - b0);
            const int S = C.f || C.gh ? kStates : 1;
            const dim3 grid((C.f ? S : 0) + C.row_blocks + C.grad_blocks, (C.nB + S - 1) / S);
            if (grid.x == 0) continue;   // rows alone, and none has a slack
            switch ((C.f ? 1 : 0) | (C.gh ? 2 : 0) | (C.grad_z ? 4 : 0)) {
                case 1: k_slack_apply<true, false, false><<<grid, kLanes, 0, stream>>>(C); break;
                case 2: k_slack_apply<false, true, false><<<grid, kLanes, 0, stream>>>(C); break;
                case 3: k_slack_apply<true, true, false><<<grid, kLanes, 0, stream>>>(C); break;
                case 4: k_slack_apply<false, false, true><<<grid, kLanes, 0, stream>>>(C); break;
                case 5: k_slack_apply<true, false, true><<<grid, kLanes, 0, stream>>>(C); break;
                case 6: k_slack_apply<false, true, true><<<grid, kLanes, 0, stream>>>(C); break;
                default: k_slack_apply<true, true, true><<<grid, kLanes, 0, stream>>>(C); break;
            }
        }
    };
    const uintptr_t span = (uintptr_t)bt->B * s->nz * sizeof(double), dist = (uintptr_t)grad_z - (uintptr_t)z;
    if (grad_z && (gh || f) && (dist < span || -dist < span)) {   // the gradient replaces z: last
        SlackArgs G = A;
        G.gh = G.f = nullptr;
        G.row_blocks = 0;
        A.grad_z = nullptr;
        A.grad_blocks = 0;
        launch(A);
        launch(G);
    } else launch(A);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess)
        return set_last_error(EXAGO_ECUDA, std::string("slack launch: ") + cudaGetErrorString(e));
    return EXAGO_OK;
}

exago_status exago_eval_all_slack(exago_net_t net, const exago_batch *bt, exago_slack_t s,
                                  const double *z, double *f, double *grad, double *gh,
                                  double *jval, double *hval, double *grad_z) {
    exago_status st = check_call(s, bt);
    if (st != EXAGO_OK || bt->B == 0) return st;
    int n = 0, meq = 0, mineq = 0;
    if ((st = exago_net_dims(net, &n, &meq, &mineq, nullptr, nullptr)) != EXAGO_OK) return st;
    if (meq / 2 != s->nb) return set_last_error(EXAGO_EINVAL, "slack set of another grid");
    // the evaluation, then the slack kernels on the same stream (bit for bit the two calls)
    if ((st = exago_eval_all(net, bt, f, grad, gh, jval, hval)) != EXAGO_OK) return st;
    return exago_eval_slack(s, bt, z, gh, meq + mineq, f, grad_z);
}

exago_status exago_eval_slack_jtv(exago_slack_t s, const exago_batch *bt, const double *v,
                                  int64_t ldv, double *out) {
    exago_status st = check_call(s, bt);
    if (st != EXAGO_OK || bt->B == 0 || s->nz == 0) return st;
    if (!v || !out) return set_last_error(EXAGO_EINVAL, "v or out is NULL");
    if (ldv < 2 * s->nb) return set_last_error(EXAGO_EINVAL, "ldv < 2 nb");
    for (int b0 = 0; b0 < bt->B; b0 += kMaxGridY) {
        const int nB = std::min(kMaxGridY, bt->B - b0);
        const unsigned *code = (const unsigned *)s->d_int + 2 * (s->used.size() + 1);
        const cudaStream_t cs = (cudaStream_t)bt->stream;
        if (s->nz <= 256) k_slack_jtv<1><<<dim3(1, nB), 256, 0, cs>>>(code, s->nz, b0, v, ldv, out);
        else k_slack_jtv<4><<<dim3((s->nz + 1023) / 1024, nB), 256, 0, cs>>>(code, s->nz, b0, v, ldv, out);
    }
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess)
        return set_last_error(EXAGO_ECUDA, std::string("slack transpose launch: ") +
                                               cudaGetErrorString(e));
    return EXAGO_OK;
}

}  // extern "C"
