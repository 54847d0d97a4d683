// Host symbolic factorisation of the bus graph for the batched block factorisation (blockfact.h).
//
// Ordering: minimum degree on the elimination graph.  Repeatedly the uneliminated bus of least
// current degree (lowest index on ties) is eliminated and its neighbours become a clique; the
// neighbour set at elimination is the block structure of its factor column.  The graphs here are
// sparse (degree <= 8 before fill), so plain sorted adjacency vectors merged on each elimination
// are enough.  Plain host code (no CUDA calls): the host tests build it with the address and
// undefined-behaviour sanitizers.
#include <algorithm>
#include <climits>
#include <cstdio>
#include <set>

#include "blockfact.h"

namespace exago {

namespace {

// out = (a U b) \ {x, y}, a and b sorted ascending without duplicates.
void merge_without(const std::vector<int> &a, const std::vector<int> &b, int x, int y,
                   std::vector<int> &out) {
    out.clear();
    out.reserve(a.size() + b.size());
    size_t i = 0, j = 0;
    while (i < a.size() || j < b.size()) {
        int v;
        if (j >= b.size() || (i < a.size() && a[i] < b[j])) v = a[i++];
        else if (i >= a.size() || b[j] < a[i]) v = b[j++];
        else { v = a[i]; i++; j++; }
        if (v != x && v != y) out.push_back(v);
    }
}

// The levels' columns, targets and longest sums below k0.
void sparse_levels(BlockSym &S) {
    S.sp_cols.assign(S.nlevels, 0);
    S.sp_tgts = S.sp_pairs = S.sp_rows = S.sp_colblks = S.sp_cols;
    for (int l = 0; l < S.nlevels; l++) {
        for (int c = S.lvl_colptr[l]; c < S.lvl_colptr[l + 1]; c++) {
            const int k = S.lvl_cols[c];
            if (k >= S.k0) break;   // ascending within a level: the columns below k0 come first
            S.sp_cols[l]++;
            S.sp_tgts[l] += (int)(S.colptr[k + 1] - S.colptr[k]);
            S.sp_rows[l] = std::max(S.sp_rows[l], (int)(S.rowptr[k + 1] - S.rowptr[k]));
            S.sp_colblks[l] = std::max(S.sp_colblks[l], (int)(S.colptr[k + 1] - S.colptr[k]) - 1);
        }
        for (int t = S.lvl_tptr[l]; t < S.lvl_tptr[l] + S.sp_tgts[l]; t++)
            S.sp_pairs[l] = std::max(S.sp_pairs[l], (int)(S.tptr[t + 1] - S.tptr[t]));
    }
}

// The largest batch for which the tail is faster than the same columns level by level.  The tail saves
// launches and the chains of narrow levels, but a 64-column panel costs its 64 dense pivots however
// few of its blocks the factor has, so small grids in large batches are faster without it.  Fitted to 39
// grids of 3 to 300 buses and 1.35 to 3 branches a bus x 1 to 16,384 states, both ways (us, c the
// columns of the tail): level by level per state 1.15e-4 a block product + 4.9e-4 a block, and 34
// a level + 0.028 a product + 0.46 a block with 128 states; panels per state 0.33 each + 0.104 a tile
// product, and 150 each with 128 states, up to which an SM has one block (2 x 2 blocks, LU: the second
// set).  The choice is at most 7% off the better one on any of them.  Without the line (tail, level by level):
// KKT 14 buses x 4,096 1,463 and 303 us, 57 x 16,384 6,899 and 2,803, 118 x 512 634 and 906; power
// flow 57 buses x 2,048 1,369 and 413, 300 x 512 737 and 1,141.
int tail_most_states(const BlockSym &S, int BS, double products) {
    const double P = S.tail_n / 64, tiles = P * (P + 1) * (P + 2) / 6 - P;
    int levels = 0;
    for (int k = 0; k < S.k0; k++) levels = std::max(levels, S.level[k] + 1);
    levels = S.nlevels - levels;
    const double blocks = (double)(S.nblk - S.colptr[S.k0]);
    const bool kkt = BS == 4;
    const double state = kkt ? 1.15e-4 * products + 4.9e-4 * blocks - 0.33 * P - 0.104 * tiles
                             : 2.9e-5 * products + 1.4e-4 * blocks - 0.55 * P - 0.19 * tiles;
    const double fixed = kkt ? 34.0 * levels + 0.028 * products + 0.46 * blocks - 150.0 * P
                             : 21.0 * levels + 0.008 * products + 0.11 * blocks - 160.0 * P;
    if (fixed < 0) return state < 0 ? 0 : INT_MAX;
    return state < 0 ? (int)std::min(1e9, 128.0 + fixed / -state) : INT_MAX;
}

}  // namespace

bool build_block_sym(int nb, const int *adj_ptr, const int *adj, BlockSym &S, std::string &err) {
    S = BlockSym();
    if (nb < 1) { err = "empty graph"; return false; }
    S.nb = nb;
    std::vector<std::vector<int>> g(nb);
    for (int v = 0; v < nb; v++) {
        for (int q = adj_ptr[v]; q < adj_ptr[v + 1]; q++) {
            const int u = adj[q];
            if (u < 0 || u >= nb) { err = "adjacency index out of range"; return false; }
            if (u != v) { g[v].push_back(u); g[u].push_back(v); }
        }
    }
    for (auto &a : g) {
        std::sort(a.begin(), a.end());
        a.erase(std::unique(a.begin(), a.end()), a.end());
    }
    const std::vector<std::vector<int>> own = g;   // A's pattern
    // minimum degree, lowest index on ties
    std::set<std::pair<int, int>> queue;
    for (int v = 0; v < nb; v++) queue.insert({(int)g[v].size(), v});
    std::vector<std::vector<int>> colbus(nb);   // neighbour buses of the k-th eliminated bus
    S.perm.resize(nb);
    S.iperm.assign(nb, -1);
    std::vector<int> tmp;
    for (int k = 0; k < nb; k++) {
        const int v = queue.begin()->second;
        queue.erase(queue.begin());
        S.perm[k] = v;
        S.iperm[v] = k;
        const std::vector<int> N = g[v];
        for (int u : N) {
            queue.erase({(int)g[u].size(), u});
            merge_without(g[u], N, u, v, tmp);
            g[u].swap(tmp);
            queue.insert({(int)g[u].size(), u});
        }
        colbus[k] = N;
        g[v].clear();
        g[v].shrink_to_fit();
    }
    // factor structure in elimination index space
    S.colptr.assign(nb + 1, 0);
    for (int k = 0; k < nb; k++) S.colptr[k + 1] = S.colptr[k] + 1 + (int64_t)colbus[k].size();
    S.nblk = S.colptr[nb];
    if (S.nblk > 0x7fffffff) { err = "factor too large"; return false; }
    S.rowidx.resize(S.nblk);
    std::vector<int64_t> rowcount(nb + 1, 0);
    for (int k = 0; k < nb; k++) {
        std::vector<int> rows;
        rows.reserve(colbus[k].size());
        for (int u : colbus[k]) rows.push_back(S.iperm[u]);
        std::sort(rows.begin(), rows.end());
        int64_t p = S.colptr[k];
        S.rowidx[p++] = k;
        for (int i : rows) {
            if (i <= k) { err = "elimination order inconsistent"; return false; }
            S.rowidx[p++] = i;
            rowcount[i + 1]++;
        }
        colbus[k].clear();
        colbus[k].shrink_to_fit();
    }
    // row structure (ascending K within each row: columns are visited in order)
    S.rowptr.assign(nb + 1, 0);
    for (int i = 0; i < nb; i++) S.rowptr[i + 1] = S.rowptr[i] + rowcount[i + 1];
    S.rowblk.resize(S.rowptr[nb]);
    S.rowcol.resize(S.rowptr[nb]);
    {
        std::vector<int64_t> fill(S.rowptr.begin(), S.rowptr.end() - 1);
        for (int k = 0; k < nb; k++)
            for (int64_t p = S.colptr[k] + 1; p < S.colptr[k + 1]; p++) {
                const int i = S.rowidx[p];
                S.rowblk[fill[i]] = (int)p;
                S.rowcol[fill[i]] = k;
                fill[i]++;
            }
    }
    // elimination tree and levels (a child precedes its parent in the order)
    S.parent.assign(nb, -1);
    S.level.assign(nb, 0);
    for (int k = 0; k < nb; k++) {
        if (S.colptr[k + 1] - S.colptr[k] > 1) S.parent[k] = S.rowidx[S.colptr[k] + 1];
        const int p = S.parent[k];
        if (p >= 0 && S.level[p] < S.level[k] + 1) S.level[p] = S.level[k] + 1;
    }
    S.nlevels = 0;
    for (int k = 0; k < nb; k++) S.nlevels = std::max(S.nlevels, S.level[k] + 1);
    S.lvl_colptr.assign(S.nlevels + 1, 0);
    for (int k = 0; k < nb; k++) S.lvl_colptr[S.level[k] + 1]++;
    for (int l = 0; l < S.nlevels; l++) S.lvl_colptr[l + 1] += S.lvl_colptr[l];
    S.lvl_cols.resize(nb);
    {
        std::vector<int> fill(S.lvl_colptr.begin(), S.lvl_colptr.end() - 1);
        for (int k = 0; k < nb; k++) S.lvl_cols[fill[S.level[k]]++] = k;
    }
    // targets (every block), grouped by level, and their update pairs (two passes: count, fill)
    S.lvl_tptr.assign(S.nlevels + 1, 0);
    S.tgt_blk.clear();
    S.tgt_diag.clear();
    S.tgt_blk.reserve(S.nblk);
    S.tgt_diag.reserve(S.nblk);
    for (int l = 0; l < S.nlevels; l++) {
        for (int c = S.lvl_colptr[l]; c < S.lvl_colptr[l + 1]; c++) {
            const int J = S.lvl_cols[c];
            for (int64_t p = S.colptr[J]; p < S.colptr[J + 1]; p++) {
                S.tgt_blk.push_back((int)p);
                S.tgt_diag.push_back((int)S.colptr[J]);
            }
        }
        S.lvl_tptr[l + 1] = (int)S.tgt_blk.size();
    }
    const int64_t ntgt = (int64_t)S.tgt_blk.size();
    std::vector<int> tgt_of_blk(S.nblk);
    for (int64_t t = 0; t < ntgt; t++) tgt_of_blk[S.tgt_blk[t]] = (int)t;
    std::vector<int64_t> count(ntgt + 1, 0);
    std::vector<int64_t> pos_of_row(nb, -1);
    auto for_pairs = [&](auto &&emit) {
        for (int J = 0; J < nb; J++) {
            for (int64_t p = S.colptr[J]; p < S.colptr[J + 1]; p++) pos_of_row[S.rowidx[p]] = p;
            for (int64_t r = S.rowptr[J]; r < S.rowptr[J + 1]; r++) {
                const int K = S.rowcol[r];
                const int pJK = S.rowblk[r];
                // blocks (I, K) of column K with I >= J: from (J, K) on
                for (int64_t q = pJK; q < S.colptr[K + 1]; q++) {
                    const int64_t pIJ = pos_of_row[S.rowidx[q]];
                    if (pIJ < 0) return false;   // would be a fill the structure lacks
                    emit(tgt_of_blk[pIJ], (int)q, pJK);
                }
            }
            for (int64_t p = S.colptr[J]; p < S.colptr[J + 1]; p++) pos_of_row[S.rowidx[p]] = -1;
        }
        return true;
    };
    if (!for_pairs([&](int64_t t, int, int) { count[t + 1]++; })) {
        err = "symbolic factorisation missed a fill block";
        return false;
    }
    S.tptr.assign(ntgt + 1, 0);
    for (int64_t t = 0; t < ntgt; t++) S.tptr[t + 1] = S.tptr[t] + count[t + 1];
    S.pairs.resize(S.tptr[ntgt]);
    {
        std::vector<int64_t> fill(S.tptr.begin(), S.tptr.end() - 1);
        for_pairs([&](int64_t t, int q, int pJK) {
            S.pairs[fill[t]++] = make_int2(q, pJK);
        });
    }
    S.flops_factor_per_block = (double)S.pairs.size();
    S.tgt_fill.assign(ntgt, 0);
    for (int k = 0; k < nb; k++)
        for (int64_t p = S.colptr[k]; p < S.colptr[k + 1]; p++) {
            const int u = S.perm[S.rowidx[p]], v = S.perm[k];
            if (u == v || std::binary_search(own[u].begin(), own[u].end(), v)) S.own_blk.push_back((int)p);
            else S.tgt_fill[tgt_of_blk[p]] = 1;
        }
    S.k0 = nb;
    sparse_levels(S);
    return true;
}

// The tail that costs least, by what the parts took on GB300 with 128 states: a level of the
// sparse part 20 us (its launches), a thousand of its 4 x 4 block products 16 us (2 x 2: 4 us),
// a panel of 64 columns 60 us (its launches and 64 dependent pivots), a dense 64 x 64 x 64 tile
// product 3.5 us.
void choose_tail(BlockSym &S, int BS, bool sym) {
    const int nb = S.nb, step = 64 / BS;
    std::vector<double> pairs(nb + 1, 0.0);   // block products whose inner column is below k
    std::vector<int> levels(nb + 1, 0);
    for (int k = 0; k < nb; k++) {
        const double d = (double)(S.colptr[k + 1] - S.colptr[k] - 1);
        pairs[k + 1] = pairs[k] + d * (d + 1) / 2;
        levels[k + 1] = std::max(levels[k], S.level[k] + 1);
    }
    const double side = sym ? 1.0 : 2.0, pair = (BS == 4 ? 0.016 : 0.004) * side;
    auto sparse = [&](int k0) { return 20.0 * levels[k0] + pair * pairs[k0]; };
    double best = sparse(nb);
    int best_k0 = nb, best_n = 0;
    for (int P = 1;; P++) {   // at most 384 panels: the sweeps hold a state's vector in shared memory
        const int R = std::min(nb, P * step);
        const double dense = P * (P + 1.0) * (P + 2.0) / 6.0 * side;
        const double cost = sparse(nb - R) + 60.0 * P + 3.5 * dense;
        if (cost < best) {
            best = cost;
            best_k0 = nb - R;
            best_n = 64 * P;
        }
        if (R == nb || P == 384 || 60.0 * P + 3.5 * dense > best) break;
    }
    if (best_n == 0) return;
    const int k0 = best_k0, R = nb - k0;
    S.k0 = k0;
    S.tail_n = best_n;
    S.tail_most = tail_most_states(S, BS, pairs[nb] - pairs[k0]);
    if (S.tail_most == 0) {
        S.k0 = nb;
        S.tail_n = 0;
        return;
    }
    sparse_levels(S);
    std::vector<int> col_of_blk(S.nblk);
    for (int k = 0; k < nb; k++)
        for (int64_t p = S.colptr[k]; p < S.colptr[k + 1]; p++) col_of_blk[p] = k;
    const int64_t ntgt = (int64_t)S.tgt_blk.size();
    S.tail_q1.resize(ntgt);
    S.tail_tgt.assign((size_t)R * (R + 1) / 2, -1);
    for (int64_t t = 0; t < ntgt; t++) {
        const int p = S.tgt_blk[t], J = col_of_blk[p];
        int64_t q = S.tptr[t + 1];
        if (J >= k0) {   // pairs ascend in K
            q = S.tptr[t];
            while (q < S.tptr[t + 1] && col_of_blk[S.pairs[q].y] < k0) q++;
            const int64_t i = S.rowidx[p] - k0, j = J - k0;
            S.tail_tgt[(size_t)(i * (i + 1) / 2 + j)] = (int)t;
        }
        S.tail_q1[t] = q;
    }
    S.tail_r1.resize(nb);
    for (int i = 0; i < nb; i++) {
        int64_t r = S.rowptr[i];
        while (r < S.rowptr[i + 1] && S.rowcol[r] < k0) r++;
        S.tail_r1[i] = r;
    }
}

}  // namespace exago
