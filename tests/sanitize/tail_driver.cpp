// Test driver: reads "buses branches" and the branches' end buses, prints the dense tail that the
// block factorisation chooses for it (choose_tail): first tail column and padded scalar size of the
// KKT step (4 x 4 blocks) and of the power-flow step (2 x 2), and the largest batch it is taken for.  Built by tests/test_tail_shapes.py.
#include <cstdio>
#include <string>
#include <vector>

#include "../../paper_2203_10587_gb300/csrc/blockfact.h"

int main() {
    int nb, nl;
    if (scanf("%d %d", &nb, &nl) != 2) return 1;
    std::vector<int> f(nl), t(nl), ptr(nb + 1, 0), adj(nl);
    for (int l = 0; l < nl; l++)
        if (scanf("%d %d", &f[l], &t[l]) != 2 || f[l] < 0 || f[l] >= nb || t[l] < 0 || t[l] >= nb) return 1;
    for (int l = 0; l < nl; l++) ptr[f[l] + 1]++;
    for (int i = 0; i < nb; i++) ptr[i + 1] += ptr[i];
    std::vector<int> at(ptr.begin(), ptr.end() - 1);
    for (int l = 0; l < nl; l++) adj[at[f[l]]++] = t[l];
    for (int bs : {4, 2}) {
        exago::BlockSym S;
        std::string err;
        if (!exago::build_block_sym(nb, ptr.data(), adj.data(), S, err)) return 2;
        exago::choose_tail(S, bs, bs == 4);
        printf("%d %d %d\n", S.k0, S.tail_n, S.tail_most);
    }
    return 0;
}
