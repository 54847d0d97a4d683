"""GPU: the dense tail of the block factorisation where it has several panels and padding rows
(identity rows that pass through the digit products), an odd number of row tiles, and, of the power
flow, two and three panels, for one state, a warp and one, and more than a block of 128.
tests/test_tail_shapes.py holds that these grids have the tails listed here.

Tolerances are those of the KKT and power-flow steps (tests/test_gpu_kkt.py, test_gpu_pflow.py).
"""
import numpy as np
import pytest

from paper_2203_10587_gb300 import synth
from test_gpu_kkt import check_state, ex, kkt_inputs, run_kkt  # noqa: F401
from test_gpu_pflow import compare_step, gpu_steps

pytestmark = pytest.mark.gpu

# buses, branches: size of the tail and padding rows in it, of the KKT step and of the power flow
TAILS = {(24, 180): ((128, 32), (64, 16)), (40, 500): ((192, 32), (128, 48)),
         (56, 1200): ((256, 32), (128, 16)), (64, 1500): ((256, 0), (128, 0)),
         (72, 2000): ((320, 32), (192, 48))}


def grid(nb, nl):
    return synth.make_grid(nb + 1, nb, nl, nb // 4, max_degree=nb - 1, shunts=True)


@pytest.mark.parametrize("B", [1, 33, 130])
@pytest.mark.parametrize("nb,nl", [(24, 180), (40, 500), (56, 1200), (72, 2000)])
def test_kkt(ex, oracle_mod, nb, nl, B):  # noqa: F811
    g = grid(nb, nl)
    b = synth.random_batch(nb, g, min(B, 2), masks=True, sigma=0.9)
    refs, jval, hval, dx, dc, _ = kkt_inputs(oracle_mod, g, b, nb)
    rep = np.arange(B) % b.B
    rhs = np.random.default_rng(nb).normal(size=(B, g.n + g.m))
    net = ex.Net(g)
    sol, inertia = run_kkt(ex, net, jval[rep], hval[rep], dx[rep], dc[rep], rhs)
    for i in sorted({0, B // 2, B - 1}):
        check_state(g, refs[rep[i]], dx[rep[i]], dc[rep[i]], rhs[i], sol[i], what=f"{nb} buses [{i}]")
    assert np.all(inertia == [g.m, 0])
    net.close()


@pytest.mark.parametrize("B", [1, 33, 130])
@pytest.mark.parametrize("nb,nl", [(40, 500), (64, 1500), (72, 2000)])
def test_pflow(ex, oracle_mod, nb, nl, B):  # noqa: F811
    from oracle import kkt
    g = grid(nb, nl)
    g.Pd *= 0.3
    g.Qd *= 0.3
    types = np.ones(nb, np.int32)
    types[g.gbus] = 2
    types[g.gbus[0]] = 3
    rng = np.random.default_rng(nb)
    X = np.zeros((B, g.n))
    X[:, nb:2 * nb] = 1.0
    X[:, 2 * nb:2 * nb + g.ng] = g.Pd.sum() / g.ng
    ns = np.flatnonzero(types != 3)
    X[:, ns] += rng.normal(0.0, 0.02, (B, ns.size))
    net = ex.Net(g)
    pf = ex.exago_pf_create(net.h, types)
    try:
        xg, mg = gpu_steps(ex, net, pf, X)
    finally:
        ex.exago_pf_destroy(pf)
    onet = oracle_mod.OracleNet(g)
    for i in sorted({0, B // 2, B - 1}):
        xr, mr = kkt.pf_newton_step(oracle_mod, onet, X[i], types)
        compare_step(g, types, X[i], xg[i], xr, mg[i], mr, f"{nb} buses [{i}]")
    net.close()
