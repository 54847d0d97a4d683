"""GPU: the dense tail of the block factorisation (the last columns of the elimination order,
factored as one dense matrix per state with exactly split products on the tensor cores), at the
sizes where it can go wrong: one panel, a panel exactly full or barely begun, padding rows, an odd
number of row tiles, batches around a warp and a block, and a state that holds a NaN.

Tolerances are those of the KKT and power-flow steps (tests/test_gpu_kkt.py, test_gpu_pflow.py): the
forward and backward bounds of a solve in another order, which do not depend on the path taken.
"""
import numpy as np
import pytest

from paper_2203_10587_gb300 import synth
from test_gpu_kkt import check_state, ex, kkt_inputs, run_kkt  # noqa: F401
from test_gpu_pflow import case, compare_step, gpu_steps

pytestmark = pytest.mark.gpu


# buses: 16 fill one panel of 64, 17 begin a second, 48 give three (an odd row tile), 100 pad
@pytest.mark.parametrize("nb,nl,B", [(5, 7, 1), (16, 24, 2), (17, 26, 33), (48, 90, 3), (100, 260, 5),
                                     (144, 420, 130)])
def test_kkt_tail_sizes(ex, oracle_mod, nb, nl, B):  # noqa: F811
    g = synth.make_grid(100 + nb, nb, nl, max(2, nb // 4), max_degree=12, shunts=True)
    b = synth.random_batch(nb, g, min(B, 3), masks=True, sigma=0.9)
    refs, jval, hval, dx, dc, rhs = kkt_inputs(oracle_mod, g, b, nb)
    rep = np.arange(B) % b.B
    rhs = np.random.default_rng(nb).normal(size=(B, rhs.shape[1]))
    net = ex.Net(g)
    sol, inertia = run_kkt(ex, net, jval[rep], hval[rep], dx[rep], dc[rep], rhs)
    for i in list(range(min(B, 5))) + [B - 1]:
        check_state(g, refs[rep[i]], dx[rep[i]], dc[rep[i]], rhs[i], sol[i], what=f"{nb} buses [{i}]")
    assert np.all(inertia == [g.m, 0])


@pytest.mark.parametrize("nb,nl,ng", [(5, 6, 2), (32, 60, 8), (33, 60, 8), (97, 250, 20)])
def test_pflow_tail_sizes(ex, oracle_mod, nb, nl, ng):  # noqa: F811
    from oracle import kkt
    g, bt, x0 = case(200 + nb, nb, nl, ng)
    rng = np.random.default_rng(nb)
    B = 4
    X = np.repeat(x0[None, :], B, axis=0)
    ns = np.flatnonzero(bt != 3)
    X[1:, ns] += rng.normal(0.0, 0.02, (B - 1, ns.size))
    net = ex.Net(g)
    pf = ex.exago_pf_create(net.h, bt)
    try:
        xg, mg = gpu_steps(ex, net, pf, X)
    finally:
        ex.exago_pf_destroy(pf)
    onet = oracle_mod.OracleNet(g)
    for i in range(B):
        xr, mr = kkt.pf_newton_step(oracle_mod, onet, X[i], bt)
        compare_step(g, bt, X[i], xg[i], xr, mg[i], mr, f"{nb} buses [{i}]")


def test_tail_nan_and_tiny_pivots_stay_in_their_state(ex, oracle_mod):  # noqa: F811
    """A NaN in one state's Hessian makes that state's solution NaN and leaves the others bit for
    bit; a state whose balance pivots vanish beside their block is counted."""
    g = synth.make_grid(7, 64, 160, 12, max_degree=12)
    b = synth.random_batch(7, g, 4)
    _, jval, hval, dx, dc, rhs = kkt_inputs(oracle_mod, g, b, 7)
    net = ex.Net(g)
    good, _ = run_kkt(ex, net, jval, hval, dx, dc, rhs)
    assert np.all(np.isfinite(good))
    bad = hval.copy()
    bad[1, :] = np.nan
    sol, inertia = run_kkt(ex, net, jval, bad, dx, dc, rhs)
    assert np.all(np.isnan(sol[1, :2 * g.nb]))
    np.testing.assert_array_equal(np.delete(sol, 1, 0), np.delete(good, 1, 0))
    # state 2 without its Jacobian and with dc far below dx: every balance pivot is below
    # 1e-13 of its block's largest entry
    j0, d0 = jval.copy(), dc.copy()
    j0[2] = 0.0
    d0[2, :2 * g.nb] = 1e-30
    _, inertia = run_kkt(ex, net, j0, hval, dx, d0, rhs)
    assert inertia[2, 0] == g.m and inertia[2, 1] == 2 * g.nb
    assert np.all(np.delete(inertia, 2, 0) == [g.m, 0])
