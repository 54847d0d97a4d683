"""GPU: KKT and power-flow steps with a workspace that holds the whole factor arrays but not the
dense last columns beside them (the size that the calls need without those): accepted, and within
the steps' own bounds (tests/test_gpu_kkt.py, test_gpu_pflow.py); one byte less is refused.
"""
import numpy as np
import pytest

from paper_2203_10587_gb300 import synth
from test_gpu_kkt import check_state, ex, kkt_inputs, run_kkt  # noqa: F401
from test_gpu_pflow import case, compare_step, gpu_steps

pytestmark = pytest.mark.gpu


def r256(v):
    return (v + 255) // 256 * 256


def blocks_of(ex, net):
    k = ex.exago_kkt_create(net.h)
    blocks = ex.exago_kkt_info(k)["blocks"]
    ex.exago_kkt_destroy(k)
    return blocks


@pytest.mark.parametrize("nb,nl,B", [(30, 41, 37), (200, 260, 5), (40, 500, 130)])
def test_kkt(ex, oracle_mod, nb, nl, B):  # noqa: F811
    import torch
    g = synth.make_grid(nb + 1, nb, nl, nb // 4, max_degree=max(12, nb - 1) if nl > 2 * nb else 8, shunts=True)
    b = synth.random_batch(nb, g, min(B, 2), masks=True, sigma=0.9)
    refs, jval, hval, dx, dc, _ = kkt_inputs(oracle_mod, g, b, nb)
    rep = np.arange(B) % b.B
    rhs = np.random.default_rng(nb).normal(size=(B, g.n + g.m))
    net = ex.Net(g)
    size = 2 * r256(blocks_of(ex, net) * 128 * B) + r256(nb * 32 * B) + r256(8 * B)
    ws = torch.empty(size, dtype=torch.uint8, device="cuda")
    sol, inertia = run_kkt(ex, net, jval[rep], hval[rep], dx[rep], dc[rep], rhs, workspace=ws)
    for i in sorted({0, B // 2, B - 1}):
        check_state(g, refs[rep[i]], dx[rep[i]], dc[rep[i]], rhs[i], sol[i], what=f"{nb} buses [{i}]")
    assert np.all(inertia == [g.m, 0])
    with pytest.raises(Exception, match="workspace"):
        run_kkt(ex, net, jval[rep], hval[rep], dx[rep], dc[rep], rhs, workspace=ws[:size - 1])
    net.close()


@pytest.mark.parametrize("nb,nl,ng", [(30, 41, 6), (300, 389, 60)])
def test_pflow(ex, oracle_mod, nb, nl, ng):  # noqa: F811
    import torch
    from oracle import kkt
    g, types, x0 = case(nb + 1, nb, nl, ng)
    rng = np.random.default_rng(nb)
    B = 5
    X = np.repeat(x0[None, :], B, axis=0)
    ns = np.flatnonzero(types != 3)
    X[1:, ns] += rng.normal(0.0, 0.02, (B - 1, ns.size))
    net = ex.Net(g)
    jp, _ = ex.exago_net_jac_pattern(net.h)
    size = (r256(g.m * 8 * B) + r256(int(jp[-1]) * 8 * B) + 4 * r256(blocks_of(ex, net) * 32 * B) +
            r256(nb * 16 * B) + r256(16 * B))
    ws = torch.empty(size, dtype=torch.uint8, device="cuda")
    pf = ex.exago_pf_create(net.h, types)
    try:
        x = torch.as_tensor(X, device="cuda")
        xn, mis = torch.empty_like(x), torch.empty(B, dtype=torch.float64, device="cuda")
        ex.exago_pf_step(pf, ex.make_batch(x, workspace=ws), xn, mis)
        with pytest.raises(Exception, match="workspace"):
            ex.exago_pf_step(pf, ex.make_batch(x, workspace=ws[:size - 1]), torch.empty_like(x), None)
        xg, mg = xn.cpu().numpy(), mis.cpu().numpy()
    finally:
        ex.exago_pf_destroy(pf)
    onet = oracle_mod.OracleNet(g)
    for i in range(B):
        xr, mr = kkt.pf_newton_step(oracle_mod, onet, X[i], types)
        compare_step(g, types, X[i], xg[i], xr, mg[i], mr, f"{nb} buses [{i}]")
    net.close()
