"""GPU: KKT and power-flow steps of small grids in large batches, where the dense last columns would
cost more than they save: no slower than with a workspace that leaves no room for them (that is, level
by level), within the steps' bounds, a state's result the same bits in any batch beyond the line, and
in any below it.

Tolerance of the times: the same launches; 1.15 for noise (median of 9).  With the dense columns in every
batch these took 2.2 to 4.9 times as long.
"""
import numpy as np
import pytest

from paper_2203_10587_gb300 import synth
from test_gpu_kkt import check_state, ex, kkt_inputs, run_kkt  # noqa: F401
from test_gpu_pflow import case, compare_step, gpu_steps
from test_gpu_small_workspace import blocks_of, r256

pytestmark = pytest.mark.gpu


def median_us(call):
    import torch
    t = []
    for _ in range(11):
        e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
        e[0].record()
        call()
        e[1].record()
        torch.cuda.synchronize()
        t.append(e[0].elapsed_time(e[1]) * 1e3)
    return float(np.median(t[2:]))


@pytest.mark.parametrize("nb,nl,B", [(14, 18, 4096), (57, 76, 8192)])
def test_kkt(ex, oracle_mod, nb, nl, B):  # noqa: F811
    import torch
    g = synth.make_grid(nb, nb, nl, nb // 5, shunts=True)
    b = synth.random_batch(nb, g, 2, masks=True, sigma=0.9)
    refs, jval, hval, dx, dc, _ = kkt_inputs(oracle_mod, g, b, nb)
    rep = np.arange(B) % 2
    rhs = np.random.default_rng(nb).normal(size=(B, g.n + g.m))
    net = ex.Net(g)
    sol, inertia = run_kkt(ex, net, jval[rep], hval[rep], dx[rep], dc[rep], rhs)
    assert np.all(inertia == [g.m, 0])
    for i in (0, B - 1):
        check_state(g, refs[rep[i]], dx[rep[i]], dc[rep[i]], rhs[i], sol[i], what=f"{nb} buses [{i}]")
    part, _ = run_kkt(ex, net, *(a[rep[:B // 2]] for a in (jval, hval, dx, dc)), rhs[:B // 2])
    np.testing.assert_array_equal(part, sol[:B // 2])
    few, _ = run_kkt(ex, net, *(a[rep[:64]] for a in (jval, hval, dx, dc)), rhs[:64])
    one, _ = run_kkt(ex, net, *(a[rep[:1]] for a in (jval, hval, dx, dc)), rhs[:1])
    np.testing.assert_array_equal(few[0], one[0])
    k = ex.exago_kkt_create(net.h)
    t = [torch.as_tensor(a, device="cuda") for a in (jval[rep], hval[rep], dx[rep], dc[rep], rhs)]
    out = torch.empty_like(t[4])
    least = 2 * r256(blocks_of(ex, net) * 128 * B) + r256(nb * 32 * B) + r256(8 * B)
    us = []
    for size in (ex.exago_kkt_workspace_size(k, B), least):
        ws = torch.empty(size, dtype=torch.uint8, device="cuda")
        us.append(median_us(lambda: ex.exago_kkt_solve(k, *t, out, None, ws)))
    ex.exago_kkt_destroy(k)
    net.close()
    assert us[0] <= 1.15 * us[1], us


@pytest.mark.parametrize("nb,nl,B", [(57, 76, 4096), (118, 159, 2048)])
def test_pflow(ex, oracle_mod, nb, nl, B):  # noqa: F811
    import torch
    from oracle import kkt
    g, types, x0 = case(nb, nb, nl, nb // 5)
    X = np.repeat(x0[None, :], B, axis=0)
    ns = np.flatnonzero(types != 3)
    X[1:, ns] += np.random.default_rng(nb).normal(0.0, 0.02, (B - 1, ns.size))
    net = ex.Net(g)
    pf = ex.exago_pf_create(net.h, types)
    xg, mg = gpu_steps(ex, net, pf, X)
    onet = oracle_mod.OracleNet(g)
    for i in (0, B - 1):
        xr, mr = kkt.pf_newton_step(oracle_mod, onet, X[i], types)
        compare_step(g, types, X[i], xg[i], xr, mg[i], mr, f"{nb} buses [{i}]")
    np.testing.assert_array_equal(gpu_steps(ex, net, pf, X[:B // 2])[0], xg[:B // 2])
    np.testing.assert_array_equal(gpu_steps(ex, net, pf, X[:64])[0][0], gpu_steps(ex, net, pf, X[:1])[0][0])
    jp, _ = ex.exago_net_jac_pattern(net.h)
    least = (r256(g.m * 8 * B) + r256(int(jp[-1]) * 8 * B) + 4 * r256(blocks_of(ex, net) * 32 * B) +
             r256(nb * 16 * B) + r256(16 * B))
    x = torch.as_tensor(X, device="cuda")
    out = torch.empty_like(x)
    us = []
    for size in (ex.exago_pf_workspace_size(pf, B), least):
        bt = ex.make_batch(x, workspace=torch.empty(size, dtype=torch.uint8, device="cuda"))
        us.append(median_us(lambda: ex.exago_pf_step(pf, bt, out, None)))
    ex.exago_pf_destroy(pf)
    net.close()
    assert us[0] <= 1.15 * us[1], us
