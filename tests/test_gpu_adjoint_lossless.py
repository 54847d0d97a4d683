"""GPU: the adjoint products on grids with lossless branches (r = 0) at a flat start, where a
branch's conductance terms are exactly zero: the products with the evaluation's own J and H, and no
more time than for the same states with ordinary angles.

Tolerances.  Values: sums of at most 64 rounded terms, each a few roundings (1e-13 of the terms'
magnitudes).  Time: the work is the same; 1.25 leaves room for noise (median of 21), and items that are
computed twice took twice as long.
"""
import numpy as np
import pytest

from paper_2203_10587_gb300 import synth
from test_gpu_int_mul import ex  # noqa: F401

pytestmark = pytest.mark.gpu


def lossless(seed, nb, nl, ng):
    """A third of the branches without resistance, one of them without a ratio or line charging
    beside it; one branch without reactance."""
    g = synth.make_grid(seed, nb, nl, ng, shunts=True, transformer_frac=0.3)
    g.r[::3] = 0.0
    g.b[:6] = 0.0
    g.tap[:6] = 0.0
    g.r[1], g.x[1] = 0.01, 0.0
    return g


def products(ex, net, bt, u, v):
    import torch
    out = [torch.empty(u.shape[0], k, dtype=torch.float64, device="cuda") for k in (net.m, net.n, net.n)]

    def call():
        ex.exago_eval_jvp(net.h, bt, u, out[0])
        ex.exago_eval_jtv(net.h, bt, v, out[1])
        ex.exago_eval_hvp(net.h, bt, u, out[2])
    return out, call


@pytest.mark.parametrize("angles", ["flat", "minus_zero", "some"])
def test_products_of_lossless_branches(ex, angles):  # noqa: F811
    import torch
    g = lossless(5, 70, 110, 14)
    b = synth.random_batch(5, g, 3, masks=True, sigma=0.7)
    b.x[:, :g.nb] = {"flat": 0.0, "minus_zero": -0.0, "some": b.x[:, :g.nb] * (np.arange(g.nb) % 5 == 0)}[angles]
    net = ex.Net(g)
    t = lambda a, dt=torch.float64: torch.as_tensor(np.ascontiguousarray(a), dtype=dt, device="cuda")
    bt = ex.make_batch(t(b.x), t(b.lam), t(b.mask, torch.uint8), obj_factor=b.sigma)
    ev = net.eval_all(bt, net.outputs(3))
    rng = np.random.default_rng(5)
    u, v = rng.normal(size=(3, net.n)), rng.normal(size=(3, net.m))
    out, call = products(ex, net, bt, t(u), t(v))
    call()
    jp, jc = ex.exago_net_jac_pattern(net.h)
    hp, hc = ex.exago_net_hess_pattern(net.h)
    for s in range(3):
        J, H = np.zeros((net.m, net.n)), np.zeros((net.n, net.n))
        J[np.repeat(np.arange(net.m), np.diff(jp)), jc] = ev["jval"][s].cpu().numpy()
        H[np.repeat(np.arange(net.n), np.diff(hp)), hc] = ev["hval"][s].cpu().numpy()
        H = H + np.tril(H, -1).T
        for got, M, w in zip(out, (J, J.T, H), (u[s], v[s], u[s])):
            err = np.abs(got[s].cpu().numpy() - M @ w)
            assert np.all(err <= 1e-13 * (np.abs(M) @ np.abs(w)) + 1e-280), s
    net.close()


def test_no_slower_at_a_flat_start(ex):  # noqa: F811
    import torch
    g = lossless(6, 10000, 13000, 2500)
    b = synth.random_batch(6, g, 64)
    net = ex.Net(g)
    rng = np.random.default_rng(6)
    t = lambda a: torch.as_tensor(np.ascontiguousarray(a), device="cuda")
    u, v = t(rng.normal(size=(64, net.n))), t(rng.normal(size=(64, net.m)))
    us = []
    for flat in (False, True):
        x = b.x.copy()
        if flat:
            x[:, :g.nb] = 0.0
        bt = ex.make_batch(t(x), t(b.lam))
        _, call = products(ex, net, bt, u, v)
        times = []
        for i in range(24):
            e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
            e[0].record()
            call()
            e[1].record()
            torch.cuda.synchronize()
            times.append(e[0].elapsed_time(e[1]) * 1e3)
        us.append(float(np.median(times[3:])))
    print(f"J u, J'v, H u: {us[0]:.1f} us with angles, {us[1]:.1f} us flat")
    assert us[1] <= 1.25 * us[0], us
    net.close()
