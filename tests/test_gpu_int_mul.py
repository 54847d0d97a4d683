"""GPU: products on the integer pipe (csrc/int_mul.cuh) where they could differ from the FP64
pipe's: random significands, ties and carries (through the slacks' gradient w cost, one product
each, compared bit for bit with numpy's), and operands outside their window (zeros, subnormals, tiny
and huge values, infinities, NaN), also in the adjoint products of states with such voltages."""
import numpy as np
import pytest

from paper_2203_10587_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ex():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2203_10587_gb300 import build, exago
    build.build()
    exago.lib()
    return exago


def values(seed, n):
    """Doubles over the window, with few and with all significand bits, and its edges."""
    rng = np.random.default_rng(seed)
    m = rng.integers(0, 1 << 52, n, dtype=np.uint64)
    m[::5] &= ~np.uint64((1 << 26) - 1)           # products that are exact, or ties
    m[1::7] |= np.uint64((1 << 52) - (1 << 20))   # roundings that carry into the exponent
    e = rng.integers(768, 1280, n).astype(np.uint64)
    e[2::11] = 768
    e[3::11] = 1279
    s = rng.integers(0, 2, n).astype(np.uint64)
    return (s << np.uint64(63) | e << np.uint64(52) | m).view(np.float64)


def test_gradient_products_bitwise(ex):
    import torch
    g = synth.make_grid(3, 40, 50, 8)
    net = ex.Net(g)
    nz, B = 4099, 6
    cost, w = values(1, nz), values(2, B)
    w[1], w[2] = 0.0, 5e-324
    cost[7], cost[8], cost[9] = 0.0, 1e-300, 1e300
    sl = ex.Slack(net, np.arange(nz) % g.nb, np.arange(nz) % 2, np.ones(nz, int), cost)
    x = torch.zeros(B, net.n, dtype=torch.float64, device="cuda")
    z = torch.zeros(B, nz, dtype=torch.float64, device="cuda")
    out = torch.empty_like(z)
    for k, extra in ((None, None), (3, np.inf), (3, np.nan)):
        ww = w.copy()
        if k is not None:
            ww[k] = extra
        bt = ex.make_batch(x, obj_weight=torch.as_tensor(ww, device="cuda"))
        ex.exago_eval_slack(sl, bt, z, grad_z=out)
        with np.errstate(all="ignore"):
            want = ww[:, None] * cost[None, :]
        np.testing.assert_array_equal(out.cpu().numpy(), want)


@pytest.mark.parametrize("vm", [0.0, 1e-310, 1e-200, 1e140, np.inf, np.nan])
def test_adjoint_outside_the_window(ex, vm):
    """J u, J'v and H u of a state one of whose voltages is extreme: the entries that the products
    with the evaluation's own J and H give, to rounding, wherever those are finite."""
    import torch
    g = synth.make_grid(9, 60, 90, 12, shunts=True)
    b = synth.random_batch(9, g, 2, sigma=0.6)
    b.x[1, g.nb + int(g.f[4])] = vm
    net = ex.Net(g)
    t = lambda a: torch.as_tensor(np.ascontiguousarray(a), device="cuda")
    bt = ex.make_batch(t(b.x), t(b.lam), obj_factor=b.sigma)
    out = net.eval_all(bt, net.outputs(2))
    rng = np.random.default_rng(9)
    u, v = rng.normal(size=(2, net.n)), rng.normal(size=(2, net.m))
    ju, jtv, hu = (torch.empty(2, k, dtype=torch.float64, device="cuda") for k in (net.m, net.n, net.n))
    ex.exago_eval_jvp(net.h, bt, t(u), ju)
    ex.exago_eval_jtv(net.h, bt, t(v), jtv)
    ex.exago_eval_hvp(net.h, bt, t(u), hu)
    jp, jc = ex.exago_net_jac_pattern(net.h)
    hp, hc = ex.exago_net_hess_pattern(net.h)
    for s in range(2):
        J, H = np.zeros((net.m, net.n)), np.zeros((net.n, net.n))
        J[np.repeat(np.arange(net.m), np.diff(jp)), jc] = out["jval"][s].cpu().numpy()
        H[np.repeat(np.arange(net.n), np.diff(hp)), hc] = out["hval"][s].cpu().numpy()
        H = H + np.tril(H, -1).T
        with np.errstate(all="ignore"):
            for got, M, w in ((ju, J, u[s]), (jtv, J.T, v[s]), (hu, H, u[s])):
                got = got[s].cpu().numpy()
                ref, mag = M @ w, np.abs(M) @ np.abs(w)
                fine = np.isfinite(mag)
                # a sum of at most 64 rounded terms of which each is a few roundings
                assert np.all(np.abs(got[fine] - ref[fine]) <= 1e-13 * mag[fine] + 1e-280), s
