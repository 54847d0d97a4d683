"""GPU: the slacks' gradient written over the slack values themselves (and over a part of them): the
balance terms and the objective still see the values as they were, bit for bit.
"""
import numpy as np
import pytest

from paper_2203_10587_gb300 import synth
from parity_util import to_device
from test_gpu_slack import ex, slack_set  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shift", [0, 1, -1])
def test_gradient_over_values(ex, shift):  # noqa: F811
    import torch
    g = synth.make_grid(131, 300, 389, 77, shunts=True)
    b = synth.random_batch(131, g, 13, masks=True, obj_weight=True, sigma=0.6)
    bus, row, sign, cost = slack_set(g, 132)
    nz = bus.shape[0]
    net = ex.Net(g)
    sl = ex.Slack(net, bus, row, sign, cost)
    d = to_device(b)
    bt = ex.make_batch(d["x"], d["lam"], d["mask"], d["pd_scale"], d["obj_weight"], b.sigma)
    z = np.random.default_rng(133).uniform(0.0, 0.2, (b.B, nz))
    res = []
    for inplace in (False, True):
        buf = torch.zeros((b.B + 2) * nz, dtype=torch.float64, device="cuda")
        zd = buf[nz:nz + b.B * nz].view(b.B, nz)
        zd.copy_(torch.as_tensor(z))
        k = nz + shift * 5
        grad = buf[k:k + b.B * nz].view(b.B, nz) if inplace else torch.zeros_like(zd)
        out = net.outputs(b.B, jac=False, hess=False)
        net.eval_all(bt, out)
        ex.exago_eval_slack(sl, bt, zd, out["gh"], g.m, out["f"], grad)
        torch.cuda.synchronize()
        res.append([t.cpu().numpy().copy() for t in (out["gh"], out["f"], grad)])
    for a, c in zip(*res):
        np.testing.assert_array_equal(a, c)
    sl.close()
    net.close()
