"""GPU: ramp-row transposes of batches of many families (periods or scenarios of a dozen and of a
few hundred states each around a base state) against the definition, at the children counts where the
blocks change.

Tolerances: a transpose sums at most a few hundred terms of size one in another order than numpy
(1e-11, as tests/test_gpu_coupling.py).  Time: families of 12 move the same bytes as families of 9, in
blocks of another shape; they may take 1.5 times as long.
"""
import numpy as np
import pytest

from paper_2203_10587_gb300 import synth
from test_gpu_slack import ex  # noqa: F401

pytestmark = pytest.mark.gpu


def families(B, size):
    p = np.arange(B) // size * size
    p[p == np.arange(B)] = -1
    return p.astype(np.int32)


# the last: enough generators for blocks of 8 to fill the chip, whatever the children
@pytest.mark.parametrize("size,ng", [(9, 23), (10, 23), (12, 23), (33, 23), (65, 23), (257, 23), (258, 23),
                                     (600, 23), (300, 9801)])
def test_families(ex, size, ng):  # noqa: F811
    import torch
    g = synth.make_grid(3, max(60, ng), max(90, ng + 40), ng)
    net = ex.Net(g)
    B = 2 * size + 5   # two whole families, a rest, and one state with no family at all
    parent = families(B, size)
    parent[-1] = -1
    nu = np.random.default_rng(size).normal(size=(B, g.ng))
    want = np.where(parent[:, None] >= 0, nu, 0.0)
    for b in range(B):
        if parent[b] >= 0:
            want[parent[b]] -= nu[b]
    c = ex.Coupling(net, parent)
    for acc in (False, True):
        out = torch.ones(B, g.ng, dtype=torch.float64, device="cuda")
        ex.exago_eval_coupling_jtv(c.h, torch.as_tensor(nu, device="cuda"), out, g.ng, accumulate=acc)
        np.testing.assert_allclose(out.cpu().numpy(), want + acc, rtol=0, atol=1e-11)
    c.close()
    net.close()


def test_families_of_a_dozen_take_no_longer(ex):  # noqa: F811
    import torch
    g = synth.make_grid(4, 900, 1215, 180)
    net = ex.Net(g)
    B = 4104
    nu = torch.randn(B, g.ng, dtype=torch.float64, device="cuda")
    out = torch.zeros_like(nu)
    us = []
    for size in (9, 12):
        c = ex.Coupling(net, families(B, size))
        t = []
        for _ in range(12):
            e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
            e[0].record()
            for _ in range(10):
                ex.exago_eval_coupling_jtv(c.h, nu, out, g.ng)
            e[1].record()
            torch.cuda.synchronize()
            t.append(e[0].elapsed_time(e[1]) * 100.0)
        us.append(float(np.median(t[2:])))
        c.close()
    print("families of 9 and 12:", us)
    assert us[1] <= 1.5 * us[0], us
    net.close()
