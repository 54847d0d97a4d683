"""GPU: slack calls that ask for one or two of the three outputs give the bits of the call that asks
for all, for fewer slacks than a block has threads and for more.

Time: of 16,384 states of 14 buses, the balance rows alone against all three outputs.  The objective's
blocks are nine tenths of the latter; 0.13 lies between the rows' share without blocks and registers
for the absent outputs (0.10) and with them (0.155).
"""
import numpy as np
import pytest

from paper_2203_10587_gb300 import synth
from test_gpu_slack import ex  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nb,nz", [(12, 40), (300, 1700)])
def test_slack_output_subsets(ex, nb, nz):  # noqa: F811
    import torch
    g = synth.make_grid(nb, nb, nb + nb // 3, nb // 4 + 1)
    net = ex.Net(g)
    rng = np.random.default_rng(nb)
    s = ex.Slack(net, rng.integers(0, nb, nz), rng.integers(0, 2, nz), rng.choice([-1, 1], nz), rng.uniform(1, 9, nz))
    B = 19
    t = lambda *sh: torch.as_tensor(rng.normal(size=sh), device="cuda")
    bt = ex.make_batch(t(B, g.n), obj_weight=t(B))
    z, gh, f, v = t(B, nz), t(B, g.m), t(B), t(B, g.m)
    full = [gh.clone(), f.clone(), torch.empty_like(z)]
    ex.exago_eval_slack(s, bt, z, full[0], g.m, full[1], full[2])
    for want in range(1, 8):
        got = [gh.clone() if want & 1 else None, f.clone() if want & 2 else None,
               torch.empty_like(z) if want & 4 else None]
        ex.exago_eval_slack(s, bt, z, got[0], g.m, got[1], got[2])
        for a, b in zip(got, full):
            assert a is None or torch.equal(a, b), want
    rows, vals = s.pattern()
    out = torch.empty_like(z)
    ex.exago_eval_slack_jtv(s, bt, v, g.m, out)
    np.testing.assert_array_equal(out.cpu().numpy(), v.cpu().numpy()[:, rows] * vals)
    s.close()
    net.close()


def test_rows_alone_of_many_small_states(ex):  # noqa: F811
    import torch
    g = synth.make_grid(14, 14, 18, 3)
    net = ex.Net(g)
    nb, B = 14, 16384
    s = ex.Slack(net, np.tile(np.arange(nb), 4), np.repeat([0, 0, 1, 1], nb), np.repeat([1, -1, 1, -1], nb),
                 np.full(4 * nb, 500.0))
    t = lambda *sh: torch.rand(*sh, dtype=torch.float64, device="cuda")
    bt = ex.make_batch(t(B, g.n))
    z, gh, f, gz = t(B, 4 * nb), t(B, g.m), t(B), t(B, 4 * nb)
    us = []
    for out in ((gh, f, gz), (gh, None, None)):
        times = []
        for _ in range(12):
            e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
            e[0].record()
            for _ in range(20):
                ex.exago_eval_slack(s, bt, z, out[0], g.m, out[1], out[2])
            e[1].record()
            torch.cuda.synchronize()
            times.append(e[0].elapsed_time(e[1]) * 50.0)
        us.append(float(np.median(times[2:])))
    print("all, rows alone:", us)
    assert us[1] <= 0.13 * us[0], us
    s.close()
    net.close()
