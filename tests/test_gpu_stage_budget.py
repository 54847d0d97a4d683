"""GPU: how much shared memory a bus tile may stage its rows in does not show in the results: grids
whose tiles all fit the smaller limit, that need the larger one, and that outgrow both in some or
most tiles, per tile size and record staging, against the configuration without the limits, bit for
bit; and the rectangular formulation against its other schedule.
"""
import numpy as np
import pytest

from paper_2203_10587_gb300 import synth
from test_gpu_state_block import batch_of, ex, run  # noqa: F401

pytestmark = pytest.mark.gpu

KEYS = ("f", "grad", "gh", "jval", "hval")


# mean degrees 2.7, 5, 6 and 10: 64-bus tiles of 1,600 to 4,300 doubles against 2,232 and 2,744
@pytest.mark.parametrize("nl,deg", [(540, 8), (1000, 14), (1200, 16), (2000, 21)])
def test_results_do_not_depend_on_the_limit(ex, nl, deg):  # noqa: F811
    import torch
    g = synth.make_grid(nl, 400, nl, 90, max_degree=deg, shunts=True)
    b = synth.random_batch(nl, g, 5, masks=True, gen_masks=True, sigma=0.6)
    bt = batch_of(ex, b, np.arange(5))
    net = ex.Net(g)
    ex.exago_net_set_config(net.h, schedule=2, occupancy=8)
    want = run(ex, net, bt, 5, KEYS)
    for cfg in (dict(schedule=1), dict(schedule=1, stage_records=1), dict(schedule=3), *(
            dict(block=t, stage_records=r) for t in (32, 64, 128, 256) for r in (0, 1)),
            dict(block=64, stage_records=3), dict(block=128, stage_records=3),
            dict(block=64, occupancy=24)):
        ex.exago_net_set_config(net.h, **{"schedule": 2, **cfg})
        got = run(ex, net, bt, 5, KEYS)
        for k in KEYS:
            assert torch.equal(got[k], want[k]), (cfg, k)
    net.close()


@pytest.mark.parametrize("nl,deg", [(540, 8), (1200, 16), (2000, 21)])
def test_rectangular(ex, nl, deg):  # noqa: F811
    from test_gpu_cartesian import run_cart, to_cartesian
    g = synth.make_grid(nl, 400, nl, 90, max_degree=deg, shunts=True)
    b = synth.random_batch(nl, g, 5, masks=True, sigma=0.6)
    x, lam = to_cartesian(g, b, 3)
    net = ex.Net(g)
    res = []
    for cfg in (dict(), dict(occupancy=8), dict(schedule=3)):
        ex.exago_net_set_config(net.h, **cfg)
        res.append(run_cart(ex, net, b, x, lam))
    for r in res[1:]:
        for k in KEYS:
            np.testing.assert_array_equal(r[k], res[0][k])
    net.close()
