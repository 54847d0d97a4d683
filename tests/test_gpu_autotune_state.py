"""GPU: the autotuner on small grids, whose untouched configuration runs one block per state: tuning
a batch size leaves its calls no slower than they were, with the same bits; a configuration set by
hand, the tuned choice among them, still runs what it says.

Tolerance of the times: the same kernel before and after; 1.2 for noise (median of 9 runs of 50
calls; without the block per state the calls took 1.6 times as long).
"""
import numpy as np
import pytest

from paper_2203_10587_gb300 import synth
from test_gpu_state_block import batch_of, ex, run  # noqa: F401

pytestmark = pytest.mark.gpu

KEYS = ("f", "grad", "gh", "jval", "hval")


def us_per_call(net, bt, out):
    import torch
    t = []
    for _ in range(10):
        e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
        e[0].record()
        for _ in range(50):
            net.eval_all(bt, out)
        e[1].record()
        torch.cuda.synchronize()
        t.append(e[0].elapsed_time(e[1]) * 20.0)
    return float(np.median(t[1:]))


@pytest.mark.parametrize("nb,nl,B", [(30, 41, 1), (200, 260, 100)])
def test_tuning_keeps_the_block_per_state(ex, nb, nl, B):  # noqa: F811
    import torch
    g = synth.make_grid(nb, nb, nl, nb // 5, shunts=True)
    b = synth.random_batch(nb, g, min(B, 5), masks=True, sigma=0.7)
    bt = batch_of(ex, b, np.arange(B) % b.B)
    net = ex.Net(g)
    want = run(ex, net, bt, B, KEYS)
    out = net.outputs(B)
    before = us_per_call(net, bt, out)
    for _ in range(2):   # a second tuning finds what the first left
        best = ex.exago_net_autotune(net.h, bt, *(out[k] for k in KEYS), reps=10)
        assert best["schedule"] in (1, 2, 3)
        after = us_per_call(net, bt, out)
        assert after <= 1.2 * before, (before, after)
    got = run(ex, net, bt, B, KEYS)
    ex.exago_net_set_config(net.h, **{k: best[k] for k in (
        "schedule", "block", "occupancy", "stage_records", "tile_group", "tiling", "chunk")})
    chosen = run(ex, net, bt, B, KEYS)
    for k in KEYS:
        assert torch.equal(got[k], want[k]) and torch.equal(chosen[k], want[k]), k
    net.close()
