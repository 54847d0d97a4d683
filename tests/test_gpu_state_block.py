"""GPU: the block-per-state schedule, which untouched configurations of small grids run: bitwise
equal to the persistent schedule (itself compared with the oracle elsewhere) at the sizes where it
can go wrong -- fewer branches than a warp, a block's threads exactly and one more, the largest grid
whose records fit, rows that do not fit beside them, one state and several waves -- with every
output subset, masks, load scales, weights, generator outages and phase shifters, a gathered
(served) batch, and inside a caller's CUDA graph."""
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


def batch_of(ex, b, rep):
    import torch
    t = lambda a, dt=torch.float64: None if a is None else torch.as_tensor(
        np.ascontiguousarray(a[rep]), dtype=dt, device="cuda")
    return ex.make_batch(t(b.x), t(b.lam), t(b.mask, torch.uint8), t(b.pd_scale), t(b.obj_weight),
                         b.sigma, gen_mask=t(b.gen_mask, torch.uint8))


def run(ex, net, bt, B, keys):
    out = {k: v for k, v in net.outputs(B).items() if k in keys}
    for v in out.values():
        v.fill_(float("nan"))
    net.eval_all(bt, out)
    return out


# branches: below a warp, 64 threads exactly and one more, 256 exactly and one more, several
# passes, and the limit of 1,280 (more fall back to the persistent schedule)
@pytest.mark.parametrize("nb,nl,B,shift", [(3, 2, 1, 0.0), (30, 41, 700, 0.0), (30, 41, 5, 0.1), (48, 64, 5, 0.2),
                                           (48, 65, 5, 0.0), (190, 256, 153, 0.0), (190, 257, 90, 0.1),
                                           (300, 389, 150, 0.1), (400, 512, 140, 0.0), (400, 513, 140, 0.0),
                                           (300, 900, 150, 0.0), (950, 1280, 150, 0.0),
                                           (950, 1281, 150, 0.0)])
def test_bitwise_equal_to_persistent(ex, nb, nl, B, shift):
    import torch
    g = synth.make_grid(nb, nb, nl, max(1, nb // 5), max_degree=12, shunts=True, shifter_frac=shift)
    b = synth.random_batch(nl, g, min(B, 7), masks=True, pd_scale=True, obj_weight=True, sigma=0.7,
                           gen_masks=nl % 2 == 1)
    bt = batch_of(ex, b, np.arange(B) % b.B)
    net, ref = ex.Net(g), ex.Net(g)
    ex.exago_net_set_config(ref.h, schedule=2)
    for keys in (("f", "grad", "gh", "jval", "hval"), ("f", "gh"), ("jval",), ("hval", "grad"), ("f",),
                 ("gh", "jval"), ("gh", "hval"), ("jval", "hval")):
        got, want = run(ex, net, bt, B, keys), run(ex, ref, bt, B, keys)
        for k in keys:
            assert torch.equal(got[k], want[k]), (nb, nl, k)


def test_served_and_captured(ex):
    import torch
    g = synth.make_grid(61, 118, 153, 30)
    b = synth.random_batch(61, g, 6, masks=True, gen_masks=True)
    net = ex.Net(g)
    bt = batch_of(ex, b, np.arange(6))
    want = run(ex, net, bt, 6, ("f", "grad", "gh", "jval", "hval"))
    srv = ex.exago_serve_create(64 << 20, 4, 2)
    try:
        nid = ex.exago_serve_register(srv, net.h)
        parts = [batch_of(ex, b, np.array([i])) for i in range(6)]
        outs = [net.outputs(1) for _ in range(6)]
        tk = [ex.exago_serve_submit(srv, nid, p, **o) for p, o in zip(parts, outs)]
        for t in tk:
            ex.exago_serve_wait(srv, t, 20000.0)
        for i, o in enumerate(outs):
            for k in o:
                assert torch.equal(o[k][0], want[k][i]), k
    finally:
        ex.exago_serve_destroy(srv)
    out = net.outputs(6)
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        bts = batch_of(ex, b, np.arange(6))
    s.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=s):
        bts.stream = torch.cuda.current_stream().cuda_stream
        net.eval_all(bts, out)
    for v in out.values():
        v.fill_(float("nan"))
    graph.replay()
    torch.cuda.synchronize()
    for k in out:
        assert torch.equal(out[k], want[k]), k
