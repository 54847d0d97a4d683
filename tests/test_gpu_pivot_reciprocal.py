"""GPU: the pivots of the dense tail are inverted as exactly as a division does it."""
import numpy as np
import pytest

from test_gpu_kkt import ex, run_kkt  # noqa: F401
from test_gpu_tail_shapes import grid

pytestmark = pytest.mark.gpu


def test_pivot_reciprocals(ex):  # noqa: F811
    """The tail's pivots are inverted by a division: on a K that is diagonal the step is that
    reciprocal bit for bit, for significands of all kinds over all normal exponents, both signs.
    (One third-order step from the hardware's approximation was up to 1 ulp off, and off at all for
    one pivot in six.)"""
    g = grid(24, 180)   # all 24 buses are in the tail
    net = ex.Net(g)
    n, B = g.n, 600
    rng = np.random.default_rng(7)
    field = rng.integers(1, 2047, (B, 2 * g.nb)).astype(np.uint64)
    edges = np.array([1, 2, 63, 64, 65, 1022, 1023, 1024, 1963, 1964, 1965, 2044, 2045, 2046], np.uint64)
    field[::3] = edges[rng.integers(0, edges.size, field[::3].shape)]
    m = rng.integers(0, 1 << 52, field.shape, dtype=np.uint64)
    m[1::5] = 0
    m[2::5] = (1 << 52) - 1
    m[3::5] >>= np.uint64(40)
    s = rng.integers(0, 2, field.shape).astype(np.uint64)
    d = (s << np.uint64(63) | field << np.uint64(52) | m).view(np.float64)
    dx = np.ones((B, n))
    dx[:, :2 * g.nb] = d
    rhs = np.zeros((B, n + g.m))
    rhs[:, :2 * g.nb] = 1.0
    jp, _ = ex.exago_net_jac_pattern(net.h)
    hp, _ = ex.exago_net_hess_pattern(net.h)
    sol, _ = run_kkt(ex, net, np.zeros((B, jp[-1])), np.zeros((B, hp[-1])), dx, np.ones((B, g.m)), rhs)
    got, want = sol[:, :2 * g.nb], 1.0 / d
    assert np.array_equal(got, want), ((got != want).mean(), d[got != want][:5])
    net.close()
