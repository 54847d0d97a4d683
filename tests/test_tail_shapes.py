"""The dense tails of the grids that the GPU tests name for them (choose_tail, host code)."""
import os
import shutil
import subprocess

import pytest

from paper_2203_10587_gb300 import synth
from test_gpu_tail_shapes import TAILS, grid
from test_host_sanitizers import CSRC, ROOT, cuda_include


@pytest.fixture(scope="module")
def driver(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("no host compiler")
    exe = str(tmp_path_factory.mktemp("tail") / "tail_driver")
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-I", cuda_include(), "-o", exe,
                           os.path.join(ROOT, "tests", "sanitize", "tail_driver.cpp"),
                           os.path.join(CSRC, "blockfact_sym.cpp")])
    return exe


def tails(driver, g):
    """(first column, size, largest batch) of the KKT step's tail and of the power flow's."""
    lines = "\n".join(f"{a} {b}" for a, b in zip(g.f, g.t))
    out = subprocess.run([driver], input=f"{g.nb} {g.nl}\n{lines}\n", capture_output=True, text=True,
                         check=True).stdout
    return [tuple(map(int, line.split())) for line in out.splitlines()]


@pytest.mark.parametrize("nb,nl", sorted(TAILS))
def test_tail_of(driver, nb, nl):
    got = []
    for (k0, n, most), bs in zip(tails(driver, grid(nb, nl)), (4, 2)):
        assert k0 == 0 and most >= 130   # every bus, in batches as large as the tests'
        got.append((n, n - bs * nb))
    assert tuple(got) == TAILS[nb, nl]


# the batches from which the columns level by level were measured to be faster, to a factor of 2
@pytest.mark.parametrize("nb,nl,kkt,pf", [(14, 42, 800, 200), (30, 90, 1900, 600), (57, 171, 2300, 1100),
                                          (118, 159, 2100, 420), (200, 270, 3000, 750)])
def test_largest_batch(driver, nb, nl, kkt, pf):
    g = synth.make_grid(nb, nb, nl, max(2, nb // 5), max_degree=8 if nl < 2 * nb else 14, shunts=True)
    for (_, _, most), want in zip(tails(driver, g), (kkt, pf)):
        assert want / 2 <= most <= want * 2


def test_tails_of_the_smallest_and_the_large(driver):
    (k0, n, most), (k1, n1, _) = tails(driver, synth.make_grid(5, 5, 5, 2))
    assert (k0, n, most, k1, n1) == (5, 0, 0, 5, 0)   # none
    assert [t[2] for t in tails(driver, synth.grid_2000())] == [2 ** 31 - 1] * 2   # in any batch
