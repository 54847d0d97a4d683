"""The dense tails of the grids that the GPU tests name for them (choose_tail, host code)."""
import os
import shutil
import subprocess

import pytest

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


@pytest.mark.parametrize("nb,nl", sorted(TAILS))
def test_tail_of(driver, nb, nl):
    g = grid(nb, nl)
    lines = "\n".join(f"{a} {b}" for a, b in zip(g.f, g.t))
    out = subprocess.run([driver], input=f"{nb} {nl}\n{lines}\n", capture_output=True, text=True, check=True).stdout
    got = []
    for line, bs in zip(out.splitlines(), (4, 2)):
        k0, n = map(int, line.split())
        assert k0 == 0   # every bus
        got.append((n, n - bs * nb))
    assert tuple(got) == TAILS[nb, nl]
