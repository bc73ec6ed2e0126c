"""A node whose lag or bin its table does not hold reports itself (the host's bounds
make the tables hold every node; this is the check behind them)."""
import os
import subprocess

import pytest

from gpu_common import torch_cuda

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))
LAG_RANGE = 2


def test_nodes_outside_of_their_table_are_reported(tmp_path):
    torch_cuda()
    from paper_2508_06672_gb300 import build
    exe = str(tmp_path / "map_range")
    subprocess.run([build.nvcc(), *build.ARCH, "-O2", "-std=c++17", "-I" + os.path.join(build.ROOT, "include"), "-I" + build.CSRC,
                    os.path.join(HERE, "device_map_range.cu"), "-o", exe], check=True, capture_output=True)
    lines = subprocess.run([exe], check=True, capture_output=True, text=True, timeout=60).stdout.split("\n")
    got = {tuple(map(int, x.split()[:2])): [int(e) for e in x.split()[2:]] for x in lines if x}
    assert len(got) == 6
    # lag 0 inside, at the first and the last lag, one before and one past them; the
    # bin's stencil at its first and last place, and beyond; a lag far outside
    integer = [0, 0, 0, 1, 1, 0, 0, 1, 1, 1]
    lagrange = [0, 1, 1, 1, 1, 0, 0, 1, 1, 1]  # the stencil reaches one lag back and two on
    for (poly, delay), err in got.items():
        assert err == [LAG_RANGE * e for e in (lagrange if delay else integer)], (poly, delay, err)
