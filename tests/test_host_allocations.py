"""The library's host code when memory runs out, on a fake device (no GPU): every
allocation of a program that goes through several grids, capture lengths, windows,
regions and graphs is made to fail once, alone and with the two after it. Whatever
call reports it, no later launch may get a buffer that is gone, too small or not
filled, nothing is allocated inside a capture, every call works again once there
is memory, and every buffer is given back."""
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


@pytest.fixture(scope="module")
def fake_device(tmp_path_factory):
    from paper_2508_06672_gb300 import build
    d = tmp_path_factory.mktemp("fake_device")
    obj, exe = str(d / "host.o"), str(d / "host")
    subprocess.run([build.nvcc(), *build.ARCH, "-O2", "-std=c++17", "-I" + os.path.join(ROOT, "include"),
                    "-I" + build.CSRC, "-c", os.path.join(HERE, "host_fake_device.cu"), "-o", obj], check=True,
                   capture_output=True)
    subprocess.run(["g++", obj, "-o", exe, "-lpthread"], check=True)
    return exe


@pytest.mark.parametrize("what", ["maps", "lagrange", "direct", "chunks", "fp32"])
def test_no_launch_on_buffers_that_a_failed_allocation_took(fake_device, what):
    runs = [subprocess.Popen([fake_device, what, count], stdout=subprocess.PIPE, text=True) for count in ("1", "3")]
    for r in runs:
        out = r.communicate(timeout=300)[0]
        assert r.returncode == 0, out[-3000:]
        assert int(out.split(":")[1].split()[0]) > 100, out


def test_direct_sort_keeps_to_the_scratch_target(fake_device):
    r = subprocess.run([fake_device, "scratch"], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout


@pytest.mark.parametrize("what", ["kept-direct", "kept-cdft"])
def test_buffers_of_captured_steps_are_given_back(fake_device, what):
    r = subprocess.run([fake_device, what], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout
