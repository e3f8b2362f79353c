"""The counts of a warp's threads on their way into a query's 64-bit counters: sums past
32 bits, and sums that are multiples of 2^32, which still hold a first witness."""
import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    from paper_1907_12933_gb300 import build
    exe = str(tmp_path_factory.mktemp("counts") / "warp_counts")
    subprocess.run([build._nvcc(), *build.ARCH, "-O2", "-std=c++17", os.path.join(HERE, "warp_counts.cu"), "-o", exe],
                   check=True)
    return exe


@pytest.mark.parametrize("adv", [0, 1, 0xffff, 0x10000, 1 << 27, (1 << 27) + 1, 1 << 31, 0xffffffff])
@pytest.mark.parametrize("pts", [0, 5, 1 << 27, 0xffffffff])
def test_sums(program, adv, pts):
    out = subprocess.run([program, str(adv), str(pts)], check=True, capture_output=True, text=True, timeout=60).stdout
    n_adv, n_points, first, left = map(int, out.split())
    assert (n_adv, n_points, left) == (2 * 96 * adv, 2 * 96 * pts, 0)
    assert first == (1000 - 95 if adv else 2**64 - 1)
