"""The error bound of a folded row's sum: sums whose low parts all grow the same way, which
pass it when the pair is not settled on the way, and sums that cancel."""
import os
import struct
import subprocess
from fractions import Fraction

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    from paper_1907_12933_gb300 import build
    exe = str(tmp_path_factory.mktemp("pairsum") / "pair_sum")
    subprocess.run([build._nvcc(), *build.ARCH, "-O2", "-std=c++17", os.path.join(HERE, "pair_sum.cu"), "-o", exe],
                   check=True)
    return exe


def terms(kind, n, rng):
    w = np.ones(n, np.float32)
    h = np.zeros((n, 2), np.float32)
    if kind == "cancel":
        w[:] = rng.standard_normal(n)
        v = rng.standard_normal(n)
        v[n // 2:n // 2 * 2] = -v[:n // 2]
        w[n // 2:n // 2 * 2] = w[:n // 2]
        h[:, 0] = v
        h[:, 1] = (v - h[:, 0].astype(np.float64)) * 0.9
    else:  # 1, then terms just too small to move it: the low part takes them all
        h[:, 0] = np.float32(2.0 ** -24 * kind)
        h[0, 0] = 1.0
    return w, h


@pytest.mark.parametrize("n", [1, 7, 8, 9, 128, 500, 1024])
@pytest.mark.parametrize("kind", [0.99, 0.9, 0.7, 0.5001, 0.33, "cancel"])
def test_error_of_a_row_sum(program, tmp_path, n, kind):
    w, h = terms(kind, n, np.random.default_rng(860 + n))
    path = tmp_path / "terms"
    path.write_bytes(struct.pack("<i", n) + np.column_stack([w, h]).astype("<f4").tobytes())
    out = subprocess.run([program, str(path)], check=True, capture_output=True, text=True, timeout=60).stdout
    got = sum(Fraction(float.fromhex(x)) for x in out.split())
    prods = [Fraction(float(a)) * (Fraction(float(b)) + Fraction(float(c))) for a, (b, c) in zip(w, h)]
    bound = (Fraction(13, 2) * n + 20) * Fraction(1, 2 ** 48) * sum(map(abs, prods))
    assert abs(got - sum(prods)) <= bound
