"""Covers over pairs that FP32 pairs cannot decide: every pair of a net with a dead neuron,
blocks of identical images at distance bound 0, and both among ordinary pairs, at counts
on both sides of the line between 2 and 8 images a CTA."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def vb():
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    import paper_1907_12933_gb300 as m
    from paper_1907_12933_gb300 import build
    build.build()
    return m


@pytest.mark.parametrize("act,dims", [("relu", [25, 10, 5]), ("identity", [30, 64, 7, 5]), ("relu", [40, 300, 70, 3])])
@pytest.mark.parametrize("n", [1, 6, 640])
@pytest.mark.parametrize("kind", ["dead", "dead output", "same", "mixed"])
def test_undecided_pairs(vb, act, dims, n, kind):
    net = synth.make_net(900, dims, act, 2.0, "normal")
    if kind == "dead":
        net["W"][0][4] = 0.0
        net["b"][0][4] = 0.0
    elif kind == "dead output":
        net["W"][-1][1] = 0.0
        net["b"][-1][1] = 1e-10
    rng = np.random.default_rng(900 + n)
    a = rng.integers(0, 256, (n, dims[0])).astype(np.uint8)
    b = a.copy()
    for i in range(n):  # blocks of 7 pairs: changed, or identical
        if kind in ("dead", "dead output") or (kind == "mixed" and (i // 7) % 2 == 0):
            pix = rng.choice(dims[0], 4, replace=False)
            b[i, pix] = np.clip(b[i, pix].astype(int) + rng.integers(-60, 61, 4), 0, 255)
    d = 0.0 if kind in ("same", "mixed") else 0.3
    vnet = vb.Net(net)
    got = vb.pair_coverage(vnet, a, b, g=1.5, d=d)
    exp = oracle.pairs_coverage(net, a, b, g=1.5, d=d)
    for k, v in exp.items():
        np.testing.assert_array_equal(got[k][:len(v)], v, err_msg=k)
    vnet.free()
