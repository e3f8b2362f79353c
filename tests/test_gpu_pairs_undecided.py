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


@pytest.mark.parametrize("act,dims", [("relu", [25, 40, 10, 5]), ("identity", [30, 64, 7, 5])])
@pytest.mark.parametrize("n", [5, 640])
@pytest.mark.parametrize("off", [0.0, 5e-10, -5e-10, 9.99e-10, 1.001e-9, -1.001e-9, 3e-9, -3e-9])
def test_distances_around_the_tie_band(vb, act, dims, n, off):
    """The bound d lies at the distance of one pair's layer, or just off it: within the tie band,
    at its edges, outside. The other pairs are images that differ in one grey level, and
    identical ones."""
    net = synth.make_net(901, dims, act, 2.0, "normal")
    rng = np.random.default_rng(901)
    a = np.tile(rng.integers(30, 225, dims[0]).astype(np.uint8), (n, 1))
    # layer 1 keeps its signs, the layers behind it lie near theirs
    net["b"][0] += 20.0
    at = 0
    for l in range(1, len(dims) - 1):
        at += dims[l]
        u = oracle.forward(net, a[0].astype(float) / 255)
        net["b"][l] -= (u[at:at + dims[l + 1]] + 0.01 * rng.standard_normal(dims[l + 1])).astype(np.float32)
    b = a.copy()
    for i in range(0, n, 2):  # every other pair is identical
        pix = rng.choice(dims[0], 3, replace=False)
        b[i, pix] += rng.integers(1, 30, 3).astype(np.uint8)
    u1, u2 = oracle.forward(net, a[0].astype(float) / 255), oracle.forward(net, b[0].astype(float) / 255)
    dist = float(np.sqrt(((u1[:dims[1]] - u2[:dims[1]]) ** 2).sum()))
    vnet = vb.Net(net)
    seen = set()
    for d in (max(0.0, dist + off), abs(off)):
        got = vb.pair_coverage(vnet, a, b, g=1.05, d=d)
        exp = oracle.pairs_coverage(net, a, b, g=1.05, d=d)
        for k, v in exp.items():
            np.testing.assert_array_equal(got[k][:len(v)], v, err_msg=k)
            if v.any():
                seen.add(k)
    assert {"ds", "dv"} <= seen
    assert {"ds_tie", "dv_tie"} <= seen or n > 5 or abs(off) > 9e-10
    vnet.free()
