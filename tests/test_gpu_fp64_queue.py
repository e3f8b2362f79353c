"""Points that wait for the FP64 pass: few of them are shared by a cluster of CTAs each, more
than there are clusters get a CTA each. Both, and the line between them, against the oracle."""
import numpy as np
import pytest

import oracle
import synth
from gpu_common import compare, run_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def vb():
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    import paper_1907_12933_gb300 as m
    from paper_1907_12933_gb300 import build
    build.build()
    return m


@pytest.mark.parametrize("dims,act", [([20, 33, 5], "sigmoid"), ([25, 20, 5], "relu"), ([40, 300, 70, 7], "sigmoid"),
                                      ([30, 1000, 9, 1024, 3], "identity")])
@pytest.mark.parametrize("points", [1, 151, 152, 153, 1217, 6859])
def test_points_by_cluster_or_by_cta(vb, dims, act, points):
    """Two equal outputs (and, where both exist, a dead neuron): every point is a margin tie."""
    net = synth.make_net(870, dims, act, 2.0, "normal")
    net["W"][0][5] = 0.0
    net["b"][0][5] = 0.0
    s, k = (3, 9) if points > 1000 else (1, 127)
    q = synth.make_query(870, 3, dims[0], s, k)
    D = oracle.eval_point(net, dict(q, pixels=q["pixels"][:0], k=0), 0)["D"]
    net["W"][-1][(D + 1) % dims[-1]] = net["W"][-1][D]
    net["b"][-1][(D + 1) % dims[-1]] = net["b"][-1][D]
    n = oracle.space_size(s, k)
    lo = min(7, n - points)
    o = oracle.verify(net, q, lo=lo, hi=lo + points)
    assert o["n_ties"] == points
    g = run_gpu(vb, net, q, "fp32", lo=lo, hi=lo + points)
    assert g["summary"]["n_recheck"][3] == points
    compare(g, o, net, q)
