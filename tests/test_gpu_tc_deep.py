"""Single queries whose tensor screen leaves points on nets of three and more layers behind
the first, with hidden layers of 192 and 256 neurons that mostly stay active: the split pass
holds two operand slots a chunk, and where its ring is too short for a layer's drain the FP32
pass takes its points. Against the FP64 pass, and on both sides of that line."""
import numpy as np
import pytest

import synth
from gpu_common import run_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def vb():
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    import paper_1907_12933_gb300 as m
    from paper_1907_12933_gb300 import build
    build.build()
    return m


@pytest.mark.parametrize("dims,stuck", [
    ([20, 64, 256, 128, 6], True),
    ([20, 64, 64, 192, 128, 3], True),
    ([50, 512, 256, 512, 9], True),
    ([30, 256, 256, 256, 19], True),
    ([20, 256, 128, 256, 6], False),   # two chunks: four slots
    ([20, 64, 256, 64, 6], False),     # the layer behind fits beside it
    ([20, 512, 512, 6], False),
])
@pytest.mark.parametrize("prec", ["bf16", "fp16"])
def test_deep_nets_through_the_split_pass(vb, dims, stuck, prec):
    net = synth.make_net(920, dims, "relu", 2.0, "normal")
    for l in range(len(dims) - 2):
        net["b"][l] += np.float32(0.5)  # most neurons active at every point
    q = synth.make_query(920, 1, dims[0], 2, 60)
    vnet = vb.Net(net)
    vb.set_folding(vnet, False)
    a = run_gpu(vb, net, q, prec, vbnet=vnet)
    b = run_gpu(vb, net, q, "fp64", vbnet=vnet)
    for key in ("flip", "flip_tie", "ss", "ss_tie", "bitmap", "ties"):
        np.testing.assert_array_equal(a[key], b[key], err_msg=key)
    for key in ("n_adversarial", "first_witness", "n_ties", "D", "n_points"):
        assert a["summary"][key] == b["summary"][key]
    n = a["summary"]["n_recheck"]
    assert n[0] > 0 and (n[1] == n[0]) == stuck
    vnet.free()
