"""Batches whose queries the general passes check, because their net, their precision or a
switch keeps them from folding, against the FP64 oracle."""
import ctypes as C

import numpy as np
import pytest

import oracle
import synth
from gpu_common import compare

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def vb():
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    import paper_1907_12933_gb300 as m
    from paper_1907_12933_gb300 import build
    build.build()
    return m


# dims, activation, precision, folding on, time budget
CASES = [
    ([30, 40, 20, 4], "sigmoid", "fp32", True, 0.0),
    ([25, 10, 5], "sigmoid", "fp32", True, 0.0),
    ([30, 40, 20, 4], "identity", "fp32", True, 0.0),
    ([24, 30, 16, 5], "relu", "fp32", True, 0.0),      # no wider than 32
    ([30, 40, 36, 33], "relu", "fp32", True, 0.0),     # more outputs than a folded net holds
    ([40, 6], "relu", "fp32", True, 0.0),              # one layer
    ([48, 64, 64, 6], "relu", "fp32", False, 0.0),
    ([48, 64, 64, 6], "relu", "bf16", False, 0.0),
    ([48, 64, 64, 6], "relu", "fp16", False, 0.0),
    ([48, 64, 64, 6], "relu", "bf16", True, 1e6),      # a budget that does not run out
    ([24, 30, 16, 5], "relu", "fp64", True, 0.0),
]


@pytest.mark.parametrize("dims,act,prec,on,budget", CASES)
@pytest.mark.parametrize("graph", [False, True])
def test_batch_through_the_general_passes(vb, dims, act, prec, on, budget, graph):
    net = synth.make_net(830, dims, act, 2.0, "normal")
    qs = [synth.make_query(830, i, dims[0], 1 + i % 3, [2, 40, 6][i % 3] + i) for i in range(9)]
    for q in qs:  # one image, whose outputs lie close together: some boxes hold a witness
        q["image"] = qs[0]["image"]
    y = oracle.eval_point(net, dict(qs[0], pixels=qs[0]["pixels"][:0], k=0), 0)["u"][-dims[-1]:]
    net["b"][-1] += (0.01 * np.arange(dims[-1]) - y).astype(np.float32)
    refs = [oracle.verify(net, q) for q in qs]
    assert sum(0 < o["n_adv"] < o["n_points"] for o in refs) >= 2 and any(o["flip"].any() for o in refs)
    vnet = vb.Net(net)
    vb.set_folding(vnet, on)
    res = vb.result_create_batch(vnet, len(qs), max_points=1 << 15, max_s=3, max_k=64, queue_cap=1 << 18)
    arr, keep = (vb._Query * len(qs))(), []
    for i, q in enumerate(qs):
        keep += [np.ascontiguousarray(q["image"], np.uint8), np.ascontiguousarray(q["pixels"], np.int32)]
        arr[i] = vb._query(keep[-2], keep[-1], q["k"])
    hs = (C.c_void_p * len(qs))(*[r.h for r in res])
    for sched in ("given", "small_first"):
        opt = vb._options(prec, True, True, graph, sched, budget)
        vb._check(vb.lib().vbmc_verify_batch(vnet.h, arr, len(qs), C.byref(opt), hs, C.c_void_p(0)))
        for q, r, o in zip(qs, res, refs):
            n = oracle.space_size(len(q["pixels"]), q["k"])
            g = {"summary": vb.result_summary(r), "n": n, "bitmap": vb.get_verdict_bitmap(r, n),
                 "ties": np.sort(vb.get_ties(r)), "witness": vb.get_witness(r, len(q["pixels"]), dims[0]),
                 **vb.get_coverage(r)}
            compare(g, o, net, q)
    for r in res:
        r.free()
    vnet.free()
