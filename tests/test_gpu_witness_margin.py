"""The margin that comes with a witness: FP64 on the whole net, against extended precision
with the bound of its own roundings, however the query was decided."""
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


def margin_and_bound(net, x, x0, s):
    """y_D - max y_i at x and what FP64 may be off by. A sum of m non-zero terms whose lanes
    share K inputs passes at most min(m, ceil(K / 32)) roundings in a lane, 5 over the lanes and
    1 for the bias, each of at most u times the terms' magnitudes; layer 1 is that of the
    unperturbed image x0 (whose lanes may hold K / 32 + 16, and v / 255 rounds) plus s terms
    for the changed pixels. An activation is 1-Lipschitz (sigmoid: 1/4, and 2 u of its own)."""
    u, f = 2.0 ** -53, np.longdouble
    act, L = net["act"], len(net["W"])
    h0, h, E = x0.astype(f) / 255, x.astype(f) / 255, None
    for l, (W, b) in enumerate(zip(net["W"], net["b"])):
        W, b = W.astype(f), b.astype(f)
        m = np.minimum((W != 0).sum(1), -(-W.shape[1] // 32)) + 7
        mag = np.abs(W) @ np.abs(h) + np.abs(b)
        if l == 0:
            mag = np.abs(W) @ (np.abs(h0) + np.abs(h - h0)) + np.abs(b)
            E = (m + 17 + s + 3) * u * mag
        else:
            E = np.abs(W) @ E + m * u * mag
        h, h0 = W @ h + b, W @ h0 + b
        if l + 1 < L:
            if act == "relu":
                h, h0 = np.maximum(h, 0), np.maximum(h0, 0)
            elif act == "sigmoid":
                h, h0, E = 1 / (1 + np.exp(-h)), 1 / (1 + np.exp(-h0)), E / 4 + 4 * u
    D = int(np.argmax(h0))
    i = max((j for j in range(len(h)) if j != D), key=lambda j: h[j])
    return h[D] - h[i], E[D] + max(E) + u * abs(h[D] - h[i])


def centred(net, q, step):
    """Output biases that bring the outputs at the unperturbed image close together."""
    n = net["dims"][-1]
    y = oracle.eval_point(net, dict(q, pixels=q["pixels"][:0], k=0), 0)["u"][-n:]
    net["b"][-1] = (net["b"][-1] + (step * np.arange(n) - y)).astype(np.float32)


CASES = [  # dims, activation, precision, non-zero weights a row (0: all), trials
    ([16, 64, 64, 64, 6], "relu", "bf16", 3, 30),
    ([16, 64, 64, 64, 6], "relu", "fp32", 3, 30),
    ([300, 200, 100, 7], "relu", "fp32", 0, 4),
    ([784, 512, 512, 10], "relu", "bf16", 0, 3),
    ([60, 1024, 1024, 10], "relu", "bf16", 0, 2),
    ([60, 40, 33, 5], "sigmoid", "fp32", 0, 6),
    ([50, 1, 3, 2], "identity", "fp64", 0, 6),
    ([40, 12], "relu", "fp32", 0, 6),
    ([70, 100, 300], "identity", "fp32", 0, 3),
]


@pytest.mark.parametrize("dims,act,prec,nnz,trials", CASES)
@pytest.mark.parametrize("fold", [True, False])
def test_margin_of_a_witness(vb, dims, act, prec, nnz, trials, fold):
    rng = np.random.default_rng(890)
    seen = 0
    for trial in range(trials):
        net = synth.make_net(890 + trial, dims, act, 2.0, "normal")
        for l in range(len(dims) - 1):
            if nnz:
                keep = np.zeros(net["W"][l].shape, dtype=bool)
                for row in keep:
                    row[rng.permutation(len(row))[:nnz]] = True
                net["W"][l] = np.where(keep, net["W"][l] * np.sqrt(dims[l] / nnz), 0).astype(np.float32)
        q = synth.make_query(890 + trial, 1, dims[0], 3, 20)
        centred(net, q, 0.001)
        vnet = vb.Net(net)
        vb.set_folding(vnet, fold)
        res = vb.Result(vnet, max_s=3, max_k=20, queue_cap=1 << 17)
        vb.verify_query(vnet, res, q["image"], q["pixels"], 20, precision=prec, coverage=False, bitmap=False)
        w = vb.get_witness(res, 3, dims[0])
        if w is not None:
            seen += 1
            m, bound = margin_and_bound(net, w["image"], np.asarray(q["image"]), 3)
            assert abs(np.longdouble(w["margin"]) - m) <= bound, (trial, w["margin"], m, bound)
        res.free()
        vnet.free()
    assert seen >= trials // 2
