"""Folded nets (first pass of ReLU nets whose neurons mostly keep their sign in the
box) against the FP64 oracle and against the general passes, at the sizes where
they can go wrong: no node at all, groups of 4 rows full and ragged, coefficients
past shared memory, more nodes than a folded net holds, ranges that start and end
anywhere, one-point boxes, clipped pixels, base ties, filters, Eq. 11."""
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


# dims, s, k, seed, precision: widths of one group, ragged groups, 2..5 layers
CASES = [
    ([40, 33, 5], 3, 6, 1, "fp32"),
    ([40, 33, 2], 1, 127, 2, "fp32"),
    ([64, 64, 64, 10], 4, 3, 3, "bf16"),
    ([64, 64, 64, 10], 3, 12, 4, "fp16"),
    ([100, 70, 50, 31], 3, 9, 5, "fp32"),
    ([100, 45, 40, 35, 7], 3, 7, 6, "fp32"),
    ([60, 64, 64, 64, 64, 32], 2, 30, 7, "bf16"),
    ([784, 512, 512, 10], 2, 9, 8, "bf16"),
    ([784, 256, 512, 256, 10], 2, 11, 9, "fp8"),
    ([784, 256, 256, 10], 16, 0, 10, "bf16"),
    ([30, 36, 36, 6], 5, 2, 11, "fp32"),
]


@pytest.mark.parametrize("dims,s,k,seed,prec", CASES)
@pytest.mark.parametrize("bias", ["zero", "normal"])
def test_against_oracle(vb, dims, s, k, seed, prec, bias):
    net = synth.make_net(700 + seed, dims, "relu", 2.0, bias)
    q = synth.make_query(700 + seed, seed, dims[0], s, k)
    n = oracle.space_size(s, k)
    compare(run_gpu(vb, net, q, prec), oracle.verify(net, q), net, q)
    lo, hi = n // 3, n - n // 5
    if lo < hi:
        compare(run_gpu(vb, net, q, prec, lo=lo, hi=hi), oracle.verify(net, q, lo=lo, hi=hi), net, q)


@pytest.mark.parametrize("prec", ["fp32", "bf16"])
@pytest.mark.parametrize("k", [2, 20, 60, 127])
def test_nodes_from_none_to_more_than_a_folded_net_holds(vb, prec, k):
    """64 to 192 hidden neurons: the count of those that can change sign grows with k
    past the 128 a folded net holds (the general passes then run); both ways and the
    FP64 pass agree on everything."""
    net = synth.make_net(811, [48, 64, 64, 64, 9], "relu", 2.0, "normal")
    q = synth.make_query(811, 3, 48, 2, k)
    vnet = vb.Net(net)
    got = {}
    for on in (True, False):
        vb.set_folding(vnet, on)
        got[on] = run_gpu(vb, net, q, prec, vbnet=vnet)
    ref = run_gpu(vb, net, q, "fp64", vbnet=vnet)
    for g in got.values():
        for key in ("flip", "flip_tie", "ss", "ss_tie", "bitmap", "ties"):
            np.testing.assert_array_equal(g[key], ref[key], err_msg=key)
        for key in ("n_adversarial", "first_witness", "n_ties", "D", "n_points"):
            assert g["summary"][key] == ref["summary"][key]
    vnet.free()


def test_many_nodes_past_shared_memory(vb):
    """96 hidden neurons that nearly all cross, 20 outputs and 8 pixels: more coefficient
    entries than shared memory keeps."""
    net = synth.make_net(812, [20, 48, 48, 20], "relu", 2.0, "normal")
    q = synth.make_query(812, 1, 20, 8, 1)
    q["image"] = np.full(20, 128, np.uint8)
    for k, s in ((1, 8), (60, 2)):
        qq = dict(q, pixels=q["pixels"][:s], k=k)
        compare(run_gpu(vb, net, qq, "fp32"), oracle.verify(net, qq), net, qq)


def test_base_ties_and_dead_neurons(vb):
    """A neuron whose base potential is exactly 0, one with no weights at all, and two
    equal outputs: every point is a tie of some kind and reaches the FP64 pass."""
    net = synth.make_net(813, [24, 40, 36, 4], "relu", 2.0, "zero")
    q = synth.make_query(813, 2, 24, 2, 5)
    net["W"][0][3] = 0.0
    net["W"][1][:, 7] = 0.0
    net["W"][1][5] = 0.0
    net["W"][2][2] = net["W"][2][1]
    o = oracle.verify(net, q)
    compare(run_gpu(vb, net, q, "fp32"), o, net, q)


@pytest.mark.parametrize("filt", [1, 2, 3])
@pytest.mark.parametrize("thr", [False, True])
def test_filters_and_threshold(vb, filt, thr):
    net = synth.make_net(814, [50, 64, 64, 8], "relu", 2.0, "normal")
    q = synth.make_query(814, 1, 50, 3, 9)
    y = oracle.eval_point(net, dict(q, pixels=q["pixels"][:0], k=0), 0)["u"][-8:]
    kw = {"filter": filt, "l2_max": 150}
    if thr:
        kw.update(property=1, threshold=float(np.sort(y)[-1] - 0.02))
    o = oracle.verify(net, dict(q, **kw))
    n = oracle.space_size(3, 9)
    vnet = vb.Net(net)
    res = vb.Result(vnet, max_points=n, max_s=3, max_k=9, queue_cap=n)
    s = vb.verify_query(vnet, res, q["image"], q["pixels"], 9, precision="bf16", filter=filt, l2_max=150,
                        threshold=kw.get("threshold"))
    g = {"summary": s, "n": n, "bitmap": vb.get_verdict_bitmap(res, n), "ties": np.sort(vb.get_ties(res)),
         "witness": vb.get_witness(res, 3, 50), **vb.get_coverage(res)}
    compare(g, o, net, q)
    res.free()
    vnet.free()


@pytest.mark.parametrize("prec", ["bf16", "fp32"])
@pytest.mark.parametrize("graph", [False, True])
def test_batch_of_folded_and_other_queries(vb, prec, graph):
    """Queries of very different k in one batch: some fold, some do not."""
    net = synth.make_net(815, [48, 64, 128, 128, 6], "relu", 2.0, "normal")
    qs = [synth.make_query(815, i, 48, 1 + i % 3, [2, 110, 5, 9][i % 4] if i % 3 < 2 else 6) for i in range(14)]
    vnet = vb.Net(net)
    res = vb.result_create_batch(vnet, len(qs), max_points=1 << 16, max_s=3, max_k=110, queue_cap=1 << 18)
    for sched in ("given", "small_first"):
        sums = vb.verify_batch(vnet, res, qs, precision=prec, bitmap=True, graph=graph, schedule=sched)
        for q, r, s in zip(qs, res, sums):
            n = oracle.space_size(len(q["pixels"]), q["k"])
            g = {"summary": s, "n": n, "bitmap": vb.get_verdict_bitmap(r, n), "ties": np.sort(vb.get_ties(r)),
                 "witness": vb.get_witness(r, len(q["pixels"]), 48), **vb.get_coverage(r)}
            compare(g, oracle.verify(net, q), net, q)
    for r in res:
        r.free()
    vnet.free()


def test_fp32_bound_holds_far_from_the_tie_band(vb):
    """Nearly equal outputs make small margins over a whole box: every verdict as the FP64
    pass decides it, whichever of the folded net's two evaluations decided it."""
    net = synth.make_net(816, [60, 128, 64, 5], "relu", 2.0, "normal")
    net["W"][2][1] = net["W"][2][0] * np.float32(1.0 + 2.0 ** -20)
    q = synth.make_query(816, 4, 60, 3, 10)
    vnet = vb.Net(net)
    a = run_gpu(vb, net, q, "bf16", vbnet=vnet)
    b = run_gpu(vb, net, q, "fp64", vbnet=vnet)
    for key in ("flip", "flip_tie", "ss", "ss_tie", "bitmap", "ties"):
        np.testing.assert_array_equal(a[key], b[key], err_msg=key)
    assert a["summary"]["n_adversarial"] == b["summary"]["n_adversarial"]
    vnet.free()


def test_tie_band_points_are_settled_on_the_folded_net(vb):
    """A hidden neuron whose potential is exactly 0 at some points of the box, and two
    outputs equal at every point: sign ties, SS pairs under ties and margin ties as the
    oracle has them, without the FP64 pass on the whole net."""
    net = synth.make_net(818, [12, 24, 20, 4], "relu", 2.0, "zero")
    q = synth.make_query(818, 2, 12, 2, 12)
    p0, p1 = (int(p) for p in q["pixels"])
    q["image"][p0], q["image"][p1] = 100, 103
    net["W"][0][5] = 0.0  # u = (x_p0 - x_p1) / 2: 0 where the steps differ by 3
    net["W"][0][5, p0], net["W"][0][5, p1] = 0.5, -0.5
    for same_outputs in (False, True):
        if same_outputs:
            D = oracle.eval_point(net, q, 0)["D"]
            net["W"][2][(D + 1) % 4] = net["W"][2][D]
        o = oracle.verify(net, q)
        assert o["flip_tie"].any() and o["ss_tie"].any() and (o["n_ties"] > 0) == same_outputs
        g = run_gpu(vb, net, q, "fp32")
        compare(g, o, net, q)


@pytest.mark.parametrize("s,k,lo,hi", [(0, 5, 0, 0), (1, 0, 0, 0), (1, 1, 0, 0), (2, 63, 1, 16000),
                                       (5, 3, 33, 34), (5, 3, 31, 16801), (3, 2, 0, 125), (11, 1, 5, 177001)])
def test_units_of_the_last_digit(vb, s, k, lo, hi):
    """Ranges whose ends fall anywhere in the 4-digit pieces of the last pixel's digit, a
    single point, one digit value, and more pixels than a box usually has."""
    net = synth.make_net(819, [30, 64, 64, 6], "relu", 2.0, "normal")
    q = synth.make_query(819, 5, 30, s, k)
    n = oracle.space_size(s, k)
    hi = min(hi, n)
    compare(run_gpu(vb, net, q, "bf16", lo=lo, hi=hi), oracle.verify(net, q, lo=lo, hi=hi), net, q)


@pytest.mark.parametrize("dims", [[20, 7, 5, 3], [20, 33, 64, 10], [20, 31, 32, 32], [20, 65, 1, 2]])
def test_covered_fraction_of_dense_and_sparse_masks(vb, dims):
    """Eq. 3's fraction from masks whose rows start anywhere in a word, against the
    oracle's loop over pairs."""
    net = synth.make_net(820, dims, "relu", 2.0, "normal")
    vnet = vb.Net(net)
    _, sw = vnet.mask_words()
    bits = sum(a * b for a, b in zip(dims[1:], dims[2:]))
    rng = np.random.default_rng(820)
    import ctypes as C
    for share in (0.0, 0.002, 0.5, 1.0):
        m = np.packbits(rng.random(32 * sw) < share, bitorder="little").view(np.uint32)
        if bits % 32:
            m[bits // 32] &= (1 << (bits % 32)) - 1
        f = C.c_double()
        assert vb.lib().vbmc_covered_fraction(vnet.h, 0, m.ctypes.data_as(C.POINTER(C.c_uint32)), C.byref(f)) == 0
        assert f.value == oracle.ss_covered_fraction(dims, m)
    vnet.free()


@pytest.mark.parametrize("prec,dims,s,k,tiles,extra", [
    ("bf16", [64, 64, 64, 10], 3, 12, 64, {}),
    ("bf16", [64, 64, 64, 10], 3, 12, 257, {"queue_cap": 40}),
    ("fp32", [40, 70, 33, 5], 5, 3, 100, {"filter": 3, "l2_max": 20}),
    ("fp32", [40, 70, 33, 5], 2, 5, 300, {"threshold": 0.0}),
    ("fp8", [784, 256, 256, 10], 3, 6, 33, {}),
    ("bf16", [784, 512, 512, 10], 5, 10, 7, {}),
])
@pytest.mark.parametrize("ties", [False, True])
def test_tile_groups_of_a_search(vb, prec, dims, s, k, tiles, extra, ties):
    """Searches whose tiles go in groups against the same tiles one by one (a search that
    asks for coverage) and against the general passes: orders with the witness early,
    late and nowhere, tiles that straddle words, more tiles than points, queues that
    overflow in a group, ties, filters; and calls after it add nothing to its counters."""
    net = synth.make_net(821, dims, "relu", 2.0, "normal")
    q = synth.make_query(821, 4, dims[0], s, k)
    extra = dict(extra)
    cap = extra.pop("queue_cap", 1 << 20)
    if ties:  # an output equal to the decided one everywhere: every point is a margin tie
        if oracle.space_size(s, k) > 20000 or extra.get("threshold") is not None:
            pytest.skip("a tie at every point")
        D = oracle.eval_point(net, q, 0)["D"]
        net["W"][-1][(D + 1) % dims[-1]] = net["W"][-1][D]
        net["b"][-1][(D + 1) % dims[-1]] = net["b"][-1][D]
    vnet = vb.Net(net)
    res = vb.Result(vnet, max_s=s, max_k=k, queue_cap=cap)
    rng = np.random.default_rng(821)
    keys = ("verdict", "n_points", "n_adversarial", "first_witness", "n_ties", "tiles_checked",
            "points_checked", "witness_tile", "base_label")

    def run(order, **kw):
        try:
            r = vb.search_query(vnet, res, q["image"], q["pixels"], k, order, precision=prec, **extra, **kw)
        except vb.VbmcError as e:
            return type(e), str(e)
        at = vb.get_witness(res, s, dims[0])["index"] if r["n_adversarial"] else None
        return [r.get(x) for x in keys] + [at, sorted(vb.get_ties(res))]

    for order in (np.arange(tiles), np.arange(tiles)[::-1], rng.permutation(tiles)):
        got = run(order)
        assert got == run(order, coverage=True)
        if cap == 1 << 20:
            vb.set_folding(vnet, False)
            assert got == run(order)
            vb.set_folding(vnet, True)


@pytest.mark.parametrize("dims,s,k", [([20, 33, 5], 2, 4), ([20, 1, 2], 1, 100), ([30, 257, 64, 3], 2, 9),
                                      ([40, 1000, 700, 7], 1, 3), ([25, 31, 32, 33, 32], 3, 2)])
def test_queued_points_shared_by_a_cluster(vb, dims, s, k):
    """Sigmoid nets (general passes) with two equal outputs: every point is a margin tie and
    is settled by the FP64 pass, each by a cluster of CTAs; more points than clusters,
    layers of fewer neurons than a warp, of more than a warp per CTA, odd ones."""
    net = synth.make_net(822, dims, "sigmoid", 2.0, "normal")
    q = synth.make_query(822, 6, dims[0], s, k)
    D = oracle.eval_point(net, q, 0)["D"]
    net["W"][-1][(D + 1) % dims[-1]] = net["W"][-1][D]
    net["b"][-1][(D + 1) % dims[-1]] = net["b"][-1][D]
    o = oracle.verify(net, q)
    assert o["n_ties"] == oracle.space_size(s, k)
    g = run_gpu(vb, net, q, "fp32")
    assert g["summary"]["n_recheck"][3] == o["n_ties"]
    compare(g, o, net, q)
