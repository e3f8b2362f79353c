"""The calls that a user of this package makes, as cases to be timed.

A case is one of
  verify    one query: the box of s pixels moved by up to k grey levels, through
            vb.verify_query and the getters that read its results (summary,
            coverage masks, verdict bitmap, ties, first witness)
  batch     uneven queries against one net (vb.verify_batch, smallest first)
  search    tiles of one query in a given order, up to the first witness
  shells    shells of growing radius, up to the first witness
  pairs     the covers over a set of image pairs (vb.pair_coverage)
  covers    the covers over the points of one box (vb.enum_coverage)
  learn     one gradient of the tile proposal and its parameters read back
  rank      tile scores and tile orders of the proposal

Nets and queries are drawn as `synth` draws them: weights N(0, w/fan_in), grey
levels uniform in 0..255, distinct pixels. "near" is the number of images from
which the one with the smallest margin is taken: queries close to the decision
boundary are those that a verifier is asked about, and those that need most
rechecks. The summary's times and its counts of points per pass say how a
result was reached and not what it is, so they are no outputs.
"""
import math

import numpy as np
import torch

import paper_1907_12933_gb300 as vb

VERDICT = {"SAFE": 0, "UNSAFE": 1, "TIES_ONLY": 2, "PARTIAL": 3}

# the nets of the benchmark's workloads, and widths that fit no tile
SIGMOID25 = "25-10-5"
RELU512 = "784-512-512-10"
RELU256 = "784-256-256-10"
RELU1024 = "784-1024-1024-1024-10"
ODD300 = "784-300-100-10"
PROPOSAL = "2352-256-256-64"

TIES = 64  # margin ties that a call reads back


def _dims(case):
    return [int(x) for x in case["dims"].split("-")]


def _name(dims):
    return "-".join(str(x) for x in dims)


def verify(name, dims, precision, s, k, **more):
    case = {"name": name, "kind": "verify", "dims": dims, "act": "relu", "precision": precision,
            "s": s, "k": k, "lo": 0, "hi": 0, "coverage": True, "near": 1, "l2": 0.0, "shell": False,
            "threshold": False}
    case.update(more)
    return case


def listed():
    return [
        # the smallest call: a 5x5 image, two pixels, 49 points; launches and copies
        verify("sigmoid25_fp32_s2k3", SIGMOID25, "fp32", 2, 3, act="sigmoid"),
        # a whole box of the 5x5 sigmoid net, 1.4 million points
        verify("sigmoid25_fp32_s5k8", SIGMOID25, "fp32", 5, 8, act="sigmoid"),
        # an interactive check of a 28x28 image: 1,331 points, part of a wave of the chip
        verify("relu512_bf16_s3k5", RELU512, "bf16", 3, 5),
        # the benchmark's query: 11.4 million points of an image near the boundary
        verify("relu512_bf16_s6k7", RELU512, "bf16", 6, 7, near=256),
        # a slice of a box that starts and ends anywhere, verdicts alone, FP16 operands
        verify("relu512_fp16_slice", RELU512, "fp16", 6, 5, near=16, lo=100003, hi=1600001, coverage=False),
        # widths that are no multiple of a tile: the plain FP32 path, inside an L2 ball
        verify("odd300_fp32_l2", ODD300, "fp32", 5, 9, near=16, l2=0.25),
        # three layers of 1024 with every cover, 923,521 points
        verify("relu1024_bf16_s4k15", RELU1024, "bf16", 4, 15, near=16),
        # the same net in E4M3, verdicts alone, 29,791 points
        verify("relu1024_fp8_s3k15", RELU1024, "fp8", 3, 15, near=16, coverage=False),
        # 64 uneven queries of 49 to 21^6 points against one net
        {"name": "relu256_bf16_batch64", "kind": "batch", "dims": RELU256, "act": "relu",
         "precision": "bf16", "nq": 64, "mix": 1004, "s_min": 2, "s_max": 6, "k_min": 3, "k_max": 10,
         "coverage": True, "graph": False},
        # 64 tiles of one box in index order, up to the first witness
        {"name": "relu512_bf16_search64", "kind": "search", "dims": RELU512, "act": "relu",
         "precision": "bf16", "s": 6, "k": 7, "tiles": 64, "near": 32, "shuffle": False},
        # the covers over 8,192 pairs of an image and a noisy copy, FP64
        {"name": "relu512_pairs8192", "kind": "pairs", "dims": RELU512, "act": "relu",
         "n": 8192, "noise": 16, "g": 2.0, "d": 1.0},
        # a mini-batch of the proposal's training: forward, backward, gradients read
        {"name": "proposal_grads_b128", "kind": "learn", "dims": PROPOSAL, "rows": 128},
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _box(rng, most, k_most=15):
    """s and k of a box of at most `most` points, spread over the logarithm of their number."""
    while True:
        want = _log(rng, 49, most)
        s = rng.randint(2, 6)
        k = int((want ** (1.0 / s) - 1) / 2)
        if 1 <= k <= k_most and (2 * k + 1) ** s <= most:
            return s, k


def draw(rng):
    kind = rng.choices(["verify", "batch", "search", "shells", "pairs", "covers", "learn", "rank"],
                       [9, 2, 1, 1, 1, 1, 1, 1])[0]
    near = rng.choice([1, 4, 16, 64])
    if kind == "verify":
        family = rng.choice(["sigmoid", "fused", "fused", "odd", "wide"])
        act = "relu"
        if family == "sigmoid":
            dims, act = [rng.randint(9, 64), rng.randint(5, 32), rng.randint(3, 10)], "sigmoid"
            precision, most = rng.choice([("fp32", 1500000), ("fp64", 100000)])
        elif family == "fused":
            dims = [784, 64 * rng.randint(1, 8), 64 * rng.randint(1, 8), rng.choice([4, 10, 26])]
            precision, most = rng.choice([("bf16", 11390625), ("fp16", 11390625), ("bf16", 400000),
                                          ("fp16", 400000), ("fp32", 1500000), ("fp64", 20000)])
        elif family == "odd":
            dims = [rng.randint(100, 900), rng.randint(20, 700), rng.randint(20, 400), rng.randint(2, 26)]
            precision, most = "fp32", 2500000
        else:
            dims = [784] + [256 * rng.randint(2, 4) for _ in range(rng.randint(2, 3))] + [10]
            precision, most = rng.choice([("bf16", 900000), ("fp16", 900000), ("fp8", 30000), ("fp32", 100000)])
        s, k = _box(rng, most)
        n = (2 * k + 1) ** s
        case = verify("", _name(dims), precision, s, k, act=act, near=near, coverage=rng.random() < 0.7,
                      threshold=rng.random() < 0.15, shell=rng.random() < 0.1,
                      l2=rng.choice([0.0, 0.0, 0.0, rng.uniform(0.1, 0.6)]))
        if rng.random() < 0.3:
            case["lo"] = rng.randrange(n // 2)
            case["hi"] = rng.randrange(case["lo"] + 1, n + 1)
    elif kind == "batch":
        case = {"kind": kind, "dims": _name([784, 64 * rng.randint(2, 4), 64 * rng.randint(2, 4), 10]),
                "act": "relu", "precision": rng.choice(["bf16", "fp16", "fp32"]),
                "nq": int(_log(rng, 4, 64)), "mix": rng.randrange(1 << 30), "coverage": rng.random() < 0.7,
                "graph": rng.random() < 0.3}
        case.update(s_min=2, s_max=5, k_min=3, k_max=10 if case["precision"] != "fp32" else 6)
    elif kind in ("search", "shells"):
        case = {"kind": kind, "dims": _name([784, 64 * rng.randint(2, 8), 64 * rng.randint(2, 8), 10]),
                "act": "relu", "precision": rng.choice(["bf16", "fp16"]), "near": near}
        case["s"], case["k"] = _box(rng, 2000000)
        if kind == "search":
            n = (2 * case["k"] + 1) ** case["s"]
            case.update(tiles=rng.randint(2, min(64, n)), shuffle=rng.random() < 0.5)
    elif kind == "pairs":
        case = {"kind": kind, "dims": rng.choice([RELU512, RELU256, ODD300]), "act": "relu",
                "n": int(_log(rng, 1, 8192)), "noise": rng.randint(1, 32), "g": rng.uniform(1.5, 4.0),
                "d": rng.uniform(0.5, 2.0)}
    elif kind == "covers":
        case = {"kind": kind, "dims": rng.choice([SIGMOID25, RELU256, ODD300]), "act": "relu",
                "g": rng.uniform(1.5, 4.0), "d": rng.uniform(0.5, 2.0)}
        small = case["dims"] == SIGMOID25
        case["act"] = "sigmoid" if small else "relu"
        case["s"], case["k"] = _box(rng, 100000 if small else 10000)
    else:
        case = {"kind": kind, "dims": _name([3 * rng.choice([25, 100, 784]), 32 * rng.randint(2, 8),
                                             32 * rng.randint(2, 8), rng.choice([16, 64, 100])]),
                "rows": int(_log(rng, 1, 256))}
    case.pop("name", None)
    return case


# ------------------------------------------------------------------- inputs

def _net(case, rng):
    """Weights N(0, w/fan_in) in FP64, rounded once: w = 2 and zero biases with ReLU, w = 1
    and biases of the same deviation with the sigmoid."""
    dims, relu = _dims(case), case["act"] == "relu"
    W, b = [], []
    for n_in, n_out in zip(dims, dims[1:]):
        sd = math.sqrt((2.0 if relu else 1.0) / n_in)
        W.append((rng.standard_normal((n_out, n_in)) * sd).astype(np.float32))
        b.append(np.zeros(n_out, np.float32) if relu else (rng.standard_normal(n_out) * sd).astype(np.float32))
    return {"dims": dims, "W": W, "b": b, "act": case["act"]}


def _forward(net, images):
    """Outputs of the net for rows of grey levels, in 64 bits."""
    h = images.astype(np.float64) / 255.0
    for l, (w, b) in enumerate(zip(net["W"], net["b"])):
        h = h @ w.astype(np.float64).T + b.astype(np.float64)
        if l + 1 < len(net["W"]):
            h = np.maximum(h, 0.0) if net["act"] == "relu" else 1.0 / (1.0 + np.exp(-h))
    return h


def _query(case, net, rng, s, near):
    h0 = net["dims"][0]
    images = rng.integers(0, 256, (near, h0), dtype=np.uint8)
    y = np.sort(_forward(net, images), axis=1)
    margin = y[:, -1] - y[:, -2]
    i = int(np.argmin(margin))
    pixels = rng.permutation(h0)[:s].astype(np.int32)
    return images[i], pixels, y[i], float(margin[i])


def _sizes(case):
    """s and k of a batch's queries: part of the case, so its work does not hang on the seed."""
    rng = np.random.default_rng(case["mix"])
    s = rng.integers(case["s_min"], case["s_max"] + 1, case["nq"])
    k = rng.integers(case["k_min"], case["k_max"] + 1, case["nq"])
    return [(int(a), int(b)) for a, b in zip(s, k)]


def _features(case, rng):
    """Rows as vb.proposal_features lays them out (image, place values of six pixels, scaled
    gradient at them) and 0/1 witness labels with at least one witness tile each."""
    f, tiles, rows = _dims(case)[0] // 3, _dims(case)[3], case["rows"]
    X = np.zeros((rows, 3 * f), np.float32)
    T = np.zeros((rows, tiles), np.float32)
    X[:, :f] = rng.integers(0, 256, (rows, f)).astype(np.float32) / 255
    for r in range(rows):
        pix = rng.permutation(f)[:6]
        place = 15.0 ** -np.arange(6)
        X[r, f + pix] = place
        X[r, 2 * f + pix] = np.clip(place * rng.standard_normal(6) * 0.3, -16, 16)
        a = rng.integers(0, tiles)
        T[r, a:a + 1 + rng.integers(0, max(1, tiles // 4))] = 1
    return X, T


def _proposal(case, rng):
    """Layers W, b of a proposal net as training starts from them."""
    d = _dims(case)
    return [((rng.standard_normal((d[l], d[l - 1])) * math.sqrt(2.0 / d[l - 1])).astype(np.float32),
             (rng.standard_normal(d[l]) * 0.01).astype(np.float32)) for l in (1, 2, 3)]


def _drawn(case, seed):
    """Everything the seed decides, on the host."""
    rng = np.random.default_rng([int(seed), 1907])
    kind = case["kind"]
    if kind in ("learn", "rank"):
        return {"layers": _proposal(case, rng), "X": _features(case, rng)}
    net = _net(case, rng)
    out = {"net": net}
    if kind == "batch":
        out["queries"] = []
        for s, k in _sizes(case):
            image, pixels, _, margin = _query(case, net, rng, s, 1)
            out["queries"].append({"image": image, "pixels": pixels, "k": k, "margin": margin})
    elif kind == "pairs":
        a = rng.integers(0, 256, (case["n"], net["dims"][0]))
        e = rng.integers(-case["noise"], case["noise"] + 1, a.shape)
        out["a"], out["b"] = a.astype(np.uint8), np.clip(a + e, 0, 255).astype(np.uint8)
    else:
        image, pixels, y, margin = _query(case, net, rng, case["s"], case.get("near", 1))
        out.update(image=image, pixels=pixels, margin=margin, y=y)
        if kind == "search":
            order = np.arange(case["tiles"], dtype=np.int32)
            out["order"] = rng.permutation(order).astype(np.int32) if case["shuffle"] else order
    return out


def prepare(case, seed):
    d = _drawn(case, seed)
    state = {"case": case, "d": d}
    kind = case["kind"]
    if kind in ("learn", "rank"):
        prop = vb.Proposal(tuple(_dims(case)), max_batch=max(case["rows"], 1), seed=1)
        for l, (w, b) in enumerate(d["layers"], start=1):
            prop.set_params(l, w, b)
        state.update(prop=prop, X=torch.from_numpy(d["X"][0]).cuda(), T=torch.from_numpy(d["X"][1]).cuda())
        return state
    net = state["net"] = vb.Net(d["net"])
    precision = case.get("precision")
    if precision in ("bf16", "fp16", "fp8"):
        vb.net_prepare(net, precision)
    if kind == "batch":
        sizes = _sizes(case)
        state["results"] = vb.result_create_batch(net, case["nq"], max_points=0, max_s=max(s for s, _ in sizes),
                                                  max_k=max(k for _, k in sizes))
    elif kind != "pairs":
        n = (2 * case["k"] + 1) ** case["s"]
        state["res"] = vb.Result(net, max_points=n, max_s=case["s"], max_k=case["k"],
                                 queue_cap=max(4096, min(n, 1 << 24)))
    if kind == "verify":
        state["filter"] = (vb.FILTER_L2 if case["l2"] else 0) | (vb.FILTER_SHELL if case["shell"] else 0)
        state["l2_max"] = _l2_max(case)
        # a reference value between the two largest outputs
        state["threshold"] = float(d["y"][-1] - 0.3 * d["margin"]) if case["threshold"] else None
    return state


def _l2_max(case):
    """A ball that reaches the given share of the way to the box's corner, in grey levels squared."""
    return int(case["l2"] * case["s"] * case["k"] ** 2)


# ---------------------------------------------------------------------- run

def _summary(r):
    return {"verdict": VERDICT[r["verdict"]], "D": r["D"], "base_margin": r["base_margin"],
            "n_points": r["n_points"], "n_adversarial": r["n_adversarial"],
            "first_witness": -1 if r["first_witness"] is None else r["first_witness"], "n_ties": r["n_ties"]}


def run(state):
    case, d, kind = state["case"], state["d"], state["case"]["kind"]
    if kind == "verify":
        res, n = state["res"], (2 * case["k"] + 1) ** case["s"]
        r = vb.verify_query(state["net"], res, d["image"], d["pixels"], case["k"], lo=case["lo"], hi=case["hi"],
                            precision=case["precision"], coverage=case["coverage"], bitmap=True,
                            filter=state["filter"], l2_max=state["l2_max"], threshold=state["threshold"])
        out = _summary(r)
        out["bitmap"] = vb.get_verdict_bitmap(res, n)
        ties = vb.get_ties(res, cap=TIES)  # the first ones, in order; most boxes hold none
        out["ties"] = np.append(ties, np.full(TIES - len(ties), -1))
        if case["coverage"]:
            out.update(vb.get_coverage(res))
        w = vb.get_witness(res, case["s"], _dims(case)[0])
        if w is None:  # the same layout without one
            w = {"index": -1, "steps": np.zeros(case["s"], np.int32), "image": d["image"], "margin": 0.0}
        out["witness"] = w
        return out
    if kind == "batch":
        rs = vb.verify_batch(state["net"], state["results"], d["queries"], precision=case["precision"],
                             coverage=case["coverage"], graph=case["graph"], schedule="small_first")
        rows = [dict(_summary(r), **(vb.get_coverage(x) if case["coverage"] else {}))
                for r, x in zip(rs, state["results"])]
        return {key: np.stack([row[key] for row in rows]) for key in rows[0]}
    if kind == "search":
        r = vb.search_query(state["net"], state["res"], d["image"], d["pixels"], case["k"], d["order"],
                            precision=case["precision"])
        return dict(_summary(r), tiles_checked=r["tiles_checked"], points_checked=r["points_checked"],
                    witness_tile=-1 if r["witness_tile"] is None else r["witness_tile"])
    if kind == "shells":
        r = vb.shell_search(state["net"], state["res"], d["image"], d["pixels"], case["k"],
                            precision=case["precision"])
        return dict(_summary(r), radius=-1 if r["radius"] is None else r["radius"],
                    points_checked=r["points_checked"], ties_total=r["ties_total"])
    if kind == "pairs":
        return vb.pair_coverage(state["net"], d["a"], d["b"], g=case["g"], d=case["d"])
    if kind == "covers":
        return vb.enum_coverage(state["net"], state["res"], d["image"], d["pixels"], case["k"], g=case["g"],
                                d=case["d"])
    prop, X = state["prop"], state["X"]
    if kind == "learn":
        loss = prop.grads(X, state["T"])
        return {"loss": loss, "layers": [prop.params(l) for l in (1, 2, 3)]}
    tiles = _dims(case)[3]
    scores = torch.empty((case["rows"], tiles), dtype=torch.float32, device="cuda")
    order = torch.empty((case["rows"], tiles), dtype=torch.int32, device="cuda")
    prop.scores(X, scores, order)
    return {"scores": scores, "order": order}


# --------------------------------------------------------------------- work

def _points(case):
    """Points of the box that the call has to check (clipping aside)."""
    s, k = case["s"], case["k"]
    n = (2 * k + 1) ** s
    inside = float(n)
    if case.get("l2"):
        ways = {0: 1}
        for _ in range(s):
            nxt = {}
            for q, c in ways.items():
                for t in range(-k, k + 1):
                    if q + t * t <= _l2_max(case):
                        nxt[q + t * t] = nxt.get(q + t * t, 0) + c
            ways = nxt
        inside = float(sum(ways.values()))
    if case.get("shell"):
        inside *= 1.0 - ((2 * k - 1) / (2.0 * k + 1)) ** s
    lo, hi = case.get("lo", 0), case.get("hi", 0) or n
    return inside * (hi - lo) / n


def work(case):
    """What a call cannot do without: weights and images read, masks and bitmap written, one
    evaluation of the net for the unperturbed image, and for each point the terms in which it
    differs from that image, one multiply-add per changed pixel and output (Eq. 1 on the change:
    the least that any treatment of the layers between leaves over; a sigmoid net: per changed
    pixel and neuron of layer 1, and whole products behind it)."""
    d, kind = _dims(case), case["kind"]
    weights = 4.0 * sum(a * b + b for a, b in zip(d, d[1:]))
    full = 2.0 * sum(a * b for a, b in zip(d, d[1:]))
    tail = 2.0 * sum(a * b for a, b in zip(d[1:], d[2:]))
    masks = sum(d[1:]) / 4.0 + sum(a * b for a, b in zip(d[1:], d[2:])) / 4.0

    def point(s, outs):
        return 2.0 * s * outs if case["act"] == "relu" else tail + 2.0 * s * d[1]

    if kind == "verify":
        return {"bytes": weights + d[0] + masks + (2 * case["k"] + 1) ** case["s"] / 8.0,
                "flops": full + _points(case) * point(case["s"], d[-1])}
    if kind == "batch":
        sizes = _sizes(case)
        return {"bytes": weights + len(sizes) * (d[0] + masks),
                "flops": sum(full + (2.0 * k + 1) ** s * point(s, d[-1]) for s, k in sizes)}
    if kind == "search":  # one tile at least
        return {"bytes": weights + d[0],
                "flops": full + (2.0 * case["k"] + 1) ** case["s"] / case["tiles"] * point(case["s"], d[-1])}
    if kind == "shells":  # the unperturbed image at least
        return {"bytes": weights + d[0], "flops": full}
    if kind == "pairs":
        return {"bytes": weights + 2.0 * case["n"] * d[0] + 2 * masks, "flops": 2.0 * case["n"] * full}
    if kind == "covers":  # value and distance covers read every potential
        return {"bytes": weights + d[0] + 2 * masks,
                "flops": full + (2.0 * case["k"] + 1) ** case["s"] * point(case["s"], sum(d[1:]))}
    if kind == "learn":  # forward, both products of the backward pass but the input's; W, b and both gradients read
        return {"bytes": 4.0 * case["rows"] * (d[0] + d[3]) + 4 * weights,
                "flops": case["rows"] * (3.0 * full - 2.0 * d[0] * d[1])}
    return {"bytes": weights + 4.0 * case["rows"] * (d[0] + 2 * d[3]), "flops": case["rows"] * full}


# -------------------------------------------------------------------- exact

def _softmax_grads(layers, X, T):
    """Loss and gradients of the listwise cross-entropy, in 64 bits: the mean over rows with a witness."""
    Ws = [(w.astype(np.float64), b.astype(np.float64)) for w, b in layers]
    h = [X.astype(np.float64)]
    for l, (w, b) in enumerate(Ws):
        z = h[-1] @ w.T + b
        h.append(np.maximum(z, 0.0) if l < 2 else z)
    z = h[3] - h[3].max(axis=1, keepdims=True)
    logp = z - np.log(np.exp(z).sum(axis=1, keepdims=True))
    t = T.astype(np.float64)
    t /= t.sum(axis=1, keepdims=True)
    loss = float(-(t * logp).sum(axis=1).mean())
    g, out = (np.exp(logp) - t) / len(X), []
    for l in (2, 1, 0):
        w, b = Ws[l]
        out.insert(0, {"W": w, "b": b, "gW": g.T @ h[l], "gb": g.sum(axis=0)})
        g = (g @ w) * (h[l] > 0)
    return loss, out, h[3]


def exact(case, seed):
    """The computed numbers in 64 bits: base margins, the proposal's scores, loss and gradients.
    Verdicts, indices and masks are whole numbers and have no such value."""
    kind = case["kind"]
    if kind in ("pairs", "covers"):
        return None
    d = _drawn(case, seed)
    if kind in ("learn", "rank"):
        loss, layers, scores = _softmax_grads(d["layers"], *d["X"])
        if kind == "rank":
            return {"scores": scores, "order": None}
        return {"loss": loss, "layers": layers}
    if kind == "batch":
        return {"base_margin": np.array([q["margin"] for q in d["queries"]])}
    if kind == "verify" and case["threshold"]:
        # Eq. 11's margin at the unperturbed image: max(y_D - V, V - max of the others)
        v = float(d["y"][-1] - 0.3 * d["margin"])
        return {"base_margin": max(float(d["y"][-1]) - v, v - float(d["y"][-2]))}
    return {"base_margin": d["margin"]}
