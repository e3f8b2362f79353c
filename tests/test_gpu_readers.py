"""Several threads reading the covers of one result."""
import threading

import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


def test_covers_read_by_several_threads():
    import paper_1907_12933_gb300 as vb
    from paper_1907_12933_gb300 import build
    build.build()
    net = synth.make_net(910, [40, 256, 250, 10], "relu", 2.0, "normal")
    q = synth.make_query(910, 1, 40, 2, 20)
    o = oracle.verify(net, q)
    vnet = vb.Net(net)
    res = vb.Result(vnet, max_s=2, max_k=20)
    vb.verify_query(vnet, res, q["image"], q["pixels"], 20, precision="fp32", bitmap=False)
    wrong = []

    def read():
        for _ in range(50):
            c = vb.get_coverage(res)
            if any(not np.array_equal(c[k], o[k]) for k in ("flip", "flip_tie", "ss", "ss_tie")):
                wrong.append(c)

    threads = [threading.Thread(target=read) for _ in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not wrong
    res.free()
    vnet.free()
