"""The one-launch float product at N = 64 runs as a cluster of four blocks that write into
each other's shared memory: no block may do so before all four have started.

The order is a property of the source (a block that starts late cannot be arranged on the
GPU), so it is read there: between the kernel's entry and its first access to a peer stand
an arrival and a wait of the whole cluster, each reached by every thread.  On the GPU the
product is run many at a time, where the blocks of different clusters compete."""
import os
import re

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SOURCE = os.path.join(ROOT, "paper_1807_01885_gb300", "csrc", "matvec_small.cuh")


def test_cluster_has_started_before_the_first_remote_store():
    with open(SOURCE) as fh:
        code = re.sub(r"//[^\n]*", "", fh.read())
    for kind, op in (("arrive", "barrier.cluster.arrive"), ("wait", "barrier.cluster.wait")):
        assert re.search(r"cluster_%s\(\) \{ asm volatile\(\"%s" % (kind, re.escape(op)), code)
    body = code[code.index("k_product_small("):]
    remote = body.index("map_shared_rank")
    arrive, wait = body.find("cluster_arrive();"), body.find("cluster_wait();")
    assert 0 <= arrive < wait < remote
    # both at the nesting level of the kernel (one) or of its row block (two): not inside a
    # branch that only some threads take
    for at in (arrive, wait):
        assert body[:at].count("{") - body[:at].count("}") <= 2


@pytest.mark.gpu
def test_many_products_at_once(cuda):
    import torch

    from paper_1807_01885_gb300 import bem
    N, count, rounds = 64, 12, 50
    r = np.random.default_rng(0)
    ks = [bem.Kernel(N, 1.0 / N, (4.0 + i) / N, 2.0, 0.3, 1.0, 0.25, precision="fp32") for i in range(count)]
    ps = [torch.tensor(r.standard_normal((N, N)), device=cuda, dtype=torch.float32) for _ in ks]
    alone = []
    for k, p in zip(ks, ps):
        alone.append(k.matvec(p))
        torch.cuda.synchronize()
    streams = [torch.cuda.Stream() for _ in ks]
    outs = [[torch.empty_like(p) for _ in range(rounds)] for p in ps]
    torch.cuda.synchronize()
    for j in range(rounds):
        for k, p, s, o in zip(ks, ps, streams, outs):
            k.matvec(p, o[j], stream=s)
    torch.cuda.synchronize()
    for a, o in zip(alone, outs):
        assert all(torch.equal(a, v) for v in o)
    for k in ks:
        assert k.check_guards() == 0
        k.close()
