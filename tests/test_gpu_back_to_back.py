"""Fused calls back to back on one stream, each reading what the one before
wrote or writing what it read: a kernel is set up while the one before
drains, and must not touch memory before that one is complete.  Three buffers
are passed round, in place and out of place, with the layouts mixed, on the
default stream, on another one and in a captured graph; whole numbers, so
the last buffer shows every one of the calls (odd p: no factor of two is lost
when a sum wraps)."""
import numpy as np
import pytest
import torch

from gpu_util import bits, expect_bits, host_inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    from paper_2109_12626_gb300 import build as B
    B.build()
    import paper_2109_12626_gb300 as P
    return P


# layouts of the calls in turn: 0 auto, 1 stream, 2 tile, 3 split, 4 bulk, 5 tree
@pytest.mark.parametrize("p,m,modes", [(3, 1, (0,)), (7, 1000, (0, 2)), (37, 262144, (1, 5)),
                                       (289, 8192, (2, 5, 3)), (33, 300001, (1, 3)),
                                       (65, 65536, (4, 1))])
@pytest.mark.parametrize("where", ["default", "stream", "graph"])
def test_chained_calls(pkg, orc, p, m, modes, where):
    dev = torch.device("cuda:0")
    x = host_inputs("int32", 131, p, m, lo=-1000, hi=1000)
    calls = 12
    want = x
    for _ in range(calls):
        want = np.broadcast_to(orc.tree_fold(np.ascontiguousarray(want), orc.I32, orc.DUAL), (p, m))
    plans = []  # one per call, so that no upload of pointers comes between the kernels
    for k in range(calls):
        plans.append(pkg.Plan(p, m, "int32", 1))
        if modes[k % len(modes)]:
            plans[-1].set(pkg.OPT_FUSED_MODE, modes[k % len(modes)])
    bufs = [torch.empty((p, m), dtype=torch.int32, device=dev) for _ in range(3)]
    rows = [list(b) for b in bufs]
    x_dev = torch.from_numpy(x).to(dev)
    at = [0]
    for k in range(calls):  # every third call in place
        at.append(at[-1] if k % 3 == 2 else (at[-1] + 1) % 3)

    def chain():
        bufs[0].copy_(x_dev)
        for k in range(calls):
            plans[k].allreduce(rows[at[k]], rows[at[k + 1]])

    torch.cuda.synchronize()
    if where == "default":
        chain()
        chain()
    else:
        stream = torch.cuda.Stream()
        with torch.cuda.stream(stream):
            chain()
        stream.synchronize()
        if where == "graph":
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph, stream=stream):
                chain()
            for b in bufs:
                b.fill_(-1)
            for _ in range(3):
                graph.replay()
    torch.cuda.synchronize()
    got = bits(bufs[at[-1]])
    assert (got == expect_bits(np.ascontiguousarray(want))).all()
    for plan in plans:
        plan.sync()
        plan.close()
