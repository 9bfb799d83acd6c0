"""The fused layouts on rows of 4-byte elements that are only 4-byte
aligned: units of four elements, side by side in groups of 4G columns, with
the columns past the last whole group one by one.  Bit for bit against the
oracle around the group sizes (32, 64 and 128 columns) and the layout rule's
edges, with guard words on both sides of every output row."""
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


CASES = [("int32", 3, 1), ("float32", 7, 31), ("int32", 7, 32), ("float32", 16, 127),
         ("int32", 40, 128), ("float32", 36, 129), ("int32", 130, 63), ("float32", 288, 511),
         ("int32", 288, 513), ("float32", 1152, 255), ("int32", 1152, 4097), ("float32", 64, 62261),
         ("float32", 31, 8257), ("int32", 300, 9731)]


@pytest.mark.parametrize("kind,p,m", CASES)
@pytest.mark.parametrize("mode", [0, 1, 2, 3, 5], ids=["auto", "stream", "tile", "split", "tree"])
@pytest.mark.parametrize("topology", ["dual", "single"])
def test_unaligned_rows_match_oracle(pkg, orc, kind, p, m, mode, topology):
    x = host_inputs(kind, 121, p, m)
    want = expect_bits(orc.tree_fold(x, orc.F32 if kind == "float32" else orc.I32,
                                     orc.DUAL if topology == "dual" else orc.SINGLE))
    dev = torch.device("cuda:0")
    dt = torch.float32 if kind == "float32" else torch.int32
    pitch = (m + 7) | 1  # odd: the rows take every alignment there is
    xb = torch.zeros((p, pitch), dtype=dt, device=dev)
    xb[:, 1:m + 1] = torch.from_numpy(x).to(dev)
    yb = torch.full((p, pitch), 7, dtype=dt, device=dev)
    xs, ys = [r[1:m + 1] for r in xb], [r[1:m + 1] for r in yb]
    with pkg.Plan(p, m, kind, 1, topology=topology) as plan:
        if mode == 3 and plan.info()["max_depth"] < 3:
            pytest.skip("split layout needs trees of depth >= 3")
        if mode:
            plan.set(pkg.OPT_FUSED_MODE, mode)
        plan.allreduce(xs, ys)
        plan.sync()
        assert plan.info()["vector_path"] == 0
    got = bits(yb).reshape(p, pitch)
    bad = np.nonzero((got[:, 1:m + 1] != want).any(axis=1))[0]
    assert bad.size == 0, "%d ranks differ, first %d" % (bad.size, bad[0])
    assert bool((yb[:, 0] == 7).all()) and bool((yb[:, m + 1:] == 7).all())
