"""Inputs of 4 GiB and more, which the streaming and split layouts load by
another instruction: every element against a sum that torch forms on the GPU
(int32 wraps, so any order gives the same bits), in place and out of place,
with a ragged tail, just below and above the limit."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    from paper_2109_12626_gb300 import build as B
    B.build()
    import paper_2109_12626_gb300 as P
    return P


LIMIT = (4 << 30) // 4


@pytest.mark.parametrize("p,mode", [(2, 1), (7, 1), (32, 1), (100, 1), (32, 3), (288, 3), (512, 3), (1152, 3)])
@pytest.mark.parametrize("over", [False, True], ids=["below", "above"])
@pytest.mark.parametrize("in_place", [False, True], ids=["separate", "in_place"])
def test_far_inputs_sum(pkg, p, mode, over, in_place):
    if mode == 3 and p == 32 and not over:
        pytest.skip("the split layout at p = 32: above the limit only")
    dev = torch.device("cuda:0")
    m = -(-LIMIT // p) + 1 if over else LIMIT // p - 1
    pitch = (m + 7) // 4 * 4  # rows 16-byte aligned
    g = torch.Generator(device=dev).manual_seed(p)
    x = torch.randint(-2**31, 2**31 - 1, (p, pitch), dtype=torch.int32, device=dev, generator=g)
    want = x[:, :m].sum(0, dtype=torch.int32)
    y = x if in_place else torch.full_like(x, 7)
    guard = y[:, m:].clone()
    with pkg.Plan(p, m, "int32", 1) as plan:
        plan.set(pkg.OPT_FUSED_MODE, mode)
        plan.allreduce([r[:m] for r in x], [r[:m] for r in y])
        plan.sync()
        assert plan.info()["vector_path"] == 1
    for i in range(p):
        assert torch.equal(y[i, :m], want), "rank %d" % i
    assert torch.equal(y[:, m:], guard)
