"""The schedule kernels on subtree cells, which run while every schedule
option is automatic: bit for bit against the oracle's fold, for both
transports between cells (flagged words for small inputs, counters beyond),
both entry points and both topologies.

Sizes are the edges of the cell layout: one cell, cells of one rank, the
first cut edges (p = 15, 16, 36), ragged last levels; slices of one unit, of
32, partly filled, several to a warp, of two blocks in a step; blocks that
start and end inside a
16-byte unit or lie within one, rows with a ragged tail."""
import ctypes

import numpy as np
import pytest
import torch

import cells_util
from gpu_util import bits, empty_like_ranks, expect_bits, host_inputs, to_device

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    from paper_2109_12626_gb300 import build as B
    B.build()
    import paper_2109_12626_gb300 as P
    return P


def _dt(orc, kind):
    return {"int32": orc.I32, "float32": orc.F32, "mat2x2u32": orc.MAT,
            "mat2x2f32": orc.MATF}[kind]


def _buffers(x, kind, layout, dev):
    pad = 1 if layout == "four_byte" else 0
    xs, keep = to_device(x, kind, dev, pad_front=pad)
    if layout == "in_place":
        return xs, xs, keep
    ys, keep_y = empty_like_ranks(xs, pad_front=pad)
    return xs, ys, (keep, keep_y)


def _check(ys, want, what):
    for i, y in enumerate(ys):
        bad = np.nonzero(bits(y) != want)[0]
        assert bad.size == 0, "%s rank %d: %d words differ, first %d" % (what, i, bad.size, bad[0])


# flagged words between cells: at most 12 MiB of inputs (24 from p = 1024)
CASES = [("int32", 1, 33, (1, 4)), ("float32", 2, 1, (1,)), ("float32", 2, 4100, (1, 3)),
         ("int32", 3, 129, (1, 129)), ("mat2x2u32", 7, 300, (1, 7)), ("int32", 15, 1000, (1, 4, 250)),
         ("float32", 16, 4099, (1, 9, 2000)), ("mat2x2f32", 31, 129, (1, 5)),
         ("int32", 36, 1003, (1, 3, 400)), ("mat2x2u32", 100, 77, (1, 7)),
         ("float32", 255, 2050, (1, 16)), ("int32", 288, 250, (1, 2)),
         ("float32", 1152, 4099, (1, 6)), ("int32", 1152, 1, (1,))]
# the same, more steps than final blocks can wait unread below a deep tree's root
CASES += [("int32", 1025, 2048, (32,)), ("int32", 1152, 2560, (20, 40)), ("float32", 2049, 2051, (32,))]
# the same, blocks whose last slice holds units in some and none in others
CASES += [("int32", 2, 2064, (16,)), ("float32", 36, 2064, (16,)), ("int32", 288, 2064, (16,)),
          ("int32", 36, 653, (20,)), ("mat2x2u32", 7, 653, (20,))]
# counters between cells
CASES += [("int32", 2, 1600001, (1, 5)), ("float32", 7, 500003, (1, 8, 600)),
          ("mat2x2u32", 36, 30001, (1, 7)), ("int32", 100, 40009, (1, 16, 5000)),
          ("float32", 288, 21250, (0, 1, 3)), ("mat2x2f32", 288, 3001, (4,)),
          ("int32", 1152, 8193, (0, 1, 5, 1000)), ("float32", 2600, 2051, (0, 3)), ("float32", 2600, 37, (1, 3))]


@pytest.mark.parametrize("kind,p,m,blocks", CASES)
@pytest.mark.parametrize("layout", ["aligned", "in_place", "four_byte"])
@pytest.mark.parametrize("run", ["dual", "single", "reduce_bcast"])
def test_cells_match_oracle(pkg, orc, kind, p, m, blocks, layout, run):
    x = host_inputs(kind, 101, p, m)
    topo = "dual" if run == "dual" else "single"
    want = expect_bits(orc.tree_fold(x, _dt(orc, kind), orc.DUAL if topo == "dual" else orc.SINGLE))
    dev = torch.device("cuda:0")
    for b in blocks:
        xs, ys, _keep = _buffers(x, kind, layout, dev)
        with pkg.Plan(p, m, kind, b, topology=topo) as plan:
            assert plan.info()["sched_cells"] > 0
            call = plan.allreduce_reduce_bcast if run == "reduce_bcast" else plan.allreduce_schedule
            for again in range(1 if layout == "in_place" else 2):
                call(xs, ys)
                plan.sync()
                _check(ys, want, "b=%d call %d" % (b, again))
        if layout != "in_place":
            for i in range(p):  # inputs untouched
                assert np.array_equal(bits(xs[i]), expect_bits(x[i])), i


def test_cells_choice(pkg):
    """On cells while every schedule option is automatic and one slice of
    them fits the GPU; any option set takes the layouts it names."""
    for key, value in ((pkg.OPT_SCHED_TRANSPORT, 1), (pkg.OPT_SCHED_TRANSPORT, 2),
                       (pkg.OPT_SCHED_LAYOUT, 1), (pkg.OPT_SCHED_COPY, 2),
                       (pkg.OPT_SCHED_SLICES, 2), (pkg.OPT_SCHED_RANKS_PER_CTA, 2),
                       (pkg.OPT_SCHED_THREADS, 64)):
        with pkg.Plan(36, 1000, "int32", 3) as plan:
            assert plan.info()["sched_cells"] > 0
            plan.set(key, value)
            assert plan.info()["sched_cells"] == 0
            plan.set(key, 0)
            assert plan.info()["sched_cells"] > 0
    with pkg.Plan(65535, 3, "int32", 1) as plan:
        assert plan.info()["sched_cells"] == 0


def test_cells_take_the_place_of_other_scratch(pkg, orc):
    """A plan on cells holds nothing of the kernels that they replace: the
    dual roots' exchange slots (four of a block each) come with the option
    that asks for those."""
    kind, p, m = "mat2x2u32", 36, 65536
    x = host_inputs(kind, 104, p, m)
    want = expect_bits(orc.tree_fold(x, orc.MAT, orc.DUAL))
    xs, _ = to_device(x, kind, torch.device("cuda:0"))
    with pkg.Plan(p, m, kind, 1) as plan:
        held = []
        for transport in (0, 1, 0, 1):
            plan.set(pkg.OPT_SCHED_TRANSPORT, transport)
            held.append(plan.info()["scratch_bytes"])
            ys, _k = empty_like_ranks(xs)
            plan.allreduce_schedule(xs, ys)
            plan.sync()
            _check(ys, want, "transport %d" % transport)
        assert held[1] - held[0] >= 4 * 16 * m and held[1] == held[2] == held[3]


@pytest.mark.parametrize("key,value", [("OPT_SCHED_TRANSPORT", 1), ("OPT_SCHED_TRANSPORT", 2),
                                       ("OPT_SCHED_LAYOUT", 1), ("OPT_SCHED_THREADS", 64),
                                       ("OPT_SCHED_COPY", 2), ("OPT_SCHED_RANKS_PER_CTA", 1)])
def test_option_that_memory_cannot_hold(pkg, key, value):
    """Four exchange slots of a 137 GB block, or word arrays, are more than
    the GPU has: the option is refused and the plan stays on cells."""
    with pkg.Plan(2, 1 << 35, "int32", 1) as plan:
        before = plan.info()
        assert before["sched_cells"] > 0
        with pytest.raises(pkg.DpdrError) as e:
            plan.set(getattr(pkg, key), value)
        assert e.value.status == pkg.DPDR_ERR_OOM
        assert plan.info() == before


def test_word_slots_of_short_calls(pkg):
    """One step needs one slot per cell and slice: 46 cells, of which fewer
    have children, on 8 slices (element by element) and the tail, 1 KB each,
    4 for the roots, and the plan's tables."""
    with pkg.Plan(288, 250, "int32", 1) as plan:
        assert plan.info()["sched_transport"] == 2 and plan.info()["sched_cells"] == 46
        assert plan.info()["scratch_bytes"] < 9 * (2 * 46 + 4) * 1024 + (1 << 17)


def test_cells_change_of_options_and_alignment(pkg, orc):
    """One plan, calls of different kinds in a row: aligned and unaligned
    buffers (other slice counts over the same counters), other block counts,
    both entry points, options set and taken back."""
    kind, p, m = "float32", 100, 40009
    x = host_inputs(kind, 102, p, m)
    want = expect_bits(orc.tree_fold(x, orc.F32, orc.SINGLE))
    dev = torch.device("cuda:0")
    xa, _ = to_device(x, kind, dev)
    xu, _keep = to_device(x, kind, dev, pad_front=1)
    with pkg.Plan(p, m, kind, 4, topology="single") as plan:
        for step in range(12):
            if step == 4:
                plan.set(pkg.OPT_BLOCKS, 37)
            if step in (6, 9):
                plan.set(pkg.OPT_SCHED_TRANSPORT, 1 if step == 6 else 0)
            xs = xu if step % 2 else xa
            ys, _k = empty_like_ranks(xs, pad_front=step % 2)
            call = plan.allreduce_reduce_bcast if step % 3 == 2 else plan.allreduce_schedule
            call(xs, ys)
            plan.sync()
            _check(ys, want, "step %d" % step)


RESTART = 1 << 29  # counters and flags start from 0 again (schedule_cells.cuh, kRestart)


@pytest.fixture(scope="module")
def base_of(tmp_path_factory):
    L = cells_util.load(str(tmp_path_factory.mktemp("cells")))
    L.cells_base.restype = ctypes.c_longlong

    def base(plan, walk, value=-1):
        got = L.cells_base(ctypes.c_void_p(plan._h), int(walk), ctypes.c_longlong(value))
        assert got >= 0
        return got
    return base


@pytest.mark.parametrize("run,p,m,b", [("dual", 36, 1003, 3), ("dual", 1152, 515, 4),
                                       ("dual", 100, 40009, 5), ("single", 255, 20003, 9),
                                       ("reduce_bcast", 100, 40009, 5)])
@pytest.mark.parametrize("before", [1, 40], ids=["at_once", "later"])
def test_cells_restart_of_the_numbers(pkg, orc, base_of, run, p, m, b, before):
    """Calls across the point where counters and flags start from 0 again.
    Calls on unaligned buffers, which use other slots than those on aligned
    ones, leave small numbers behind first: were they not cleared, the same
    numbers would mean another call's values afterwards."""
    kind, dev = "int32", torch.device("cuda:0")
    topo = "dual" if run == "dual" else "single"
    with pkg.Plan(p, m, kind, b, topology=topo) as plan:
        info = plan.info()
        assert info["sched_cells"] > 0
        walk = run == "reduce_bcast" or info["sched_transport"] == 1

        def calls(count, pad, seed):
            v = host_inputs(kind, seed, p, m, lo=-1000, hi=1000)
            want = expect_bits(orc.tree_fold(v, orc.I32, orc.DUAL if topo == "dual" else orc.SINGLE))
            xs, _k = to_device(v, kind, dev, pad_front=pad)
            for k in range(count):
                ys, _y = empty_like_ranks(xs, pad_front=pad)
                (plan.allreduce_reduce_bcast if run == "reduce_bcast" else plan.allreduce_schedule)(xs, ys)
                plan.sync()
                _check(ys, want, "seed %d call %d" % (seed, k))

        calls(2, 1, 1)
        calls(1, 0, 2)
        assert 0 < base_of(plan, walk) < 10000
        base_of(plan, walk, RESTART - before)
        calls(4 + before // 2, 0, 3)
        assert base_of(plan, walk) < 10000
        calls(3, 1, 4)
        calls(2, 0, 5)


@pytest.mark.parametrize("p,m", [(30, 777), (100, 40009)], ids=["words", "counters"])
@pytest.mark.parametrize("run", ["schedule", "reduce_bcast"])
def test_cells_graph_replay(pkg, orc, p, m, run):
    """Epochs and counter bases move on the device: a captured call replays
    with new inputs, and plain calls go on between replays."""
    kind, dev = "int32", torch.device("cuda:0")
    xs = [torch.empty(m, dtype=torch.int32, device=dev) for _ in range(p)]
    ys = [torch.empty(m, dtype=torch.int32, device=dev) for _ in range(p)]
    with pkg.Plan(p, m, kind, 3, topology="single") as plan:
        bound = plan.bind(xs, ys)
        call = bound.allreduce_schedule if run == "schedule" else bound.allreduce_reduce_bcast
        s = torch.cuda.Stream()
        s.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(s):
            call()
        torch.cuda.current_stream().wait_stream(s)
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            call()
        for seed in (1, 2, 3, 4):
            x = host_inputs(kind, 110 + seed, p, m, lo=-1000, hi=1000)
            for i in range(p):
                xs[i].copy_(torch.from_numpy(x[i]))
                ys[i].fill_(-7)
            if seed == 3:
                call()
            else:
                g.replay()
            torch.cuda.synchronize()
            _check(ys, expect_bits(orc.tree_fold(x, orc.I32, orc.SINGLE)), "seed %d" % seed)
        plan.sync()


@pytest.mark.parametrize("p,m,b", [(7, 1000, 4), (36, 1000, 1), (1152, 500, 4), (100, 40009, 5)])
@pytest.mark.parametrize("run", ["dual", "reduce_bcast"])
def test_cells_silent_rank_times_out_and_recovers(pkg, orc, p, m, b, run):
    """A rank that never publishes -- a leaf, an inner rank of a cell, a
    cell's root, a tree's root -- makes its partners' waits expire; the plan
    works again afterwards."""
    from paper_2109_12626_gb300 import DpdrError
    kind = "int32"
    topo = "dual" if run == "dual" else "single"
    x = host_inputs(kind, 103, p, m, lo=-1000, hi=1000)
    want = expect_bits(orc.tree_fold(x, orc.I32, orc.DUAL if run == "dual" else orc.SINGLE))
    xs, _ = to_device(x, kind, torch.device("cuda:0"))
    with pkg.Plan(p, m, kind, b, topology=topo) as plan:
        assert plan.info()["sched_cells"] > 0
        call = plan.allreduce_reduce_bcast if run == "reduce_bcast" else plan.allreduce_schedule
        plan.set(pkg.OPT_WAIT_LIMIT_NS, 20_000_000)
        c0 = plan.query()["child0"]
        ranks = {0, 1, 2, p // 2, p - 2, p - 1} | {int(np.nonzero(c0 >= 0)[0][k]) for k in (0, -2)}
        if plan.info()["sched_cells"] == 1:
            ranks.discard(p - 1)  # one cell: nobody waits for its root
        for skip in sorted(ranks):
            plan.set(pkg.OPT_SKIP_RANK, skip)
            ys, _ = empty_like_ranks(xs)
            call(xs, ys)
            with pytest.raises(DpdrError) as e:
                plan.sync()
            assert e.value.status == pkg.DPDR_ERR_TIMEOUT, skip
            plan.set(pkg.OPT_SKIP_RANK, -1)
            call(xs, ys)
            plan.sync()
            _check(ys, want, "after %d" % skip)
