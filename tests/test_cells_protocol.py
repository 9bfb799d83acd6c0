"""The slots of flagged words between the schedule kernel's subtree cells: a
sender waits for no slot, so every slot must have been read, by all that read
it, before it is written again, however long any warp is held back
(cells_protocol.cu replays the exchanges over the library's own cells, slices
and slot counts)."""
import ctypes

import numpy as np
import pytest

import cells_util


@pytest.fixture(scope="module")
def replay(tmp_path_factory):
    lib = cells_util.load(str(tmp_path_factory.mktemp("cells")))

    def run(p, m, esize, single, b, aligned, warps=2432, down_slots=0, empty=False, bad=0):
        out = (ctypes.c_int * 8)()
        rc = lib.words_protocol(p, ctypes.c_int64(m), esize, int(single), b, int(aligned), warps,
                                down_slots, int(empty), out)
        assert rc == bad, "p=%d m=%d b=%d: %s, channel %s, cell %d at depth %d, step %d" % (
            p, m, b,
            ("sound", "slot written unread", "waits for ever", "too many steps", "no room")[rc],
            ("up", "down", "dual")[out[3]], out[4], out[5], out[6])
        return {"steps": out[0], "cells": out[1], "depth": out[2]}
    return run


# blocks of one length (whole slices), 8 to 20 steps: shallow and deep trees
@pytest.mark.parametrize("single", [False, True], ids=["dual", "single"])
@pytest.mark.parametrize("p", [1, 2, 3, 7, 16, 36, 100, 255, 288, 1025, 1152, 2049, 2300, 4000])
def test_slots_are_read_before_they_are_written(replay, p, single):
    for steps in (1, 2, 8, 9, 12, 20):
        got = replay(p, steps * 64, 4, single, steps, True)
        assert got["steps"] >= min(steps, 8) // 2


# blocks that differ by a unit, so that the last slice of some holds none
# (m = 2064, b = 16: 33 units, then 32 in each), aligned rows, element by
# element on others, 2x2 matrices; and a slice that no block fills
@pytest.mark.parametrize("single", [False, True], ids=["dual", "single"])
@pytest.mark.parametrize("p", [2, 3, 36, 288, 1152])
def test_empty_slices(replay, p, single):
    for m, b in ((2064, 16), (2048, 16), (129 * 20 + 3, 20), (2560, 20), (33 * 20 - 7, 20), (65 * 31 - 30, 31)):
        for aligned in (True, False):
            replay(p, m, 4, single, b, aligned)
        replay(p, m // 4, 16, single, b, True)


def test_random_partitions(replay):
    rng = np.random.default_rng(11)
    for _ in range(300):
        p = int(np.exp(rng.uniform(np.log(2), np.log(600))))
        m = int(np.exp(rng.uniform(0, np.log(20000))))
        replay(p, m, int(rng.choice([4, 16])), rng.random() < 0.5, int(rng.integers(1, min(m, 60) + 1)),
               rng.random() < 0.6, int(rng.choice([4 * 4 * 152, 3 * 4 * 152, 4 * 152])))


def test_replay_sees_slots_written_too_soon(replay):
    """The replay itself: eight slots for final blocks are too few below a
    deep tree's root, and rounds without units (the cells hear nothing from
    each other) leave two slots too few between the dual roots."""
    for p, single in ((1025, True), (1152, True), (2049, True), (2049, False)):
        replay(p, 1280, 4, single, 20, True, down_slots=8, bad=1)
        replay(p, 512, 4, single, 8, True, down_slots=8)
    for p in (2, 32, 36, 288):
        replay(p, 2064, 4, False, 16, True, empty=True, bad=1)


def test_more_cells_than_fit(replay):
    """Two warps per cell are the least (a slice and the tail): with more
    cells than that the cut is given up before any cell is laid out."""
    for p, cells in ((20000, 2866), (9000, 1294)):
        assert replay(p, 1000, 4, False, 1, True, bad=4)["cells"] == cells
    assert replay(8000, 1000, 4, False, 1, True)["cells"] <= 1216
