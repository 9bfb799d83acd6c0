"""The slots of flagged words between the schedule kernel's subtree cells: a
sender waits for no slot, so every slot must have been read, by all that read
it, before it is written again, however long any warp is held back
(cells_protocol.cu replays the exchanges over the library's own cells, slices
and slot counts)."""
import ctypes

import pytest

import cells_util


@pytest.fixture(scope="module")
def replay(tmp_path_factory):
    lib = cells_util.load(str(tmp_path_factory.mktemp("cells")))

    def run(p, m, esize, single, b, aligned, warps=2432):
        out = (ctypes.c_int * 8)()
        rc = lib.words_protocol(p, ctypes.c_int64(m), esize, int(single), b, int(aligned), warps, out)
        assert rc == 0, "p=%d m=%d b=%d: %s, channel %s, cell %d at depth %d, step %d" % (
            p, m, b, ("", "slot written unread", "waits for ever")[rc],
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
