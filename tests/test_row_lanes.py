"""Rows past 2 KiB: every lane of the warp that folds one has a vector of it, whatever
the row's alignment, so that its loads need no condition (no GPU: the arithmetic of the
row group's launch and fold, restated)."""
import os
import re

import pytest

from paper_1412_1127_gb300 import build


def constant(name, text):
    return re.search(r"%s = ([^;]+);" % name, text).group(1)


@pytest.mark.parametrize("size", [4, 8])
def test_every_lane_has_a_vector(size):
    text = open(os.path.join(build.CSRC, "group.cuh")).read()
    assert constant("GROUP_GV", text) == "8" and constant("GROUP_BYTES", text) == "GROUP_GV * 32 * 16"
    group_bytes = 8 * 32 * 16
    launch = open(os.path.join(build.CSRC, "rowgroup.cu")).read()
    assert "a.cols * (int64_t)sizeof(T) <= GROUP_BYTES / 2) go<T, NC, W0, W1, GROUP_GV / 2>" in launch
    epv = 16 // size
    for cols in range(group_bytes // 2 // size + 1, group_bytes // size + 1):
        lanes = 1
        while lanes < 32 and lanes * 4 * 16 < cols * size:  # accr_rowreduce's choice
            lanes *= 2
        assert lanes == 32
        for head in range(epv):
            nvec = (cols - head) // epv
            assert nvec > lanes - 1
            # the last index a lane forms, and the one it falls back to
            rounds = -(-(cols // epv) // lanes)
            assert rounds <= 8
