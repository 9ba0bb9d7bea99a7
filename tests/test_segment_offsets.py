"""accr_segmented_reduce's host check of its offsets finds a decrease whatever the
offsets hold (no GPU: the check's own source is compiled by itself)."""
import ctypes
import os
import re
import subprocess

import numpy as np
import pytest

from paper_1412_1127_gb300 import build

I64 = np.iinfo(np.int64)


@pytest.fixture(scope="module")
def check(tmp_path_factory):
    src = open(os.path.join(build.CSRC, "segments.cu")).read()
    struct = re.search(r"struct LongSegments \{.*?\n\};", src, re.S).group(0)
    body = re.search(r"template <typename O>\nstatic int64_t copy_offsets.*?\n\}\n", src, re.S).group(0)
    d = tmp_path_factory.mktemp("offsets")
    cpp, lib = os.path.join(d, "check.cpp"), os.path.join(d, "check.so")
    with open(cpp, "w") as f:
        f.write("#include <stdint.h>\n#include <algorithm>\n#include <vector>\n" + struct + "\n" + body +
                'extern "C" int64_t run(const int64_t *off, int64_t nseg, void *dst, int wide, int64_t *longer) {\n'
                "    LongSegments L;\n"
                "    const int64_t bad = wide ? copy_offsets(off, nseg, (int64_t *)dst, 1024, 16384, L)\n"
                "                             : copy_offsets(off, nseg, (uint32_t *)dst, 1024, 16384, L);\n"
                "    *longer = 0;\n    for (auto &v : L.mid) *longer += (int64_t)v.size();\n"
                "    for (auto &v : L.tiled) *longer += (int64_t)v.size();\n"
                "    return bad;\n}\n")
    subprocess.run(["g++", "-O2", "-std=c++17", "-fwrapv", "-shared", "-fPIC", cpp, "-o", lib], check=True)
    L = ctypes.CDLL(lib)
    L.run.restype = ctypes.c_int64
    L.run.argtypes = [ctypes.c_void_p, ctypes.c_int64, ctypes.c_void_p, ctypes.c_int, ctypes.c_void_p]

    def f(off, wide):
        off = np.ascontiguousarray(off, dtype=np.int64)
        dst = np.zeros(off.size, dtype=np.int64 if wide else np.uint32)
        longer = ctypes.c_int64()
        return L.run(off.ctypes.data, off.size - 1, dst.ctypes.data, int(wide), ctypes.byref(longer)), dst, longer.value
    return f


@pytest.mark.parametrize("wide", [False, True])
@pytest.mark.parametrize("at", [0, 1, 510, 511, 512, 1500])
@pytest.mark.parametrize("value", [I64.min, I64.min + 1, -1, -(1 << 62)])
def test_an_overflowing_decrease_is_found(check, wide, at, value):
    off = np.arange(1502, dtype=np.int64) * 7 + 5
    off[at + 1] = value
    assert check(off, wide)[0] == at


def test_the_last_offset_alone(check):
    assert check([1, I64.min], True)[0] == 0
    assert check([5, 9, 9, I64.min], True)[0] == 2
    assert check([5, 9, 8, I64.max], True)[0] == 1


@pytest.mark.parametrize("wide", [False, True])
def test_offsets_come_out_relative_to_the_first(check, wide):
    off = np.cumsum(np.concatenate([[3], np.arange(2000) % 1300]))
    bad, dst, longer = check(off, wide)
    assert bad == -1 and np.array_equal(dst.astype(np.int64), off - 3)
    assert longer == int((np.diff(off) > 1024).sum())


@pytest.mark.parametrize("far", [1 << 52, (1 << 52) + 1, 1 << 62, I64.max - 4000])
def test_offsets_beyond_any_array(check, far):
    """Large offsets that do not decrease pass; a decrease behind them is found."""
    off = np.arange(1502, dtype=np.int64) + 5
    off[700:] += far - 2000
    assert check(off, True)[0] == -1
    for at in (3, 698, 699, 1400):
        bad = off.copy()
        bad[at + 1] = bad[at] - 1
        assert check(bad, True)[0] == at
