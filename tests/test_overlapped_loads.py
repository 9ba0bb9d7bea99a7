"""Kernels launched while their predecessor may still run read their inputs by
ordinary loads: PTX defines the read-only path (ld.global.nc, __ldg, const
__restrict__ parameters) only for memory that nothing writes while the kernel lives.
The sources are looked through (no GPU)."""
import glob
import os
import re

from paper_1412_1127_gb300 import build

READ_ONLY = re.compile(r"__ldg\s*\(|__restrict__|\.global(\.\w+)*\.nc\b")


# kernels of ordinary launches, which start after everything before them
ORDINARY = {"standardize_kernel", "map_kernel", "bfs_init_kernel", "bfs_tile_kernel"}


def around(lines, i):
    """The name of the function line i stands in: the last one called or declared on
    the nearest line above that starts at the margin."""
    while not re.match(r"[A-Za-z_]", lines[i]) or "(" not in lines[i]:
        i -= 1
    return re.findall(r"(\w+)\(", lines[i])[-1]


def test_no_read_only_loads_in_overlapped_kernels():
    bad, kept = [], set()
    for f in glob.glob(os.path.join(build.CSRC, "*.cu*")):
        lines = re.sub(r"//[^\n]*", "", open(f).read()).split("\n")
        for i, line in enumerate(lines):
            if READ_ONLY.search(line):
                fn = around(lines, i)
                (kept.add(fn) if fn in ORDINARY else bad.append((os.path.basename(f), fn, line.strip())))
    assert not bad, bad
    for fn in kept:  # and they are launched so
        for f in glob.glob(os.path.join(build.CSRC, "*.cu")):
            assert not re.search(r"launch_overlapped\(\s*%s\b" % fn, open(f).read()), fn


def test_streaming_loads_stay_behind_the_wait():
    """Inline loads are volatile and clobber memory, as the wait does."""
    for f in glob.glob(os.path.join(build.CSRC, "*.cu*")):
        for m in re.finditer(r"asm( volatile)?\(\s*\"ld\.global[^;]*;\"(.*?)\);", open(f).read(), re.S):
            assert m.group(1) and '"memory"' in m.group(2), (os.path.basename(f), m.group(0)[:80])


def test_tensor_memory_is_taken_behind_the_wait():
    """Its allocation waits without a limit: no CTA holds any while it waits for a
    predecessor that may want some."""
    text = re.sub(r"//[^\n]*", "", open(os.path.join(build.CSRC, "matmul_tc.cu")).read())
    body = text[text.index("bf16x3_gemm_kernel("):text.index("split_kernel(")]
    assert 0 < body.index("grid_wait()") < body.index("tcgen05.alloc")
