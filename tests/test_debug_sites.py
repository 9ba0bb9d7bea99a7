"""Debug builds check every global store of the segment kernel and of the k-nearest scan
(no GPU: the sources are looked through), as accr_debug_report says."""
import os
import re

from paper_1412_1127_gb300 import build


def source(name):
    return re.sub(r"//[^\n]*", "", open(os.path.join(build.CSRC, name)).read())


def test_segment_stores_are_checked():
    text = source("segments.cuh")
    kernel = text[text.index("__global__"):]
    store = kernel[kernel.index("auto store ="):kernel.index("};", kernel.index("auto store ="))]
    assert store.index("ACCR_DCHECK(s >= 0 && s < p.nseg") < store.index("store_var(")
    assert kernel.count("store_var(") == store.count("store_var(")
    tile = text[text.index("segment_tile("):text.index("__global__")]
    check = tile.index("ACCR_DCHECK(i < p.ntiled")
    assert all(m.start() > check for m in re.finditer(r"store_var\(|p\.tiles_done\[", tile))
    for line in tile.split("\n"):
        if re.search(r"p\.partials\[[^]]*\]\s*=", line):
            assert "ACCR_DCHECK(" in line, line


def test_nearest_scan_stores_are_checked():
    text = source("patterns.cu")
    kernel = text[text.index("nearest_kernel(const"):text.index("nearest_launch(const")]
    stores = [l for l in kernel.split("\n") if re.search(r"p\.(tmin|wmin)\[[^]]*\]\s*=", l)]
    assert len(stores) == 2 and all("ACCR_DCHECK(gt < p.threads" in l for l in stores), stores
