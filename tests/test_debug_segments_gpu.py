"""The bounds-checked debug library runs segments of every form, and k-nearest at its
tightened bounds, with no violation."""
import json
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r"""
import json
import numpy as np, torch
from paper_1412_1127_gb300 import api, _native
assert _native.LIB_PATH.endswith("libaccr_debug.so"), _native.LIB_PATH
_, _, checked = api.accr_debug_report(clear=True)
bad = []
g = np.random.default_rng(3)
for seed, tiling in ((0, None), (1, (4096, 8192))):
    if tiling: api.accr_batch_tiling(*tiling)
    L = np.concatenate([g.integers(0, 50, 500), g.integers(500, 20000, 60), [300000, 0, 1200001, 70000]])
    g.shuffle(L)
    off = np.concatenate([[0], np.cumsum(L)]).astype(np.int64) + 3
    v = torch.from_numpy(g.integers(-1000, 1000, int(off[-1]))).cuda()
    s, m = (torch.zeros(len(L), dtype=torch.int64, device="cuda") for _ in range(2))
    c = torch.cat([torch.zeros(1, dtype=torch.int64, device="cuda"), v.cumsum(0)])
    o = torch.from_numpy(off).cuda()
    want = c[o[1:]] - c[o[:-1]]
    for clauses in ([api.clause("add", s)], [api.clause("max", m), api.clause("add", s)]):
        s.zero_()
        api.accr_segmented_reduce(v, off, clauses, flags=api.ACCR_SYNC)
        if not torch.equal(s, want): bad.append(("segments", seed, len(clauses)))
y, x = np.mgrid[0:1024, 0:1024]
pts = torch.from_numpy(np.stack([x.ravel(), y.ravel()], 1).astype(np.float32)).cuda()
for k in (1, 10, 16):
    idx, d2 = torch.empty(k, dtype=torch.int64, device="cuda"), torch.empty(k, device="cuda")
    api.accr_nearest_k(pts, 3.3, 512.2, k, idx, d2, flags=api.ACCR_SYNC)
    want = torch.topk((pts[:, 0] - 3.3) ** 2 + (pts[:, 1] - 512.2) ** 2, k, largest=False).values
    if not torch.allclose(d2, want, rtol=1e-5): bad.append(("nearest", k))
torch.cuda.synchronize()
v, site, _ = api.accr_debug_report(clear=True)
print(json.dumps({"checked": checked, "violations": v, "site": site, "bad": bad}))
"""


@pytest.mark.gpu
def test_segments_and_nearest_without_violations():
    from paper_1412_1127_gb300 import build
    build.build(debug=True)
    env = dict(os.environ, ACCR_LIBRARY=build.DEBUG_LIB, PYTHONPATH=ROOT)
    r = subprocess.run([sys.executable, "-c", CHILD], cwd=ROOT, env=env, capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stderr[-4000:]
    out = json.loads(r.stdout.strip().splitlines()[-1])
    assert out["checked"] is True and out["bad"] == [], out
    assert out["violations"] == 0, "first failing site %d" % out["site"]
