"""The first call on a stream, with the default stream busy: what the library
allocates for the stream is zeroed before the call's kernel reads it, and the call
does not wait for the default stream.  A process of its own, so that every stream's
first call is its first."""
import json
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r"""
import ctypes, json
import numpy as np, torch
from paper_1412_1127_gb300 import api
dev = "cuda"
g = torch.Generator().manual_seed(7)
sink = torch.empty(256 * 152, device=dev)
ints = torch.randint(-1000, 1000, (1 << 20,), generator=g, dtype=torch.int32).to(dev)
flt = torch.randn(1 << 20, generator=g).to(dev)
pts = torch.rand(1 << 19, 2, generator=g).to(dev)
off = np.arange(0, (1 << 20) + 1, 64, dtype=np.int64)
grid = (torch.rand(300, 2000, generator=g) < 0.8).to(torch.uint8).to(dev)
lens = [1000] * 3000
mk = lambda n, d: torch.zeros(n, dtype=d, device=dev)

def region(o): api.accr_reduce(ints, [api.clause("add", o[0])])
def rows(o): api.accr_rowreduce(ints.view(4, -1), [api.clause("add", o[0])])
def segments(o): api.accr_segmented_reduce(ints, off, [api.clause("add", o[0])])
def nearest(o): api.accr_nearest_k(pts, 0.4, 0.6, 10, o[0], o[1])
def standardize(o): api.accr_standardize(flt, o[0], o[1])
def bfs(o): api.accr_grid_bfs(grid, 150 * 2000 + 1000, o[0].view(300, 2000), mode="persistent")
def described(o):                               # descriptors are made ahead of the call: they take Python a while
    return api.regions_array([(ints[1000 * (i % 1000):][:n], [api.clause("add", o[0][i:i + 1])], 0) for i, n in enumerate(lens)])
def batch(o): api.check(api.lib().accr_batch_reduce(o[-1][0], len(lens), 0, torch.cuda.current_stream().cuda_stream))
def prepared(o):
    h = ctypes.c_void_p()
    api.check(api.lib().accr_batch_create(o[-1][0], len(lens), 0, ctypes.byref(h)))
    api.check(api.lib().accr_batch_launch(h, torch.cuda.current_stream().cuda_stream))
def batch_outs():
    o = [mk(3000, torch.int64)]
    return o + [described(o)]
CALLS = {
    "region": (region, lambda: [mk(1, torch.int64)]), "rows": (rows, lambda: [mk(4, torch.int64)]),
    "segments": (segments, lambda: [mk(len(off) - 1, torch.int64)]),
    "nearest": (nearest, lambda: [mk(10, torch.int64), mk(10, torch.float32)]),
    "standardize": (standardize, lambda: [mk(1 << 20, torch.float32), mk(2, torch.float64)]),
    "bfs": (bfs, lambda: [mk(600000, torch.int32)]), "batch": (batch, batch_outs),
    "prepared": (prepared, batch_outs),
}
ref = {}
for name, (f, outs) in CALLS.items():          # on the default stream, idle
    ref[name] = outs()
    f(ref[name])
    torch.cuda.synchronize()
bad, waited = [], []
for name, (f, outs) in CALLS.items():
    o, s = outs(), torch.cuda.Stream()          # streams of torch's pool, each for the first time
    torch.cuda.synchronize()
    api.accr_probe_fma(76, 3000000, sink)       # half of the SMs, tens of milliseconds
    end = torch.cuda.Event(); end.record()
    with torch.cuda.stream(s):
        f(o)
        s.synchronize()
    if end.query(): waited.append(name)
    torch.cuda.synchronize()
    if not all(torch.equal(a, b) for a, b in zip(o, ref[name]) if torch.is_tensor(a)): bad.append(name)
print(json.dumps({"bad": bad, "waited": waited}))
"""


@pytest.mark.gpu
def test_first_calls_beside_a_busy_default_stream():
    r = subprocess.run([sys.executable, "-c", CHILD], cwd=ROOT, env=dict(os.environ, PYTHONPATH=ROOT),
                       capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-3000:]
    out = json.loads(r.stdout.strip().splitlines()[-1])
    assert out["bad"] == []
    # cooperative launches may need the SMs the other stream holds; nothing else waits
    assert set(out["waited"]) <= {"standardize", "bfs"}, out
