"""The matrix nest at the sizes where its tiles change (SIMT tiles of 32, 64 and
128, tensor-core tiles of 32 to 224 columns) and on matrices that start anywhere:
rows and bases off the 16-byte grid."""
import numpy as np
import pytest
import torch

import oracle
from guard import guarded
from tolerances import bf16x3_tol
from paper_1412_1127_gb300 import api, inputs

pytestmark = pytest.mark.gpu

U = 2.0 ** -24


def shifted(x, off):
    """x on the GPU, its first element `off` elements past a 256-byte boundary."""
    flat = torch.empty(x.size + off, dtype=torch.float32, device="cuda")
    flat[off:] = torch.from_numpy(x.reshape(-1)).cuda()
    return flat[off:].view(x.shape)


def run(a, b, mode, off=(0, 0)):
    c = guarded(a.shape, torch.float32, float("nan"))
    api.accr_matmul_nest(shifted(a, off[0]), shifted(b, off[1]), c.t, mode=mode, flags=api.ACCR_SYNC)
    return c.check("c (%s, len %d)" % (mode, a.shape[0])).cpu().numpy()


@pytest.mark.parametrize("n", [31, 33, 95, 480, 767, 961, 1000, 1024, 1217, 1441, 1536])
def test_every_tile(n):
    a, b = inputs.uniform_matrix(n, n, salt=n), inputs.uniform_matrix(n, n, salt=n + 1)
    assert np.array_equal(run(a, b, "serial"), oracle.matmul_listing1_threads(a, b))
    t, s = oracle.matmul_truth_threads(a, b)
    assert np.all(np.abs(run(a, b, "simt").astype(np.float64) - t) <= (n + 2) * U * s)
    c = run(a, b, "bf16x3")
    assert np.all(np.abs(c.astype(np.float64) - t) <= bf16x3_tol(a, b, s))


@pytest.mark.parametrize("n", [1, 3, 5, 64, 66, 67, 301])
@pytest.mark.parametrize("off", [(1, 0), (2, 3), (3, 1)])
def test_unaligned_bases(n, off):
    a, b = inputs.small_int_matrix(n, n, salt=n), inputs.small_int_matrix(n, n, salt=n + 5)
    exact = (a.astype(np.int64) @ b.astype(np.int64)).astype(np.float32)
    for mode in ["serial", "simt", "bf16x3"]:
        assert np.array_equal(run(a, b, mode, off), exact), mode


def test_status_word_of_an_earlier_call_is_not_this_calls():
    """Calls on one stream share the split buffers and the status word."""
    for n in (64, 700, 64, 1300, 64):
        a, b = inputs.small_int_matrix(n, n, salt=n), inputs.small_int_matrix(n, n, salt=n + 5)
        assert np.array_equal(run(a, b, "bf16x3"), (a.astype(np.int64) @ b.astype(np.int64)).astype(np.float32))
