"""imrt_eval_csr_noalloc's objective: written to host, pinned and device memory alike, and no row or tile of
rows left out of it or added twice."""
import ctypes

import numpy as np
import pytest

from paper_0908_4421_gb300 import _lib as L
from paper_0908_4421_gb300 import phantom

pytestmark = pytest.mark.gpu


def _call(torch, case, x, G_address):
    dev = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (case.row_ptr, case.col, case.val, case.mask, x)]
    z = torch.empty(case.m, device="cuda")
    csr = L.imrt_csr(case.m, case.n, case.nnz, dev[0].data_ptr(), dev[1].data_ptr(), dev[2].data_ptr(), 1)
    L.check(L.load().imrt_eval_csr_noalloc(ctypes.byref(csr), dev[3].data_ptr(), case.n_structures,
                                           case.thresholds.ctypes.data, case.weights.ctypes.data, dev[4].data_ptr(),
                                           z.data_ptr(), G_address, torch.cuda.current_stream().cuda_stream))
    return z.cpu().numpy()


def test_objective_into_host_pinned_and_device_memory():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    case = phantom.random_case(3, m=700, n=45, density=0.2, n_structures=2, empty_rows=10)
    x = np.random.Generator(np.random.PCG64(1)).uniform(0.0, 1.0, case.n).astype(np.float32)
    host = ctypes.c_double(-1.0)
    _call(torch, case, x, ctypes.addressof(host))
    assert host.value > 0.0
    pinned = torch.full((3,), -1.0, dtype=torch.float64).pin_memory()
    device = torch.full((3,), -1.0, dtype=torch.float64, device="cuda")
    for G in (pinned, device):
        _call(torch, case, x, G[1:].data_ptr())
        assert G.cpu().tolist() == [-1.0, host.value, -1.0]


@pytest.mark.parametrize("m", [1, 33, 20001, 38913, 524288, 524289, 1050001])  # tiles of 32, 64 and 96 rows
def test_no_row_and_no_tile_is_lost_or_counted_twice(m):
    """Every voxel is under-dosed by about the same, so its share of the objective exceeds the tolerance: F is
    FP64 but for e = T - z, rounded to FP32 (2^-24), and squared; all terms are positive."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    rng = np.random.Generator(np.random.PCG64(m))
    n, j = 9, np.arange(m)
    lengths = 1 + j % 3
    case = type("Case", (), {})()
    case.m, case.n, case.nnz, case.n_structures = m, n, int(lengths.sum()), 2
    case.row_ptr = np.concatenate([[0], np.cumsum(lengths)]).astype(np.int64)
    case.col = (np.arange(case.nnz) - np.repeat(case.row_ptr[:-1], lengths) + np.repeat(j % 7, lengths)).astype(np.int32)
    case.val = rng.uniform(0.01, 1.0, case.nnz).astype(np.float32)
    case.mask = np.where(rng.random(m) < 0.5, 3, 1).astype(np.uint8)
    case.thresholds = np.array([[20.0, np.nan], [30.0, np.nan]], np.float32)
    case.weights = np.array([[2.0, 0.0], [1.0, 0.0]], np.float32)
    x = rng.uniform(0.0, 2.0, n).astype(np.float32)
    G = ctypes.c_double(-1.0)
    z = _call(torch, case, x, ctypes.addressof(G)).astype(np.float64)
    second = (case.mask >> 1) & 1
    F = 2.0 / m * (20.0 - z) ** 2 + second / max(int(second.sum()), 1) * (30.0 - z) ** 2
    G64 = float(F.sum())
    tolerance = (2.0 ** -23 + 1e-9) * G64
    assert F.min() > 2 * tolerance
    assert abs(G.value - G64) <= tolerance
