"""imrt_eval_csr_noalloc's objective: written to host, pinned and device memory alike."""
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
