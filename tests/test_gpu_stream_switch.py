"""A plan whose stream changes between calls: what plan_info prepared on the first (the forward schedule and, for
beamlet-major copies beyond 64 MiB, the L2 prefetch targets) is complete before a solve on the second reads it."""
import numpy as np
import pytest

from paper_0908_4421_gb300 import Options, Plan
from paper_0908_4421_gb300 import _lib as L

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [L.FP32, L.FP16])
def test_solve_on_another_stream_than_info(precision):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    m, n, per = 180000, 1000, 100  # 18M entries: 72 MB in FP16, 108 MB in FP32
    col = (torch.arange(per, device="cuda") * 10 + torch.arange(m, device="cuda")[:, None] % 10).to(torch.int32).reshape(-1)
    val = torch.rand(m * per, device="cuda", generator=torch.Generator(device="cuda").manual_seed(3)) + 0.01
    row_ptr = torch.arange(m + 1, device="cuda") * per
    mask = (torch.arange(m, device="cuda") % 3 + 1).to(torch.uint8)
    thr, w = np.array([[3.0, 5.0], [np.nan, 1.0]], np.float32), np.array([[2.0, 3.0], [0.0, 1.0]], np.float32)
    torch.cuda.synchronize()
    options = Options(precision=precision, k_trials=2, max_iter=6, delta=0.0, polish_iter=2)
    with Plan(row_ptr, col, val, mask, thr, w, m=m, n=n, options=options) as plan:
        expected = (plan.solve().objective, plan.get_x())
    first, second = torch.cuda.Stream(), torch.cuda.Stream()
    with Plan(row_ptr, col, val, mask, thr, w, m=m, n=n, options=options) as plan:
        plan.set_options(stream=first.cuda_stream)
        plan.info()
        plan.set_options(stream=second.cuda_stream)
        assert plan.solve().objective == expected[0]
        assert np.array_equal(plan.get_x(), expected[1])
