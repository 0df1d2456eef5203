"""A team solve does not depend on what the device pool's memory held before: where voxel 0 lies outside
every beam, the team solver never writes its r in a trial pass, and nothing may read it. The pool is filled with
NaN by evaluations of plans at NaN fluence, whose per-voxel vectors are as large as a small plan's nine r buffers."""
import numpy as np
import pytest

from paper_0908_4421_gb300 import Options, Plan, phantom
from paper_0908_4421_gb300 import _lib as L

pytestmark = pytest.mark.gpu


def _nan_pool(m, count):
    """`count` plans of m voxels evaluated at NaN, then closed."""
    row_ptr = np.arange(m + 1, dtype=np.int64)
    case = (row_ptr, np.zeros(m, np.int32), np.ones(m, np.float32), np.ones(m, np.uint8),
            np.array([[1.0, np.nan]], np.float32), np.array([[1.0, 0.0]], np.float32))
    plans = [Plan(*case, m=m, n=4, options=Options(lambda0=1.0)) for _ in range(count)]
    for p in plans:
        p.eval(np.full(4, np.nan, np.float32))
        p.close()


@pytest.mark.parametrize("precision", [L.FP32, L.FP16, L.FP8E4M3])
@pytest.mark.parametrize("k_trials", [1, 4])
def test_solve_after_the_pool_held_nan(precision, k_trials):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    case = phantom.random_case(17, m=2000, n=61, density=0.2, n_structures=2, empty_rows=0)
    keep = np.repeat(np.arange(case.m) >= 1040, np.diff(case.row_ptr))  # 960 voxels with entries: whole slices without
    lengths = np.where(np.arange(case.m) >= 1040, np.diff(case.row_ptr), 0)
    row_ptr = np.concatenate([[0], np.cumsum(lengths)]).astype(np.int64)
    args = (row_ptr, case.col[keep], case.val[keep], case.mask, case.thresholds, case.weights)
    options = Options(precision=precision, k_trials=k_trials, solver=L.SOLVER_TEAM, max_iter=25, delta=0.0)
    results = []
    for rep in range(6):
        if rep:
            _nan_pool(9 * 2016, 3 + rep)
        with Plan(*args, m=case.m, n=case.n, options=options) as plan:
            res = plan.solve()
            results.append((res.iterations, res.objective, plan.get_x().tobytes()))
    assert results[0][0] > 0 and len(set(results)) == 1
