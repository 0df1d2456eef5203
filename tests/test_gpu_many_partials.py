"""The Armijo controller where G has more objective partials than one warp adds whole (256; the device-wide
schedules leave one per 1,024 voxels): the objective a solve ends with is plan_eval's at its x, which another
kernel path adds, and the iterations are those of the CTA-local schedule, whose partials are one a CTA."""
import numpy as np
import pytest

from paper_0908_4421_gb300 import Options, Plan

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m", [262144, 262145, 1100000, 2500000])  # 256, 257, 1075 and 2442 partials
@pytest.mark.parametrize("variant,k_trials", [(1, 1), (2, 1), (2, 8)])
def test_objective_over_many_partials(m, variant, k_trials):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    rng = np.random.Generator(np.random.PCG64(m))
    j = np.arange(m)
    col = np.stack([j % 5, 5 + j % 7, 12 + j % 4], 1).astype(np.int32).ravel()
    val = rng.uniform(0.05, 1.0, col.size).astype(np.float32)
    mask = rng.integers(0, 4, m).astype(np.uint8)
    mask[-1] = 1
    thr, w = np.array([[3.0, 5.0], [np.nan, 1.0]], np.float32), np.array([[2.0, 3.0], [0.0, 1.0]], np.float32)
    arrays = [torch.from_numpy(a).cuda() for a in (np.arange(m + 1, dtype=np.int64) * 3, col, val, mask)]
    iterations = []
    for v in (0, variant):
        with Plan(*arrays, thr, w, m=m, n=16,
                  options=Options(kernel_variant=v, k_trials=k_trials, max_iter=12, delta=0.0)) as plan:
            res = plan.solve()
            G = plan.eval(plan.get_x())[0]
            iterations.append(res.iterations)
            # both add the same FP64 partials: m / 1024 roundings of 2^-53 at most
            assert res.status == 0 and G > 0.0 and abs(res.objective - G) <= m / 1024 * 2.0 ** -53 * G
    assert iterations[0] == iterations[1] > 0
