"""lambda0 of the step-size rule against the FP64 oracle where a thread of the norm holds more than one
beamlet (n > 512), at the edges of its thread and warp shares."""
import numpy as np
import pytest

from paper_0908_4421_gb300 import Options, Plan, phantom

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [511, 513, 1030, 3001])
@pytest.mark.parametrize("variant", [0, 2])
def test_rule_beyond_one_beamlet_a_thread(orc, n, variant):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    case = phantom.random_case(n, m=1500, n=n, density=0.02, n_structures=2, empty_rows=20)
    with Plan.from_case(case, Options(kernel_variant=variant)) as plan:
        got = plan.info()["lambda0_rule"]
    # every number is >= 0, so FP32 errors stay relative: a pass adds at most one rounding per entry of a row
    # and of a column and 8 for the coefficients, and lambda = v . w holds 50 passes twice over
    longest = int(np.diff(case.row_ptr).max()) + int(np.bincount(case.col, minlength=n).max())
    bound = 102 * (longest + 8) * 2.0 ** -24
    assert abs(got / orc.lambda0_rule(case) - 1.0) <= bound
