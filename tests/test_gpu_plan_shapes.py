"""Plan creation makes the forward pass's work schedules that its step-size rule runs or hides; other plans make
one with the first call that needs it (plan_info reads device_bytes before it asks for the schedule)."""
import dataclasses

import numpy as np
import pytest

from paper_0908_4421_gb300 import Options, Plan, phantom
from paper_0908_4421_gb300 import _lib as L

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("solver,precision,lambda0,under,early", [
    (L.SOLVER_GRAPH, L.FP16, 0.0, True, True),
    (L.SOLVER_GRAPH, L.FP32, 1.0, False, True),
    (L.SOLVER_TEAM, L.FP16, 0.0, True, True),
    (L.SOLVER_TEAM, L.FP16, 1.0, False, False),
    (L.SOLVER_TEAM, L.FP32, 1.0, False, False),
])
def test_schedules_are_made_with_the_plan_or_at_first_use(solver, precision, lambda0, under, early):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    case = phantom.random_case(8, m=900, n=70, density=0.3, n_structures=2, empty_rows=20)
    thresholds = case.thresholds.copy()
    if not under:
        thresholds[:, 0] = np.nan
    case = dataclasses.replace(case, thresholds=thresholds)
    x = np.full(case.n, 0.5, np.float32)
    options = dict(precision=precision, lambda0=lambda0)
    with Plan.from_case(case, Options(solver=solver, **options)) as plan:
        first = plan.info()["device_bytes"]
        assert (plan.info()["device_bytes"] == first) == early
        G, z, g = plan.eval(x)
    with Plan.from_case(case, Options(**options)) as plan:  # the same results whenever it is made
        G0, z0, g0 = plan.eval(x)
    assert G == G0 and np.array_equal(z, z0) and np.array_equal(g, g0)
