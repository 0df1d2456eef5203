"""The algorithmic bytes a plan reports count what a solve's passes read and write: no dose is stored."""
import pytest

from paper_0908_4421_gb300 import Options, Plan, phantom
from paper_0908_4421_gb300 import _lib as L

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,value_bytes", [(L.FP32, 4), (L.FP16, 2), (L.FP8E4M3, 1)])
@pytest.mark.parametrize("solver", [L.SOLVER_GRAPH, L.SOLVER_TEAM])
def test_bytes_of_the_passes(precision, value_bytes, solver):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    c = phantom.random_case(4, m=900, n=70, density=0.3, n_structures=2, empty_rows=20)

    def passes(vb):
        # 16-bit indices both ways (one segment); row offsets and x, mask, r order and r; segment offsets, r and g
        return (c.nnz * (vb + 2) + (c.m + 1) * 8 + c.n * 4 + c.m * (1 + 4 + 4),
                c.nnz * (vb + 2) + (c.n + 1) * 8 + c.m * 4 + c.n * 4)

    with Plan.from_case(c, Options(precision=precision, solver=solver, max_iter=8, polish_iter=0)) as plan:
        info, res = plan.info(), plan.solve()
    fwd, bwd = passes(value_bytes)
    assert (info["fwd_bytes"], info["bwd_bytes"]) == (fwd, bwd)
    assert res.bytes == fwd * res.passes + bwd * res.grad_passes
