"""plan_eval / plan_dose through every form of the caller's arrays: host and device, 16-byte aligned
(x read in place, results written in place) and not, n a multiple of 4 and not, results sharing memory
with x. Every form gives the same bits, and they match FP64 products of the same arrays."""
import numpy as np
import pytest

from paper_0908_4421_gb300 import Options, Plan, phantom

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,n,variant", [(1, 1, 0), (33, 4, 0), (3001, 56, 0), (3001, 57, 0), (2050, 64, 1),
                                         (2050, 63, 1), (2050, 64, 2), (2050, 65, 2)])
def test_eval_array_forms(m, n, variant):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    case = phantom.random_case(m + n, m=m, n=n, density=0.3, n_structures=2 if m > 1 else 1, empty_rows=m // 10)
    D = phantom.csr_to_dense(case)
    rng = np.random.Generator(np.random.PCG64(5))
    x = rng.uniform(0.0, 1.0, n).astype(np.float32)
    with Plan.from_case(case, Options(kernel_variant=variant, lambda0=1.0)) as plan:
        G0, z0, g0 = plan.eval(x)
        z64 = D @ x.astype(np.float64)
        # a row's FP32 sum of at most n products, all >= 0
        assert np.all(np.abs(z0 - z64) <= (n + 2) * 2.0 ** -23 * z64)
        for shift in (0, 1):  # floats past a 16-byte boundary
            xd = torch.zeros(n + 8, device="cuda")[shift:shift + n]
            xd.copy_(torch.from_numpy(x))
            zd = torch.full((m + 8,), -1.0, device="cuda")
            gd = torch.full((n + 8,), -1.0, device="cuda")
            z, g = zd[shift:shift + m], gd[shift:shift + n]
            G, _, _ = plan.eval(xd, z_out=z, g_out=g)
            assert G == G0 and np.array_equal(z.cpu().numpy(), z0) and np.array_equal(g.cpu().numpy(), g0)
            # nothing outside the results is written
            assert torch.all(zd[shift + m:] == -1.0) and torch.all(gd[shift + n:] == -1.0)
            assert np.array_equal(plan.dose(xd), z0)
            both = xd.clone()
            G, _, _ = plan.eval(both, z_out=z, g_out=both)  # g over x
            assert G == G0 and np.array_equal(both.cpu().numpy(), g0)
        shared = torch.zeros(m + n + 8, device="cuda")
        shared[:n] = torch.from_numpy(x)
        plan.dose(shared[:n], out=shared[:m])  # z over x
        assert np.array_equal(shared[:m].cpu().numpy(), z0)


@pytest.mark.parametrize("exponent", [-45, -33, 0, 30, 36])
def test_step_size_rule_scales_exactly(exponent):
    """D scaled by a power of two scales every number of the power iteration exactly, so lambda0 times the
    scale squared keeps its bits; the squares of the iterates reach far beyond the FP32 range."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    case = phantom.random_case(11, m=900, n=70, density=0.3, n_structures=2, empty_rows=20)
    rules = []
    for k in (0, exponent):
        val = np.ldexp(case.val, k).astype(np.float32)
        with Plan(case.row_ptr, case.col, val, case.mask, case.thresholds, case.weights, m=case.m, n=case.n) as plan:
            rules.append(plan.info()["lambda0_rule"])
    assert np.isfinite(rules[1]) and rules[1] > 0.0
    assert rules[1] * 4.0 ** exponent == rules[0]
