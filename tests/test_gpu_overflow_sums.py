"""Triple sums that overflow are infinite, as the sum of their products is, not NaN."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2107_14564_gb300 import binding
    return binding


@pytest.mark.parametrize("prec,value", [("fp64", 1e150), ("fp64", 1e102), ("fp32", 1e20)])
def test_sums_that_overflow_are_infinite(lib, prec, value):
    """1e150: every product overflows; 1e102: finite products (1e306) whose sum of 24^3 voxels does not fit."""
    plan = lib.Plan(32, 32.0, np.linspace(1.0, 8.0, 9), precision=prec)
    s = plan.ng_eval
    assert plan.n_triplets > 0 and s ** 3 * 1e306 == np.inf
    f = torch.full((plan.n_shells,) + (s,) * 3, value, dtype=plan.real_dtype, device="cuda")
    f[0] = -f[0]  # bins of shell 0 alone or with two others are negative
    got = plan.contract(f).cpu().numpy()
    plan.check()
    for x, t in zip(got, plan.triplets):
        assert x == (-np.inf if [t["a"], t["b"], t["c"]].count(0) % 2 else np.inf)
    plan.close()
