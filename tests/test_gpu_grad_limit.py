"""bsp_grad takes plans of up to 64 shells and refuses more before it touches anything."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_more_than_64_shells_are_refused():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2107_14564_gb300 import binding
    ng = 128
    for ns in (64, 65):
        plan = binding.Plan(ng, float(ng), np.linspace(1.0, 41.0, ns + 1), precision="fp32")
        spec = torch.zeros(plan.spec_shape(), dtype=torch.complex64, device="cuda")
        g = torch.ones(plan.n_triplets, dtype=torch.float64, device="cuda")
        held = binding.bsp_plan_info(plan.handle)[3]
        if ns == 64:
            assert bool((plan.grad(spec, g) == 0).all())  # an empty field has no gradient
        else:
            with pytest.raises(binding.BispecError) as e:
                plan.grad(spec, g)
            assert e.value.status == 6  # BSP_ERR_NOT_SUPPORTED
            assert binding.bsp_plan_info(plan.handle)[3] == held
            b, _ = plan.estimate(spec)
            assert bool((b == 0).all())
        plan.close()
