"""bsp_contract on plans under a memory budget: the caller's fields are whole, whatever the slabs.

The integer fields of the contraction's own test: every FP32 run and every FP64 sum is exact, so the
sums must be numpy's, to the rounding of the one multiplication by the grid ratio. Slabs of one plane,
a thinner last slab, equal slabs, and a grid of the warp passes.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,ng,ns,top,planes", [
    ("fp32", 16, 1, 4.0, 1), ("fp32", 64, 12, 16.0, 7), ("fp32", 128, 16, 32.0, 40), ("fp32", 128, 16, 32.0, 32),
    ("fp64", 16, 1, 4.0, 1), ("fp64", 64, 12, 16.0, 7), ("fp64", 96, 30, 31.0, 24),
])
def test_contract_whole_fields_under_a_budget(prec, ng, ns, top, planes):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2107_14564_gb300 import binding
    edges = np.linspace(1.0, top, ns + 1)
    whole = binding.Plan(ng, float(ng), edges, precision=prec)
    s = whole.ng_eval
    whole.close()
    elem = 8 if prec == "fp64" else 4
    plan = binding.Plan(ng, float(ng), edges, precision=prec, mem_budget_bytes=planes * ns * s * s * elem)
    assert plan.slabs == (planes, -(-s // planes)) and plan.slabs[1] > 1
    rng = np.random.default_rng(ng * 100 + ns)
    f = rng.integers(-2, 3, size=(ns, s, s, s))
    got = plan.contract(torch.from_numpy(f).to(plan.real_dtype).cuda()).cpu().numpy()
    plan.check()
    h = f.reshape(ns, -1)
    scale = (ng / s) ** 3
    assert plan.n_triplets > 0
    for i, b in enumerate(plan.triplets):
        assert got[i] == pytest.approx(scale * float(np.sum(h[b["a"]] * h[b["b"]] * h[b["c"]])), rel=1e-15, abs=0.0)
    plan.close()
