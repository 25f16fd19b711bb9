"""The contraction bytes a CUDA-core plan reports: each level's samples of its shells' fields, read once."""
import ctypes as C

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
def test_contraction_bytes(prec):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2107_14564_gb300 import _lib, binding
    ng, ns = 128, 16
    plan = binding.Plan(ng, float(ng), np.linspace(1.0, 32.0, ns + 1), precision=prec)
    b, f = (C.c_double * 5)(), (C.c_double * 5)()
    _lib.check(_lib.load().bsp_plan_stage_work(plan.handle, b, f))
    assert len(plan.tuning) > 1
    values = 0
    for level, (g, _) in enumerate(plan.tuning):
        t = plan.triplets[plan.bin_level == level]
        shells = ns if g == plan.ng_eval else len(set(t["a"]) | set(t["b"]) | set(t["c"]))
        values += shells * g ** 3
    assert b[3] == values * (8 if prec == "fp64" else 4)
    plan.close()
