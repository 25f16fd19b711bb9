"""The CUDA-core contraction on integer fields, whose sums are exact in FP32 and FP64.

Fields hold integers in [-2, 2], so every product is at most 8, every FP32 run of 1024 voxels stays
below 2^24 and every sum is an exact integer: the kernels must give numpy's integer sums times the
grid ratio, without a tolerance beyond that one product's rounding. Sizes cover runs shorter than
1024 voxels, whole runs with and without remainders, voxel counts that are no multiple of 64 or 32,
one to forty shells (tiles and blocks partly filled), every coarser contraction level, and 2D.
"""
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


CASES = [  # precision, dim, ng, shells, top
    ("fp32", 3, 16, 1, 4.0), ("fp32", 3, 32, 8, 8.0), ("fp32", 3, 54, 5, 17.3), ("fp32", 3, 64, 12, 16.0),
    ("fp32", 3, 72, 20, 23.0), ("fp32", 3, 128, 16, 32.0), ("fp32", 3, 128, 40, 41.0), ("fp32", 2, 54, 3, 17.3),
    ("fp32", 2, 384, 15, 31.0), ("fp64", 3, 16, 1, 4.0), ("fp64", 3, 32, 8, 8.0), ("fp64", 3, 54, 5, 17.3),
    ("fp64", 3, 64, 12, 16.0), ("fp64", 3, 96, 30, 31.0), ("fp64", 2, 54, 3, 17.3), ("fp64", 2, 384, 15, 31.0),
]


@pytest.mark.parametrize("prec,dim,ng,ns,top", CASES)
def test_contract_integer_fields(lib, prec, dim, ng, ns, top):
    plan = lib.Plan(ng, float(ng), np.linspace(1.0, top, ns + 1), precision=prec, dim=dim)
    s = plan.ng_eval
    rng = np.random.default_rng(ng * 100 + ns)
    f = rng.integers(-2, 3, size=(ns,) + (s,) * dim)
    got = plan.contract(torch.from_numpy(f).to(plan.real_dtype).cuda()).cpu().numpy()
    plan.check()
    assert plan.n_triplets > 0
    for level, (g, _) in enumerate(plan.tuning):
        t = s // g
        h = f[(slice(None),) + (slice(None, None, t),) * dim].reshape(ns, -1)
        scale = (ng / g) * (ng / g) * ((ng / g) if dim == 3 else 1.0)
        for i in np.flatnonzero(plan.bin_level == level):
            b = plan.triplets[i]
            want = float(np.sum(h[b["a"]] * h[b["b"]] * h[b["c"]]))
            assert got[i] == pytest.approx(scale * want, rel=1e-15, abs=0.0)
    plan.close()
