"""The FP32 contraction where a block takes several groups of runs: exact sums of integer fields.

64 shells at Ng = 256 give the top level 512 groups of 32 runs and some tens of blocks of tiles, more than 64 blocks
per SM, so blocks take two or more groups, the last ones fewer, whole runs and remainders mixed. Fields hold
integers in [-2, 2]: every FP32 run is exact and so is every FP64 sum, whatever its order. 120 bins spread
over the plan's levels, on the plan that holds all fields and on one under a budget, whose bsp_contract sums
every bin on the evaluation grid.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("planes", [0, 100])
def test_blocks_of_several_groups(planes):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2107_14564_gb300 import binding
    ng, ns = 256, 64
    plan = binding.Plan(ng, float(ng), np.linspace(1.0, 85.0, ns + 1), precision="fp32",
                        mem_budget_bytes=planes * ns * ng * ng * 4)
    assert plan.ng_eval == ng and plan.slabs[0] == planes
    gen = torch.Generator(device="cuda").manual_seed(7)
    f = torch.randint(-2, 3, (ns, ng, ng, ng), device="cuda", generator=gen, dtype=torch.int8)
    got = plan.contract(f.float()).cpu().numpy()
    plan.check()
    for i in np.linspace(0, plan.n_triplets - 1, 120).astype(int):
        b = plan.triplets[i]
        t = ng // plan.tuning[plan.bin_level[i]][0]
        x, y, z = (f[int(b[k]), ::t, ::t, ::t] for k in "abc")
        want = int((x * y * z).sum(dtype=torch.int64))  # products within [-8, 8]
        assert got[i] == pytest.approx(float(t) ** 3 * want, rel=1e-15, abs=0.0)
    plan.close()
