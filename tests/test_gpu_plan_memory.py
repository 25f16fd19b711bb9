"""What an FP32 plan holds besides its fields and pass buffers: partial sums that do not grow with the voxels.

A level's partial sums are at most 64 rows per SM of one block's outputs (12 tiles of 64 doubles), or
one row of each; the tables (work items, tiles, bins) stay below 32 MB at these sizes. One double per 32 runs of
1024 voxels and output would take 0.6 GB here.
"""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("planes", [0, 32])
def test_partial_sums_are_bounded(planes):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2107_14564_gb300 import binding
    ng, ns = 256, 100
    edges = np.linspace(1.0, 85.0, ns + 1)
    plan = binding.Plan(ng, float(ng), edges, precision="fp32", mem_budget_bytes=planes * ns * ng * ng * 4)
    s = plan.ng_eval
    assert s == ng and plan.slabs[0] == planes
    held = ns * s * s * (planes or s) * 4
    for e in edges[1:]:
        r = math.isqrt(math.ceil(e * e) - 1) + 1
        pitch = (r + 7) // 8 * 8
        held += (s * (2 * r - 1) * pitch + s * s * pitch) * 8
    n_sm = torch.cuda.get_device_properties(0).multi_processor_count
    row = 12 * 64 * 8
    assert plan.device_bytes - held < len(plan.tuning) * 64 * n_sm * row + 32e6
    plan.close()


@pytest.mark.parametrize("prec,ng,ns,top", [("fp64", 128, 16, 32.0), ("fp32", 96, 30, 31.0)])
def test_generic_passes_hold_unpadded_rows(prec, ng, ns, top):
    """Rows of the generic 3D passes' buffers hold r k_z. Padded to 8, the buffers would be 18.7 MB (FP64) and
    10.2 MB (FP32) larger; everything else (tables, FP64 partial sums) takes less than 6 MB."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2107_14564_gb300 import binding
    edges = np.linspace(1.0, top, ns + 1)
    plan = binding.Plan(ng, float(ng), edges, precision=prec)
    s, elem = plan.ng_eval, 8 if prec == "fp64" else 4
    held = ns * s ** 3 * elem
    for e in edges[1:]:
        r = math.isqrt(math.ceil(e * e) - 1) + 1
        held += (s * (2 * r - 1) * r + s * s * r) * 2 * elem
    assert plan.device_bytes - held < 6e6
    plan.close()
