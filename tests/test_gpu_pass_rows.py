"""Shell fields at every evaluation grid of the warp passes, with radii around the passes' tiles.

Rows of the pass buffers are padded to 8 k_z and a warp of the X (to 256 points) and Y (to 384)
passes takes 4 neighbouring k_z: shell radii cover every remainder by 4 and 8, a radius below 4, grids
on both sides of the two limits, and lines that fill no whole block. Bound: that of the FP32 fields'
parity tests, 2e-6 of a shell's largest value.
"""
import numpy as np
import pytest

import fieldgen
from oracle import fbe
from oracle import plan as P

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ng,edges,beta", [
    (128, (1.0, 1.5, 7.0, 13.5, 22.0, 33.0), None), (128, (1.0, 2.0, 18.5, 34.0, 41.5), 0.5),
    (192, (1.0, 3.0, 23.0, 48.2, 60.9), None), (192, (1.0, 12.0, 45.0, 63.0), 0.5),
    (256, (1.0, 9.0, 66.0, 71.3, 84.0), None), (384, (118.2, 121.4, 125.0), 0.5),
    (512, (128.0, 131.0, 133.5), None),
])
def test_shell_fields_over_radii(ng, edges, beta):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2107_14564_gb300 import binding
    delta = fieldgen.quadratic_field(ng, float(ng), 1.5, 0.05, ng).astype(np.float32)
    spec = np.ascontiguousarray(np.fft.rfftn(delta.astype(np.float64)).astype(np.complex64))
    gp = binding.Plan(ng, float(ng), np.array(edges), precision="fp32", rsd=beta is not None, beta=beta or 0.0)
    assert gp.ng_eval == ng
    pl = P.make_plan(ng, float(ng), np.array(edges))
    spec64 = spec.astype(np.complex128)
    if beta is not None:
        spec64 = spec64 * fbe.kaiser_factor_half(ng, beta)
    got = gp.shell_fields(torch.from_numpy(spec).cuda()).cpu().numpy()
    gp.check()
    want = fbe.shell_fields_on_grid(spec64, pl, ng)
    for n in range(pl.ns):
        assert np.abs(got[n] - want[n]).max() <= 2e-6 * np.abs(want[n]).max(), n
    gp.close()
