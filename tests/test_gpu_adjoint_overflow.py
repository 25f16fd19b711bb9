"""The adjoint products form no product that the bins do not need: one that overflows would spoil the rest."""
import numpy as np
import pytest

from oracle import grad as G
from oracle import plan as P

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_adjoint_takes_no_product_outside_the_bins():
    """Shells |m|^2 = 4, 5, 6: no triangle has two sides in the first shell, whose field squared would
    overflow FP32 here. The gradient is finite and the oracle's."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2107_14564_gb300 import binding
    ng = 128
    edges = np.array([2.0, 2.2, 2.4, 2.6])
    gp = binding.Plan(ng, float(ng), edges, precision="fp32")
    trips = [(int(t["a"]), int(t["b"]), int(t["c"])) for t in gp.triplets]
    assert trips and all(t.count(0) < 2 for t in trips)
    rng = np.random.default_rng(3)
    pl = P.make_plan(ng, float(ng), edges)
    shell = P.shell_index_half(pl)
    amp = np.choose(shell.clip(0), (2e21, 1e12, 1e12)) * (shell >= 0)
    spec = amp * (rng.standard_normal(shell.shape) + 1j * rng.standard_normal(shell.shape))
    delta = np.fft.irfftn(spec, s=(ng,) * 3, axes=(0, 1, 2))
    spec = np.fft.rfftn(delta)
    g = rng.standard_normal(len(trips))
    want = G.vjp(delta, pl, trips, gp.triplets["tsum"], g)
    got = gp.grad(torch.from_numpy(spec.astype(np.complex64)).cuda(), torch.from_numpy(g).cuda()).cpu().numpy()
    gp.check()
    assert np.isfinite(got).all()
    assert np.abs(got - want).max() / np.abs(want).max() < 1e-4  # the FP32 bound of the adjoint's parity tests
    gp.close()
