"""The adjoint products over every padded shell count and pair range, against the FP64 oracle.

The kernel is built for 8, 16, 24, 32, 48 and 64 padded shells and walks its pairs in lists by the
range of third shells they reach; each case lies just inside one of the sizes. The upstream gradient
is non-zero on 40 bins drawn over all kept ones, so that the oracle's sum stays short.
"""
import numpy as np
import pytest

import fieldgen
from oracle import grad as G
from oracle import plan as P

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ns,prec", [(2, "fp32"), (9, "fp32"), (17, "mixed_bf16x3"), (26, "fp32"), (34, "fp32"),
                                     (50, "mixed_bf16x3")])
def test_adjoint_over_shell_counts(ns, prec):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2107_14564_gb300 import binding
    ng, top = 128, 41.0 if ns > 30 else 32.0
    top = max(top, ns + 1.0) if ns < 41 else 42.0
    edges = np.linspace(1.0, top, ns + 1)
    delta = fieldgen.quadratic_field(ng, float(ng), 1.5, 0.2, 40 + ns).astype(np.float32)
    gp = binding.Plan(ng, float(ng), edges, precision=prec)
    pl = P.make_plan(ng, float(ng), edges)
    rng = np.random.default_rng(ns)
    pick = np.sort(rng.choice(gp.n_triplets, size=min(40, gp.n_triplets), replace=False))
    g = np.zeros(gp.n_triplets)
    g[pick] = rng.standard_normal(len(pick))
    t = gp.triplets[pick]
    want = G.vjp(delta.astype(np.float64), pl, [tuple(int(x) for x in v) for v in zip(t["a"], t["b"], t["c"])],
                 t["tsum"], g[pick])
    d = torch.from_numpy(delta).cuda()
    got = gp.grad(gp.spectrum(d), torch.from_numpy(g).cuda()).cpu().numpy()
    gp.check()
    assert np.abs(got - want).max() / np.abs(want).max() < 1e-4  # the FP32 bound of the adjoint's parity tests
    gp.close()
