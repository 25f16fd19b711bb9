"""The warp passes at the sides the other tests of single passes leave out: shell fields at 768 and 1024, the forward
spectrum at 192, 512, 768 and 1024.

Fields: random modes of two thin shells whose radius needs the whole grid; single x-planes against the sum over
k_x of Eq. (2.8) and a numpy inverse transform in FP64. Bound: that of the FP32 fields' parity tests, 2e-6 of a
shell's largest value (the planes hold the origin's, where all modes add up).
Spectrum: against the FP64 transform of the same FP32 field on the shells' modes. Bound: that of the
spectrum's parity test, 1e-5 of the largest mode.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _modes(rng, lo, hi, count):
    """Distinct modes with k_z > 0 and lo <= |m| < hi."""
    out = set()
    while len(out) < count:
        v = rng.standard_normal((count, 3))
        m = np.rint(v / np.linalg.norm(v, axis=1)[:, None] * rng.uniform(lo, hi, (count, 1))).astype(int)
        q = (m * m).sum(axis=1)
        for x in m[(q >= lo * lo) & (q < hi * hi) & (m[:, 2] > 0)]:
            out.add(tuple(int(c) for c in x))
    return np.array(sorted(out))


@pytest.mark.parametrize("ng,edges", [(768, (172.2, 172.8, 173.4)), (1024, (257.5, 258.0, 258.5))])
def test_shell_fields_of_long_lines(ng, edges):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2107_14564_gb300 import binding
    plan = binding.Plan(ng, float(ng), np.array(edges), precision="fp32")
    assert plan.ng_eval == ng
    rng = np.random.default_rng(ng)
    spec = torch.zeros(plan.spec_shape(), dtype=torch.complex64, device="cuda")
    modes, amps = [], []
    for lo, hi in zip(edges[:-1], edges[1:]):
        m = _modes(rng, lo, hi, 20000)
        a = (rng.standard_normal(len(m)) + 1j * rng.standard_normal(len(m)) + 1.0).astype(np.complex64)
        i = torch.from_numpy(m % ng).cuda()
        spec[i[:, 0], i[:, 1], i[:, 2]] = torch.from_numpy(a).cuda()
        modes.append(m)
        amps.append(a.astype(np.complex128))
    got = plan.shell_fields(spec)
    plan.check()
    for n in range(2):
        m, a = modes[n], amps[n]
        for x in (0, 1, ng // 3, ng - 1):
            half = np.zeros((ng, ng // 2 + 1), dtype=np.complex128)
            np.add.at(half, (m[:, 1] % ng, m[:, 2]), a * np.exp(2j * np.pi * ((m[:, 0] * x) % ng) / ng))
            want = np.fft.irfft2(half, s=(ng, ng), axes=(0, 1)) * ng ** 2
            if x == 0:
                peak = np.abs(want).max()
                assert peak > 20000  # the origin: 2 Re of the amplitudes' sum
            assert np.abs(got[n, x].cpu().numpy() - want).max() <= 2e-6 * peak
    plan.close()


@pytest.mark.parametrize("ng", [192, 512, 768, 1024])
def test_spectrum_of_long_lines(ng):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2107_14564_gb300 import binding
    top = {192: 40.5, 512: 90.5, 768: 120.5, 1024: 150.5}[ng]
    plan = binding.Plan(ng, float(ng), np.array([top - 1.0, top - 0.5, top]), precision="fp32")
    delta = torch.randn((ng,) * 3, dtype=torch.float32, device="cuda", generator=torch.Generator(device="cuda").manual_seed(ng))
    got = plan.spectrum(delta)
    plan.check()
    plan.close()
    want = torch.fft.rfftn(delta.double())
    del delta
    k = torch.fft.fftfreq(ng, 1.0 / ng, device="cuda", dtype=torch.float64).round()
    kz = torch.arange(ng // 2 + 1, device="cuda", dtype=torch.float64)
    worst, largest = 0.0, 0.0
    for x in range(ng):
        q = k[x] ** 2 + k[:, None] ** 2 + kz[None, :] ** 2
        inside = (q >= (top - 1.0) ** 2) & (q < top * top)
        assert bool((got[x][~inside] == 0).all())
        if bool(inside.any()):
            worst = max(worst, float((got[x][inside] - want[x][inside]).abs().max()))
            largest = max(largest, float(want[x][inside].abs().max()))
    assert worst < 1e-5 * largest
