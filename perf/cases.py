"""The work a user of the bispectrum library has it do, as timed cases.

Every case is one pass through the public Python binding: an estimate of every bin of one field
(FP64, FP32 or split-BF16 plans; cubes and 2D boxes; with and without redshift space, memory
budgets and host buffers), a captured batch of estimates, the shell fields, or the differentiable
estimate with its gradient. Fields are the quadratic non-Gaussian ones of the paper's Sec. 3,
delta = delta_G + f (delta_G^2 - mean), drawn on the GPU from the seed; sizes are those of the
repository's benchmark, tests and of the paper's own runs.
"""
import math

import numpy as np
import torch

from paper_2107_14564_gb300 import autograd, binding

GIB = 1 << 30


def listed():
    base = dict(kind="estimate", dim=3, lo=1.0, n_mu=20, n_t=20, beta=0.0, n_index=1.5, f_ng=0.05, budget=0)
    return [
        # a whole small analysis in double precision (parity runs, notebooks): latency and launches
        dict(base, name="fp64-ng32", ng=32, box=32.0, ns=8, hi=8.0, n_mu=10, n_t=10, precision="fp64", n_index=2.0,
             f_ng=0.1),
        # the paper's 2D box (Sec. 2.1): 15 rings 2 k_f wide on a 384^2 square; the smallest call in single precision
        dict(base, name="ring2d-fp32-ng384", dim=2, ng=384, box=215.0, ns=15, hi=31.0, n_mu=10, n_t=10,
             precision="fp32", n_index=2.0, f_ng=0.5),
        # one realisation of a small simulation suite
        dict(base, name="fp32-ng128", ng=128, box=128.0, ns=16, hi=32.0, n_mu=10, n_t=10, precision="fp32"),
        # the double-precision check a user runs beside a single-precision analysis
        dict(base, name="fp64-ng128", ng=128, box=128.0, ns=16, hi=32.0, n_mu=10, n_t=10, precision="fp64"),
        # the paper's own 3D runs (Sec. 3): Ng = 384, L = 215, N_r = 30 shells one k_f wide, far below Nyquist
        dict(base, name="bf16x3-ng384-paper30", ng=384, box=215.0, ns=30, hi=31.0, n_mu=10, n_t=10,
             precision="mixed_bf16x3", n_index=2.0, f_ng=0.5),
        # the ordinary single-precision analysis: 24 shells to half the Nyquist wavenumber
        dict(base, name="fp32-ng256", ng=256, box=256.0, ns=24, hi=64.0, precision="fp32"),
        # the benchmark: redshift space, 32 shells, tensor cores
        dict(base, name="bf16x3-ng512-rsd", ng=512, box=512.0, ns=32, hi=128.0, beta=0.5, precision="mixed_bf16x3"),
        # the largest grid in FP32, its shell fields streamed slab by slab under a memory budget
        dict(base, name="fp32-ng768-8gib", ng=768, box=768.0, ns=24, hi=192.0, precision="fp32", budget=8 * GIB),
        # a pipeline that reads spectra into pinned host memory and wants host results
        dict(base, name="host-bf16x3-ng256", kind="host", ng=256, box=256.0, ns=24, hi=64.0,
             precision="mixed_bf16x3"),
        # an ensemble of 64 realisations on uneven grids, captured once and replayed
        dict(base, name="batch64-fp32", kind="batch", n128=16, n192=24, n256=24, ns=16, n_mu=10, n_t=10,
             precision="fp32"),
        # field-level inference: forward estimate, loss against the analytic bispectrum, gradient
        dict(base, name="grad-fp32-ng256", kind="grad", ng=256, box=256.0, ns=24, hi=64.0, precision="fp32"),
        # the shell fields themselves (for a caller's own statistics)
        dict(base, name="fields-fp32-ng384", kind="fields", ng=384, box=384.0, ns=8, hi=96.0, n_mu=10, n_t=10,
             precision="fp32"),
    ]


# ---------------------------------------------------------------- draws over the same ranges
GRIDS = {"fp64": (32, 36, 48, 54, 64, 72, 96, 108, 128, 144, 192),
         "fp32": (32, 48, 64, 72, 96, 108, 128, 144, 192, 216, 256, 288, 384, 432, 512),
         "mixed_bf16x3": (64, 72, 96, 128, 144, 192, 216, 256, 288, 384, 432, 512)}
WARP = (128, 192, 256, 384)
RATE = {"fp64": 0.4e12, "fp32": 12e12, "mixed_bf16x3": 100e12}  # rough, to keep draws below the largest listed case


def draw(rng):
    while True:
        c = _draw(rng)
        w = work(c)
        if w["flops"] / RATE[c["precision"]] < 0.1 and w["bytes"] < 4e9:
            return c


def _draw(rng):
    kind = rng.choice(["estimate"] * 5 + ["host", "batch", "grad", "grad", "fields", "ring"])
    prec = rng.choice(["fp64"] + ["fp32"] * 2 + ["mixed_bf16x3"] * 2)
    cells = rng.choice([1, 5, 10, 20])
    c = dict(kind=kind, dim=3, lo=1.0, n_mu=cells, n_t=cells, beta=0.0, n_index=rng.choice([1.5, 2.0]),
             f_ng=rng.choice([0.05, 0.1]), budget=0)
    if kind == "batch":
        c.update(n128=rng.randint(1, 12), n192=rng.randint(0, 12), n256=rng.randint(0, 12), ns=rng.randint(6, 16),
                 precision=rng.choice(["fp32", "mixed_bf16x3"]))
        return c
    if kind == "ring":
        ng = rng.choice([96, 128, 144, 192, 256, 288, 384, 512, 768, 1024])
        c.update(kind="estimate", dim=2, precision=rng.choice(["fp32", "fp64"]))
    elif kind in ("grad", "fields"):
        ng = rng.choice(WARP)
        c["precision"] = rng.choice(["fp32", "fp32", "mixed_bf16x3"]) if kind == "grad" else "fp32"
    else:
        ng = rng.choice(GRIDS[prec])
        c["precision"] = prec
    hi = ng * rng.uniform(1 / 8, 1 / 3.1)
    most = int(min(16 if kind == "fields" else 40, hi - 1.0))
    ns = max(2, int(round(math.exp(rng.uniform(math.log(3), math.log(max(most, 4)))))))
    ns = min(ns, max(most, 2))
    c.update(ng=ng, box=float(ng), ns=ns, hi=round(hi, 3))
    if c["dim"] == 3 and rng.random() < 0.3:
        c["beta"] = 0.5
    if kind == "estimate" and c["dim"] == 3 and ng in (192, 256, 384, 512) and prec != "fp64" and rng.random() < 0.3:
        c["budget"] = max(ns * ng * ng * 4 * 4, ns * ng ** 3)  # about a quarter of the shell fields
    return c


# ---------------------------------------------------------------- inputs
def _edges(c, ng=None):
    hi = c["hi"] if ng is None else ng / 4.0
    return np.linspace(c["lo"], hi, c["ns"] + 1)


def _field(ng, box, c, seed, dim=3):
    """delta(x) in FP64 on the GPU: power law P = k^-n with the quadratic term of Eq. (3.1)."""
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    shape = (ng,) * dim
    wk = torch.fft.rfftn(torch.randn(shape, generator=gen, device="cuda", dtype=torch.float64))
    wk *= _amplitude(ng, box, c["n_index"], dim)
    dg = torch.fft.irfftn(wk, s=shape)
    del wk
    sq = dg * dg
    return dg + c["f_ng"] * (sq - sq.mean())


def _amplitude(ng, box, n_index, dim):
    m = torch.fft.fftfreq(ng, d=1.0 / ng, device="cuda", dtype=torch.float64)
    mz = torch.arange(ng // 2 + 1, device="cuda", dtype=torch.float64)
    q = mz ** 2
    for _ in range(dim - 1):
        q = (m ** 2).reshape((-1,) + (1,) * q.dim()) + q
    q.view(-1)[0] = 1.0
    amp = (((2 * math.pi / box) ** 2 * q) ** (-n_index / 2) / (box / ng) ** dim).sqrt_()
    amp.view(-1)[0] = 0.0
    return amp


def _spec(ng, box, c, seed, dim=3):
    s = torch.fft.rfftn(_field(ng, box, c, seed, dim))
    return (s if c["precision"] == "fp64" else s.to(torch.complex64)).contiguous()


def _batch_grids(c):
    return [ng for ng in (128, 192, 256) for _ in range(c["n%d" % ng])]


def _plan(c, ng, box, edges):
    return binding.Plan(ng, box, edges, c["n_mu"], c["n_t"], rsd=c["beta"] != 0.0, beta=c["beta"],
                        precision=c["precision"], mem_budget_bytes=c["budget"], dim=c["dim"])


def _analytic(c, k):
    """Eq. (3.2) at side lengths k = (k1, k2, k3), units of k_f."""
    p = [(np.asarray(x) * (2 * math.pi / c["box"])) ** -c["n_index"] for x in k]
    return 2 * c["f_ng"] * (p[0] * p[1] + p[1] * p[2] + p[2] * p[0])


def prepare(case, seed):
    c = case
    if c["kind"] == "batch":
        plans, specs = {}, []
        for i, ng in enumerate(_batch_grids(c)):
            if ng not in plans:
                plans[ng] = _plan(c, ng, float(ng), _edges(c, ng))
            specs.append(_spec(ng, float(ng), c, 1000 * seed + i))
        return dict(kind="batch", batch=binding.Batch([plans[ng] for ng in _batch_grids(c)], specs))
    plan = _plan(c, c["ng"], c["box"], _edges(c))
    if c["kind"] == "grad":
        t = plan.triplets
        b_ana = torch.from_numpy(_analytic(c, (t["k1"], t["k2"], t["k3"]))).cuda()
        delta = _field(c["ng"], c["box"], c, seed).float().requires_grad_()
        return dict(kind="grad", plan=plan, delta=delta, b_ana=b_ana)
    spec = _spec(c["ng"], c["box"], c, seed, c["dim"])
    if c["kind"] == "host":
        spec = spec.cpu().pin_memory()
    return dict(kind=c["kind"], plan=plan, spec=spec)


def run(state):
    kind = state["kind"]
    if kind == "batch":
        return state["batch"].run()
    plan = state["plan"]
    if kind == "estimate":
        return plan.estimate(state["spec"])
    if kind == "host":
        return plan.estimate_host(state["spec"])
    if kind == "fields":
        return plan.shell_fields(state["spec"])
    b = autograd.bispectrum(state["delta"], plan)
    loss = ((b - state["b_ana"]) / state["b_ana"]).square().sum()
    grad, = torch.autograd.grad(loss, state["delta"])
    return b.detach(), grad


# ---------------------------------------------------------------- the work a pass cannot do without
def _geometry(edges):
    """(q thresholds, r per shell): mode m is in shell n iff q[n] <= |m|^2 < q[n + 1]."""
    q = [int(math.ceil(e * e)) for e in edges]
    q[0] = max(1, q[0])
    return q, [math.isqrt(x - 1) + 1 for x in q[1:]]


def _pairs(q):
    """(a, b, number of c, largest c) of the shell pairs whose triangles can close."""
    ns = len(q) - 1
    far = [math.sqrt(x - 1) for x in q[1:]]
    for a in range(ns):
        for b in range(a + 1):
            cs = [x for x in range(b + 1) if math.sqrt(q[a]) <= far[b] + far[x]]
            if cs:
                yield a, b, len(cs), cs[-1]


def _estimate_work(c, ng, edges):
    """Half-ball modes read, bins written; pruned FFTs and triple products on the smallest exact grids."""
    q, r = _geometry(edges)
    dim = c["dim"]
    m = 3 * (r[-1] - 1) + 1
    size = 16 if c["precision"] == "fp64" else 8
    modes = math.pi * (q[-1] - q[0]) / 2 if dim == 2 else 2 * math.pi / 3 * (q[-1] ** 1.5 - q[0] ** 1.5)
    fft = 0.0
    for x in r:
        lines = x if dim == 2 else math.pi / 2 * x * x + m * x
        fft += 5 * m * math.log2(m) * (lines + m ** (dim - 1) / 2)
    prod, bins = 0.0, 0
    for a, b, n, cmax in _pairs(q):
        prod += (1 + 2 * n) * float(r[a] + r[b] + r[cmax] - 2) ** dim
        bins += n
    out = 8 * (bins + c["ns"] * c["n_mu"] * c["n_t"])
    return modes * size, out, fft, prod


def work(case):
    c = case
    if c["kind"] == "batch":
        each = {ng: _estimate_work(c, ng, _edges(c, ng)) for ng in set(_batch_grids(c))}
        got = [each[ng] for ng in _batch_grids(c)]
        return dict(bytes=sum(x[0] + x[1] for x in got), flops=sum(x[2] + x[3] for x in got))
    read, out, fft, prod = _estimate_work(c, c["ng"], _edges(c))
    if c["kind"] == "fields":
        s = float(_fields_grid(c)) ** 3
        return dict(bytes=read + 4 * c["ns"] * s, flops=fft)
    if c["kind"] == "grad":  # delta in, gradient out; fields and products forward and back
        return dict(bytes=8.0 * c["ng"] ** 3 + out, flops=2 * fft + 2 * prod)
    return dict(bytes=read + out, flops=fft + prod)


# ---------------------------------------------------------------- the same in 64 bits, by plain torch
def _smooth(n, top):
    """The smallest even 2-3-5-smooth number from n, at most top."""
    for m in range(n + n % 2, top, 2):
        k = m
        for f in (2, 3, 5):
            while k % f == 0:
                k //= f
        if k == 1:
            return m
    return top


def _fields_grid(c):
    """The side shell_fields samples on: the smallest of its grids above 3 (r - 1), else ng."""
    need = 3 * (_geometry(_edges(c))[1][-1] - 1) + 1
    return next((s for s in (128, 192, 256, 384, 512, 768) if need <= s < c["ng"]), c["ng"])


def _axes(n, r):
    """Indices of the modes -(r-1) .. r-1 on a full axis of n, in that order."""
    return torch.arange(-(r - 1), r, device="cuda") % n


def _box(spec, ng, r, dim):
    """The modes |m_i| < r of a half spectrum, and their |m|^2 and m_z^2."""
    i = _axes(ng, r)
    m = torch.arange(-(r - 1), r, device="cuda", dtype=torch.float64) ** 2
    z = torch.arange(r, device="cuda", dtype=torch.float64) ** 2
    if dim == 2:
        return spec[i][:, :r], m[:, None] + z, z
    return spec[i][:, i][:, :, :r], m[:, None, None] + m[:, None] + z, z


def _to_grid(box, n, r, dim):
    out = torch.zeros((n,) * (dim - 1) + (n // 2 + 1,), dtype=torch.complex128, device="cuda")
    i = _axes(n, r)
    k = min(r, n // 2 + 1)
    if dim == 2:
        out[i[:, None], torch.arange(k, device="cuda")] = box[..., :k]
    else:
        out[i[:, None, None], i[:, None], torch.arange(k, device="cuda")] = box[..., :k]
    return torch.fft.irfftn(out, s=(n,) * dim, norm="forward")


def _shells(c, ng, edges, spec, n, unit=False):
    """The shell fields [ns][n^dim] of a half spectrum (or of ones) by masked inverse transforms."""
    q, r = _geometry(edges)
    box, m2, z2 = _box(spec, ng, r[-1], c["dim"])
    box = torch.ones_like(box, dtype=torch.complex128) if unit else box.to(torch.complex128)
    if c["beta"] and not unit:
        box = box * (1 + c["beta"] * z2 / m2.clamp(min=1))
    return torch.stack([_to_grid(box * ((m2 >= q[i]) & (m2 < q[i + 1])), n, r[-1], c["dim"]).reshape(-1)
                        for i in range(c["ns"])])


def _sums(fields, pairs):
    """[pairs][ns]: sums over the voxels of d_a d_b d_c."""
    a = torch.tensor([p[0] for p in pairs], device="cuda")
    b = torch.tensor([p[1] for p in pairs], device="cuda")
    got = torch.zeros((len(pairs), len(fields)), dtype=torch.float64, device="cuda")
    step = max(1, (1 << 27) // len(pairs))
    for v in range(0, fields.shape[1], step):
        f = fields[:, v:v + step]
        got += (f[a] * f[b]) @ f.T
    return got


def _bins(c, ng, box, edges, spec):
    """Kept bins (a, b, c), their values, triangle counts and fields, in 64 bits."""
    q, r = _geometry(edges)
    dim = c["dim"]
    n = _smooth(3 * (r[-1] - 1) + 1, ng)
    pairs = [(a, b) for a, b, _, _ in _pairs(q)]
    ntri = torch.round(_sums(_shells(c, ng, edges, spec, n, unit=True), pairs) / float(n) ** dim).cpu().numpy()
    fields = _shells(c, ng, edges, spec, n)
    sums = _sums(fields, pairs).cpu().numpy() / float(n) ** dim
    keep = [(i, a, b, x) for i, (a, b) in enumerate(pairs) for x in range(b + 1) if ntri[i, x] > 0]
    norm = (box / ng) ** (3 * dim) / box ** dim
    num = np.array([sums[i, x] for i, _, _, x in keep])
    tri = np.array([ntri[i, x] for i, _, _, x in keep])
    return [(a, b, x) for _, a, b, x in keep], norm * num / tri, num, tri, norm, fields, n


def _kbar(q, dim):
    top = math.isqrt(q[-1] - 1)
    m = np.arange(-top, top + 1, dtype=np.int64) ** 2
    cnt = np.bincount(m, minlength=q[-1])[:q[-1]]
    one = cnt
    for _ in range(dim - 1):
        cnt = np.rint(np.fft.irfft(np.fft.rfft(cnt, 2 * q[-1]) * np.fft.rfft(one, 2 * q[-1]), 2 * q[-1]))[:q[-1]]
    k = np.sqrt(np.arange(q[-1]))
    return [float((cnt[q[i]:q[i + 1]] * k[q[i]:q[i + 1]]).sum() / cnt[q[i]:q[i + 1]].sum()) for i in range(len(q) - 1)]


def _grid(c, edges, bins, num, tri, norm):
    """Merged (mu, t) cells per k1 shell; NaN where no bin falls."""
    k = _kbar(_geometry(edges)[0], c["dim"])
    top, den = np.zeros((c["ns"], c["n_mu"], c["n_t"])), np.zeros((c["ns"], c["n_mu"], c["n_t"]))
    for (a, b, x), s, t in zip(bins, num, tri):
        mu = 0.5 * (k[a] / k[b] + k[b] / k[a] - (k[x] / k[a]) * (k[x] / k[b]))
        i = min(int((min(max(mu, 0.5), 1.0) - 0.5) * (2.0 * c["n_mu"])), c["n_mu"] - 1)
        j = min(int((min(max(k[b] / k[a], 0.5), 1.0) - 0.5) * (2.0 * c["n_t"])), c["n_t"] - 1)
        top[a, i, j] += s
        den[a, i, j] += t
    with np.errstate(invalid="ignore"):
        return np.where(den > 0, norm * top / np.where(den > 0, den, 1.0), np.nan)


def exact(case, seed):
    c = case
    if c["kind"] == "batch":
        return [_bins(c, ng, float(ng), _edges(c, ng), _spec(ng, float(ng), c, 1000 * seed + i))[1]
                for i, ng in enumerate(_batch_grids(c))]
    ng, box, edges = c["ng"], c["box"], _edges(c)
    if c["kind"] == "grad":
        return _exact_grad(c, ng, box, edges, seed)
    spec = _spec(ng, box, c, seed, c["dim"])
    if c["kind"] == "fields":
        n = _fields_grid(c)
        return _shells(c, ng, edges, spec, n).reshape((c["ns"],) + (n,) * 3)
    bins, b, num, tri, norm, _, _ = _bins(c, ng, box, edges, spec)
    return b, _grid(c, edges, bins, num, tri, norm)


def _exact_grad(c, ng, box, edges, seed):
    """Bins and d loss / d delta: the pair products back through the masked transforms."""
    delta = _field(ng, box, c, seed).float().double().requires_grad_()
    spec = torch.fft.rfftn(delta)
    bins, b, _, tri, norm, fields, n = _bins(c, ng, box, edges, spec.detach())
    k = _kbar(_geometry(edges)[0], 3)
    ana = _analytic(c, [[k[x[i]] for x in bins] for i in range(3)])
    g = 2 * (b - ana) / ana ** 2 * norm / tri / float(n) ** 3
    where = {}
    for t, x in enumerate(bins):
        for i in range(3):
            o = tuple(x[:i] + x[i + 1:])
            where.setdefault(o, np.zeros(c["ns"]))[x[i]] += g[t]
    a = torch.tensor([o[0] for o in where], device="cuda")
    d = torch.tensor([o[1] for o in where], device="cuda")
    w = torch.from_numpy(np.stack(list(where.values()))).cuda()
    back = torch.empty_like(fields)
    step = max(1, (1 << 27) // len(where))
    for v in range(0, fields.shape[1], step):
        f = fields[:, v:v + step]
        back[:, v:v + step] = w.T @ (f[a] * f[d])
    leaf = spec.detach().requires_grad_()
    r = _geometry(edges)[1][-1]
    q = _geometry(edges)[0]
    total = torch.zeros_like(spec.detach())
    for i in range(c["ns"]):
        part, m2, z2 = _box(leaf, ng, r, 3)
        part = part * ((m2 >= q[i]) & (m2 < q[i + 1]))
        if c["beta"]:
            part = part * (1 + c["beta"] * z2 / m2.clamp(min=1))
        total += torch.autograd.grad(_to_grid(part, n, r, 3), leaf, back[i].reshape((n,) * 3))[0]
    grad, = torch.autograd.grad(spec, delta, total)
    return b, grad
