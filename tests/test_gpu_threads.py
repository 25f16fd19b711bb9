"""Two host threads drive a plan each, on streams of their own, with blocks of unequal shared memory.

A kernel's shared-memory limit belongs to the process. Launches that set the plan's own size were refused
when the other thread had lowered it in between: 18 of 4000 calls, for the FP32 contraction as for the
generic passes.
"""
import threading

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("call,prec,shapes,count", [
    ("contract", "fp32", ((32, 2, 8.0), (64, 12, 16.0)), 4000),
    ("estimate", "fp64", ((32, 2, 8.0), (54, 4, 17.0)), 4000),
    ("grad", "fp32", ((128, 9, 32.0), (128, 16, 32.0)), 300),
])
def test_plans_of_two_threads(call, prec, shapes, count):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2107_14564_gb300 import binding
    gen = torch.Generator(device="cuda").manual_seed(1)
    jobs = []
    for ng, ns, top in shapes:
        plan = binding.Plan(ng, float(ng), np.linspace(1.0, top, ns + 1), precision=prec)
        out = torch.empty(plan.n_triplets, dtype=torch.float64, device="cuda")
        spec = torch.randn(plan.spec_shape(), dtype=plan.complex_dtype, device="cuda", generator=gen)
        if call == "contract":
            args = (binding.bsp_contract, plan.shell_fields(spec), out)
        elif call == "estimate":
            args = (binding.bsp_estimate, spec, out, None)
        else:
            out = torch.empty((ng,) * 3, dtype=torch.float32, device="cuda")
            args = (binding.bsp_grad, spec, torch.ones(plan.n_triplets, dtype=torch.float64, device="cuda"), out)
        stream = torch.cuda.Stream()
        args[0](plan.handle, *args[1:])
        torch.cuda.synchronize()
        jobs.append((plan, args, out, out.clone(), stream))
        out.zero_()
    torch.cuda.synchronize()
    start = threading.Barrier(len(jobs))
    refused = []

    def drive(plan, args, stream):
        start.wait()
        for _ in range(count):
            try:
                args[0](plan.handle, *args[1:], stream.cuda_stream)
            except binding.BispecError as e:
                refused.append(str(e))

    threads = [threading.Thread(target=drive, args=(j[0], j[1], j[4])) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not refused, (len(refused), refused[0])
    for plan, _, out, want, _ in jobs:
        assert torch.equal(out, want)
        plan.close()
