"""Creating an FP32 plan of many shells takes about as long as an FP64 plan of the same bins.

Both count the bins' triangles in FP64, which is most of the time; FP32 adds the grouping of its tiles into
blocks, which at 128 rings once took longer than all the rest (1008 ms against 430).
"""
import time

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_many_ring_plan_creation():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2107_14564_gb300 import binding
    edges = np.linspace(1.0, 257.0, 129)
    took = {}
    for prec in ("fp64", "fp32"):
        times = []
        for _ in range(4):  # the first one loads the kernels
            t = time.perf_counter()
            plan = binding.Plan(1024, 1024.0, edges, precision=prec, dim=2)
            times.append(time.perf_counter() - t)
            plan.close()
        took[prec] = min(times[1:])
    assert took["fp32"] < 1.5 * took["fp64"], took
