"""Calls from several host threads, each with its own plan and stream: a kernel's shared-memory limit is one
per process, so no thread's launch may depend on another's."""
import threading

import numpy as np
import pytest

import inputs
from tests.gpu_util import lib_or_skip, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,sizes", [(1, (16, 2048, 256)), (2, (16, 256, 64)), (3, (8, 32, 16))])
def test_threads_with_plans_of_different_sizes(d, sizes):
    """Adjoint and forward calls of small and large grids from as many threads: no call fails, and every result is the one
    of the plan called alone, bit for bit."""
    L, torch = lib_or_skip()
    work = []
    for i, M in enumerate(sizes):
        p = L.Plan(inputs.random_points(300, d, 10 + i), M, 2.0, 3, "fp64")
        f = to_dev(torch, inputs.samples_complex(300, 20 + i), torch.complex128)
        work.append((p, f, p.adjoint(f).clone(), torch.cuda.Stream()))
    torch.cuda.synchronize()
    errors, start = [], threading.Barrier(len(work))

    def run(p, f, want, stream):
        try:
            h, g = torch.empty_like(want), torch.empty_like(f)
            start.wait()
            for _ in range(3000 if d < 3 else 1000):
                p.adjoint(f, h, stream=stream.cuda_stream)
                p.forward(h, g, stream=stream.cuda_stream)
            stream.synchronize()
            if not torch.equal(h, want):
                errors.append("result differs")
        except Exception as e:   # reported by the main thread
            errors.append(repr(e))

    threads = [threading.Thread(target=run, args=w) for w in work]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert errors == []
    assert np.isfinite(work[0][2].cpu().numpy()).all()
