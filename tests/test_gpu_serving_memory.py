"""The serving loop's admission estimate covers the device memory that building a point set takes."""
import pytest

import inputs
from tests.gpu_util import lib_or_skip

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,M,N,precision", [
    (2, 64, 20000, "fp32"), (2, 64, 20000, "fp64"), (2, 64, 400000, "fp32"), (2, 64, 400000, "fp64"), (2, 32, 500, "fp64"),
    (2, 128, 100000, "fp32"), (3, 16, 40000, "fp32"), (3, 16, 40000, "fp64"), (3, 16, 2000, "fp32"), (1, 64, 5000, "fp64"),
])
def test_estimate_covers_the_build(d, M, N, precision):
    """At its peak a build holds the plan with its weights, the degree-2M float64 plan of the CG (whose bytes a
    plan of the same points tells), and the CG's vectors: six of the larger of N and (2M)^d, one of either."""
    L, torch = lib_or_skip()
    from paper_2302_00414_gb300.serve import Backend, PointSet
    be = Backend(weights_iters=1)
    ps = PointSet(0, d, M, inputs.random_points(N, d, 3), precision)
    p = be.build_plan(ps, torch.cuda.current_stream())
    sub = L.Plan(ps.x, 2 * M, 2.0, 8 if d <= 2 else 4, "fp64")
    K = (2 * M) ** d
    held = p.device_bytes + sub.device_bytes + 16 * (6 * max(N, K) + N + K)
    est = be.estimate_bytes(ps)
    assert est >= held
    assert est <= 4 * held      # and does not turn sets away for memory they do not take
    be.release(p)
    sub.close()
