"""The B-spline window's taps on the GPU (eq. window_bspline): their values, and what they cost beside the
Kaiser-Bessel window's."""
import math
from fractions import Fraction

import numpy as np
import pytest

import inputs
from tests.gpu_util import lib_or_skip, to_dev

pytestmark = pytest.mark.gpu


def _bspline(y, n):
    """The centred cardinal B-spline of order n at y by truncated powers, in exact rational arithmetic (in floating
    point that form loses five digits at order 16)."""
    z = [Fraction(y) + Fraction(n, 2) - k for k in range(n + 1)]
    return float(sum((-1) ** k * math.comb(n, k) * t ** (n - 1) for k, t in enumerate(z) if t > 0) / math.factorial(n - 1))


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("d,m", [(1, 1), (1, 5), (1, 8), (2, 1), (2, 2), (2, 4), (2, 7), (2, 8), (3, 1), (3, 2), (3, 4), (3, 6)])
def test_taps_of_one_point(d, m, prec):
    """One sample of 1 spreads to the product of its taps.  The recursion adds positive terms: three roundings an order,
    2m orders, so 6 m u relative per axis; the float32 tensor-core products add 24 u of the largest value."""
    L, torch = lib_or_skip()
    u = 2.0 ** -24 if prec == "fp32" else 2.0 ** -53
    M, Ms = 16, 32
    cd = torch.complex64 if prec == "fp32" else torch.complex128
    for off in (0.0, 0.25, 0.9375):     # on a node, inside, near the next one: exact in both precisions
        x = np.full((1, d), (5 + off) / Ms)
        p = L.Plan(x, M, 2.0, m, prec, window="bspline")
        f = torch.ones(1, dtype=cd, device="cuda")
        g = torch.empty((Ms,) * d, dtype=cd, device="cuda")
        st = L.load().infft_spread_grid(p.handle, L.MODE_PLAIN, f.data_ptr(), g.data_ptr(),
                                        torch.cuda.current_stream().cuda_stream)
        assert st == L.OK
        delta = [(5 + off - c + Ms / 2) % Ms - Ms / 2 for c in range(Ms)]   # the grid is periodic
        axis = np.array([_bspline(v, 2 * m) if abs(v) < m else 0.0 for v in delta])
        ref = axis
        for _ in range(d - 1):
            ref = np.multiply.outer(ref, axis)
        assert np.max(np.abs(g.cpu().numpy().astype(np.complex128) - ref)) <= (6 * m * d + 24) * u * ref.max()


@pytest.mark.parametrize("d,M,N,m", [(2, 32, 300, 4), (2, 32, 300, 7), (2, 128, 2000, 7), (3, 32, 3000, 2), (3, 32, 3000, 4),
                                     (3, 64, 20000, 4)])
@pytest.mark.parametrize("direction", ["adjoint", "forward"])
def test_cost_beside_kaiser_bessel(d, M, N, m, direction):
    """Sparse sets, where evaluating the taps is a large part: a point's taps take about m multiply-adds each from the
    recursion and eleven from the Kaiser-Bessel polynomials, so the call takes at most twice as long."""
    L, torch = lib_or_skip()
    x = inputs.random_points(N, d, 12)
    f = to_dev(torch, inputs.samples_complex(N, 13), torch.complex64)
    h = torch.zeros((M,) * d, dtype=torch.complex64, device="cuda")
    best = {}
    for window in ("kb", "bspline"):
        p = L.Plan(x, M, 2.0, m, "fp32", window=window)
        call = (lambda: p.adjoint(f, h)) if direction == "adjoint" else (lambda: p.forward(h, f))
        for _ in range(5):
            call()
        times = []
        for _ in range(7):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(20):
                call()
            b.record()
            torch.cuda.synchronize()
            times.append(a.elapsed_time(b))
        best[window] = min(times)
    assert best["bspline"] <= 2 * best["kb"]
