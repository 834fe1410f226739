"""The float32 d = 3 spread on the tensor cores (m <= 4): grids against the float64 spread."""
import numpy as np
import pytest

import inputs
from tests.gpu_util import lib_or_skip, to_dev

pytestmark = pytest.mark.gpu
U = 2.0 ** -24


def _grid(L, torch, p, f):
    g = torch.empty((p.Ms,) * 3, dtype=torch.complex64 if p.precision == "fp32" else torch.complex128, device="cuda")
    st = L.load().infft_spread_grid(p.handle, L.MODE_PLAIN, f.data_ptr(), g.data_ptr(),
                                    torch.cuda.current_stream().cuda_stream)
    assert st == L.OK
    return g.cpu().numpy().astype(np.complex128)


@pytest.mark.parametrize("m", [1, 2, 3, 4])
@pytest.mark.parametrize("gen,N", [("random", 1), ("random", 65), ("random", 4001), ("layer", 700), ("nodes", 1000)])
@pytest.mark.parametrize("window", ["kb", "bspline"])
def test_grid_matches_float64(m, gen, N, window):
    """Largest error of a cell against the largest cell of the sum of absolute contributions.  Per
    contribution: two factors split to 2^-22 each, a sample, three taps with at most 16 u of the
    window's maximum each and their product, per group of 8 points two sums; a cell meets at most N points:
    (2 * 4 + 4 * 16 + N / 4) u with u = 2^-24.  "layer": chunks of 64 points in one plane of cells."""
    L, torch = lib_or_skip()
    M = 16
    x = inputs.random_points(N, 3, 80 + m)
    if gen == "layer":
        x[:, 0] = 0.25 + 1e-3
        x[:, 1:] *= 0.2
    if gen == "nodes":
        x = np.round(x * 2 * M) / (2 * M)
        x[::3] += 1e-9
    f = inputs.samples_complex(N, 81)
    p = L.Plan(x, M, 2.0, m, "fp32", window=window)
    q = L.Plan(x, M, 2.0, m, "fp64", window=window)
    f32 = to_dev(torch, f, torch.complex64)
    g, G = _grid(L, torch, p, f32), _grid(L, torch, q, f32.to(torch.complex128))
    S = _grid(L, torch, q, f32.abs().to(torch.complex128))
    assert np.max(np.abs(g - G)) <= (8 + 64 + N / 4) * U * np.max(np.abs(S))
