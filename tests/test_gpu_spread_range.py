"""The float32 spreads on the tensor cores (Algorithm 2.4 step 1, d = 2 and d = 3) with samples at the
lower end of float32's range."""
import numpy as np
import pytest

import inputs
from tests.gpu_util import lib_or_skip, to_dev

pytestmark = pytest.mark.gpu
U = 2.0 ** -24


def _grid(L, torch, p, f):
    g = torch.empty((p.Ms,) * p.d, dtype=torch.complex64 if p.precision == "fp32" else torch.complex128, device="cuda")
    st = L.load().infft_spread_grid(p.handle, L.MODE_PLAIN, f.data_ptr(), g.data_ptr(),
                                    torch.cuda.current_stream().cuda_stream)
    assert st == L.OK
    return g.cpu().numpy().astype(np.complex128)


@pytest.mark.parametrize("d,m", [(2, 2), (2, 4), (2, 8), (3, 1), (3, 2), (3, 4)])
@pytest.mark.parametrize("window", ["kb", "bspline"])
@pytest.mark.parametrize("e", [100, 112, 118, 123])
def test_small_samples_keep_their_bits(d, m, window, e):
    """Samples of 2^-e and below (all normal numbers from 2^-125 on) against the float64 spread: the
    bound of samples of order one, (8 + 64 + N / 4) u of the largest sum of absolute contributions, and half
    a unit of float32's last place, 2^-150, for each of at most N groups and roundings of a cell."""
    L, torch = lib_or_skip()
    N, M = 600, 16
    x = inputs.random_points(N, d, 50 + m)
    f = inputs.samples_complex(N, 51) * 2.0 ** -e
    p = L.Plan(x, M, 2.0, m, "fp32", window=window)
    q = L.Plan(x, M, 2.0, m, "fp64", window=window)
    f32 = to_dev(torch, f, torch.complex64)
    g = _grid(L, torch, p, f32)
    G = _grid(L, torch, q, f32.to(torch.complex128))
    S = _grid(L, torch, q, torch.complex(f32.real.abs().double() + f32.imag.abs().double(),
                                         torch.zeros(N, dtype=torch.float64, device="cuda")))
    # the window of a cell's points is small: a few dozen of the N points meet it, but the bound takes all
    assert np.max(np.abs(g - G)) <= (8 + 64 + N / 4) * U * np.max(np.abs(S)) + 2 * N * 2.0 ** -150
    # and relative to the largest cell as close as the same samples of order one, within a factor of two
    one = to_dev(torch, inputs.samples_complex(N, 51), torch.complex64)
    g1, G1 = _grid(L, torch, p, one), _grid(L, torch, q, one.to(torch.complex128))
    err1 = np.max(np.abs(g1 - G1)) / np.max(np.abs(G1))
    assert np.max(np.abs(g - G)) <= 2 * err1 * np.max(np.abs(G)) + 2 * N * 2.0 ** -150
