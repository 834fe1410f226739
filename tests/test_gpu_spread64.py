"""The float64 window polynomials and the float64 d = 2 spread (Algorithm 2.4 step 1) against the oracle."""
import numpy as np
import pytest

import inputs
from oracle import nfft as NF
from oracle import windows as W
from tests.gpu_util import lib_or_skip, rel, to_dev
from tests.test_gpu_spread_mma import _points

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m", [2, 3, 4, 5, 6, 7, 8])
@pytest.mark.parametrize("gen,N", [("random", 1), ("random", 33), ("nodes", 700), ("corners", 900)])
def test_spread_every_width(m, gen, N):
    """Algorithm 2.4 at the bound of the other float64 comparisons with the oracle."""
    L, torch = lib_or_skip()
    M = 32
    x = _points(gen, N, 2 * M, 90 + m)
    f = inputs.samples_complex(N, 91)
    w = inputs.rng(92).uniform(0.5, 1.5, N)
    p = L.Plan(x, M, 2.0, m, "fp64")
    p.set_weights(w.astype(np.complex128))
    h = p.adjoint(to_dev(torch, f), mode=L.MODE_DCF).cpu().numpy()
    assert rel(h, NF.adjoint_nfft(x, w * f, M, 2.0, m)) < 1e-12


@pytest.mark.parametrize("d", [1, 2, 3])
@pytest.mark.parametrize("M,sigma", [(16, 1.0), (16, 2.0), (10, 31.5 / 10), (8, 4.0), (4, 8.0)])
@pytest.mark.parametrize("m", [1, 4, 6])
def test_window_polynomials_any_oversampling(d, M, sigma, m):
    """The window steepens with the oversampling (beta up to 2 pi m).  Step 1 alone, since the deconvolution
    amplifies rounding by up to (I0(beta) M_sigma / 2m)^d at sigma = 1.  A tap is within 128 u of the window's
    maximum on either side (the polynomial's 22 terms; the oracle's argument beta sqrt(..), whose rounding
    counts beta <= 38 times), a cell's sum of at most N contributions within N u."""
    L, torch = lib_or_skip()
    Ms = 2 * int(np.ceil(np.ceil(sigma * M) / 2))
    if 2 * m + 2 > Ms:
        pytest.skip("the window is wider than the grid")
    N = 300
    x = inputs.random_points(N, d, 93)
    f = inputs.samples_complex(N, 94)
    p = L.Plan(x, M, sigma, m, "fp64")
    fd = to_dev(torch, f)
    g = torch.empty((Ms,) * d, dtype=torch.complex128, device="cuda")
    st = L.load().infft_spread_grid(p.handle, L.MODE_PLAIN, fd.data_ptr(), g.data_ptr(),
                                    torch.cuda.current_stream().cuda_stream)
    assert st == L.OK
    vals, cand, valid = NF.window_slot_values(W.KB, x, M, Ms, m)
    ref = np.fft.ifftshift(NF.spread(x, f, Ms, m, NF.tensor_coeffs(vals), cand, valid))
    near = NF.spread(x, np.abs(f), Ms, m, np.ones((N,) + (2 * m + 2,) * d), cand, valid)
    top = float(np.i0(np.pi * m * (2 - M / Ms))) ** d * np.max(np.abs(near))
    assert np.max(np.abs(g.cpu().numpy() - ref)) <= (2 * 128 * d + N) * 2.0 ** -53 * top
