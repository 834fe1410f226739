"""Interpolation (Algorithm 2.1 step 3) at every window width, and with B_opt (Remark 4.6): item and chunk
edges of the kernels that put the lanes of a warp on one point's cells."""
import numpy as np
import pytest

import inputs
from oracle import nfft as NF
from tests.gpu_util import lib_or_skip, rel, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,m", [(2, k) for k in range(1, 9)] + [(3, k) for k in range(1, 7)])
@pytest.mark.parametrize("N", [1, 5, 131, 2500])
def test_forward_fp32_every_width(d, m, N):
    """Float32 against the oracle's Algorithm 2.1 at the bound of the other float32 comparisons."""
    L, torch = lib_or_skip()
    M = 16
    x = inputs.random_points(N, d, 60 + m)
    x[::7] = np.round(x[::7] * 2 * M) / (2 * M)     # some on grid nodes (2m + 1 taps)
    fh = inputs.coeffs_complex((M,) * d, 61)
    p = L.Plan(x, M, 2.0, m, "fp32")
    out = p.forward(to_dev(torch, fh, torch.complex64)).cpu().numpy()
    assert rel(out, NF.nfft(x, fh, M, 2.0, m)) < 1e-5


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("m", [2, 4, 7])
@pytest.mark.parametrize("N", [1, 30, 1300])
def test_stored_coefficients_both_ways(prec, m, N):
    """Algorithm 4.4 and Remark 4.6 with given coefficients are adjoint to one another:
    <B_opt F D h, f> = <h, D F^* B_opt^* f>, and the first matches a direct evaluation, both within
    float rounding of the sums ((2m + 2)^2 products and the FFT: 1e-5, 1e-12)."""
    L, torch = lib_or_skip()
    from oracle import windows as W
    M, S = 16, 2 * m + 2
    Ms = 2 * M
    x = inputs.random_points(N, 2, 62)
    b = inputs.coeffs_complex((N, S, S), 63)
    cd = torch.complex64 if prec == "fp32" else torch.complex128
    tol = 1e-5 if prec == "fp32" else 1e-12
    p = L.Plan(x, M, 2.0, m, prec)
    p.set_bopt(b)
    h = inputs.coeffs_complex((M, M), 64)
    f = inputs.samples_complex(N, 65)
    out = p.inverse_adjoint(to_dev(torch, h, cd)).cpu().numpy().astype(np.complex128)
    back = p.adjoint(to_dev(torch, f, cd), mode=L.MODE_BOPT).cpu().numpy().astype(np.complex128)
    k = np.arange(-M // 2, M // 2)
    dinv = 1.0 / (Ms * W.what(W.KB, k[:, None], M, Ms, m).ravel())
    gh = np.zeros((Ms, Ms), dtype=complex)
    gh[np.ix_(k % Ms, k % Ms)] = h * dinv[:, None] * dinv[None, :]
    g = np.fft.ifft2(gh) * Ms * Ms
    cell = np.floor(Ms * (x - np.floor(x + 0.5))).astype(int)
    s = np.arange(S) - m
    ref = np.array([np.sum(b[j] * g[np.ix_((cell[j, 0] + s) % Ms, (cell[j, 1] + s) % Ms)]) for j in range(N)])
    assert rel(out, ref) < tol
    lhs, rhs = np.vdot(f, out), np.vdot(back, h)
    assert abs(lhs - rhs) <= tol * np.linalg.norm(f) * np.linalg.norm(out) + tol * np.linalg.norm(back) * np.linalg.norm(h)
