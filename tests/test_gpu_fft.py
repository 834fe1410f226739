"""The pruned FFT passes (Algorithm 2.4 steps 2-3, Algorithm 2.1 steps 1-2) at every line length:
the stages' radices (8s, then 4s) and the block's lines per length differ from size to size."""
import numpy as np
import pytest

import inputs
from oracle import nfft as NF
from oracle import windows as W
from tests.gpu_util import lib_or_skip, rel, to_dev

pytestmark = pytest.mark.gpu

SIZES = [4, 8, 16, 32, 64, 128, 256, 512, 1024, 2048, 4096]


def _m(n):
    return min(4, n // 2 - 1)


@pytest.mark.parametrize("n", SIZES)
@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("A,B,nblk", [(3, 1, 1), (1, 5, 2), (2, 37, 1)])
def test_fft_axis_every_length(n, prec, A, B, nblk):
    """infft_fft_axis against numpy's float64 FFT.  With u the unit roundoff a radix-2^k FFT with
    correctly rounded twiddles is within 8 u log2(n) of the whole transform in the 2-norm (a stage
    of k levels rounds a product once and k sums; eight covers the product's two and the sums'
    k <= 3); the deconvolution adds 2 u of each entry, so both sides are compared before it."""
    L, torch = lib_or_skip()
    M, m = n // 2, _m(n)
    p = L.Plan(inputs.random_points(10, 1, 1), M, 2.0, m, prec)
    g = inputs.rng(2 * n + B)
    x = g.uniform(-1, 1, (A, n, B)) + 1j * g.uniform(-1, 1, (A, n, B))
    cd = torch.complex64 if prec == "fp32" else torch.complex128
    xd = to_dev(torch, x, cd)
    out = torch.empty(A * M * B, dtype=cd, device="cuda")
    st = L.load().infft_fft_axis(p.handle, L.MODE_PLAIN, A, B, nblk, xd.data_ptr(), out.data_ptr(),
                                 torch.cuda.current_stream().cuda_stream)
    assert st == L.OK
    h = out.cpu().numpy().astype(np.complex128).reshape(nblk, A, M // nblk, B).transpose(1, 0, 2, 3).reshape(A, M, B)
    full = np.fft.fft(xd.cpu().numpy().astype(np.complex128), axis=1)
    k = np.arange(-M // 2, M // 2)
    dinv = 1.0 / (n * W.what(W.KB, k[:, None], M, n, m).ravel())
    off = np.linalg.norm(h / dinv[None, :, None] - full[:, k % n, :])
    u = 2.0 ** -24 if prec == "fp32" else 2.0 ** -53
    # (the window's transform itself is evaluated to a few ulps of float64 on either side)
    assert off <= (8 * np.log2(n) + 2) * u * np.linalg.norm(full) + 64 * 2.0 ** -53 * np.linalg.norm(full)


@pytest.mark.parametrize("n", SIZES)
def test_forward_every_length(n):
    """The zero-padded inverse passes through the forward NFFT in float64 (the bound of the other
    comparisons with the oracle's Algorithm 2.1)."""
    L, torch = lib_or_skip()
    M, m = n // 2, _m(n)
    x = inputs.random_points(200, 1, 3)
    fh = inputs.coeffs_complex((M,), 4)
    p = L.Plan(x, M, 2.0, m, "fp64")
    assert rel(p.forward(to_dev(torch, fh)).cpu().numpy(), NF.nfft(x, fh, M, 2.0, m)) < 1e-12
