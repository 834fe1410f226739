"""The forms of the d = 2 adjoint's FFT passes (Algorithm 2.4 steps 2 and 3) carry the deconvolution factors
and twiddles to the same precision."""
import math

import numpy as np
import pytest

import inputs
from tests.gpu_util import lib_or_skip

pytestmark = pytest.mark.gpu
U = 2.0 ** -24


@pytest.mark.parametrize("form", ["0", "1"])
@pytest.mark.parametrize("M", [32, 64, 256])
def test_gain_of_the_bins(M, form, monkeypatch):
    """The gain of an output bin, averaged over sample vectors, is its systematic error: a deconvolution factor
    rounded to float32 is off by 2.4e-8 (u / sqrt 6, per axis, another in every bin), 3.4e-8 for two axes.
    With the factors and twiddles to twice the precision what is left is the average of the roundings, 1e-7 over
    sqrt(2 * 160) or 6e-9, and a few 1e-9 of products rounded before the low part is added: the gains scatter
    by less than u / 3 = 2e-8 around their mean."""
    L, torch = lib_or_skip()
    monkeypatch.setenv("INFFT_FUSED_MERGE_FFT", form)
    N, K, m = 2000, 160, 4
    x = inputs.random_points(N, 2, 90)
    p, q = L.Plan(x, M, 2.0, m, "fp32"), L.Plan(x, M, 2.0, m, "fp64")
    gen = torch.Generator(device="cuda")
    gen.manual_seed(91)
    num = torch.zeros((M, M), dtype=torch.float64, device="cuda")
    den = torch.zeros_like(num)
    for _ in range(K):
        f = torch.randn(N, dtype=torch.complex64, device="cuda", generator=gen)
        a, b = p.adjoint(f).to(torch.complex128), q.adjoint(f.to(torch.complex128))
        num += (b.conj() * a).real
        den += b.abs() ** 2
    gain = (num / den).cpu().numpy()
    assert np.isfinite(gain).all()
    assert math.sqrt(((gain - gain.mean()) ** 2).mean()) < U / 3


@pytest.mark.parametrize("order", [(24, 32, 28), (32, 24, 28)])
def test_fused_batch_of_degrees_on_one_grid(order, monkeypatch):
    """Jobs of one grid size and different degrees share a launch of the fused kernel: each has the shared memory of
    the largest layout, and the result of its own call bit for bit."""
    L, torch = lib_or_skip()
    monkeypatch.setenv("INFFT_FUSED_MERGE_FFT", "1")
    plans, fs, hs, alone = [], [], [], []
    for i, M in enumerate(order):
        plans.append(L.Plan(inputs.random_points(900 + i, 2, 92 + i), M, 63.5 / M, 4, "fp32"))
        fs.append(torch.from_numpy(inputs.samples_complex(900 + i, 95 + i)).to("cuda", torch.complex64))
        hs.append(torch.empty((M, M), dtype=torch.complex64, device="cuda"))
        alone.append(plans[-1].adjoint(fs[-1]).cpu().numpy())
    assert {p.Ms for p in plans} == {64}
    L.adjoint_batched(plans, fs, hs, L.MODE_PLAIN)
    for h, a in zip(hs, alone):
        assert np.array_equal(h.cpu().numpy(), a)
