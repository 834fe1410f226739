"""The float32 spreads on the tensor cores (Algorithm 2.4 step 1) cell by cell: bounds that count the points a
cell meets, samples that are not finite, and the forms of the batched d = 2 adjoint that share the spread."""
import numpy as np
import pytest

import inputs
from oracle import nfft as NF
from tests.gpu_util import lib_or_skip, rel, to_dev

pytestmark = pytest.mark.gpu
U = 2.0 ** -24


def _grid(L, torch, p, f):
    g = torch.empty((p.Ms,) * p.d, dtype=torch.complex64 if p.precision == "fp32" else torch.complex128, device="cuda")
    st = L.load().infft_spread_grid(p.handle, L.MODE_PLAIN, f.data_ptr(), g.data_ptr(),
                                    torch.cuda.current_stream().cuda_stream)
    assert st == L.OK
    return g.cpu().numpy().astype(np.complex128)


def _meets(x, Ms, m):
    """The most points whose 2m + 1 taps along every axis reach one cell."""
    base = np.floor(Ms * (x - np.floor(x + 0.5))).astype(int) % Ms
    count = np.zeros((Ms,) * x.shape[1], int)
    np.add.at(count, tuple(base.T), 1)
    for a in range(x.shape[1]):
        count = sum(np.roll(count, s, axis=a) for s in range(-m, m + 1))
    return int(count.max())


@pytest.mark.parametrize("d,M,N,m", [(2, 32, 3001, 2), (2, 32, 3001, 4), (2, 32, 3001, 8), (2, 32, 300, 4),
                                     (3, 16, 4001, 1), (3, 16, 4001, 2), (3, 16, 4001, 4), (3, 16, 300, 4)])
@pytest.mark.parametrize("window", ["kb", "bspline"])
def test_error_by_the_points_a_cell_meets(d, M, N, m, window):
    """Per contribution: two factors split to 2^-22 each (8 u), and a sample and d taps with at most 16 u of the
    window's maximum each; per group of 8 points two sums.  Largest error of a cell against the largest sum of absolute
    contributions: (8 + 16 (d + 1) + n / 4) u, n the most points that meet a cell."""
    L, torch = lib_or_skip()
    x = inputs.random_points(N, d, 30 + m)
    f32 = to_dev(torch, inputs.samples_complex(N, 31), torch.complex64)
    p, q = (L.Plan(x, M, 2.0, m, prec, window=window) for prec in ("fp32", "fp64"))
    g, G = _grid(L, torch, p, f32), _grid(L, torch, q, f32.to(torch.complex128))
    S = _grid(L, torch, q, f32.abs().to(torch.complex128))
    n = _meets(x, 2 * M, m)
    assert n < N / 2
    assert np.max(np.abs(g - G)) <= (8 + 16 * (d + 1) + n / 4) * U * np.max(np.abs(S))


@pytest.mark.parametrize("d,M,m", [(2, 32, 4), (2, 32, 8), (3, 16, 4)])
@pytest.mark.parametrize("value", [float("nan"), float("inf"), -float("inf")])
def test_sample_that_is_not_finite(d, M, m, value):
    """It reaches every coefficient of its own transform, no cell beyond its tile's padded edge, and no other job of a
    batch."""
    L, torch = lib_or_skip()
    N = 900
    x = inputs.random_points(N, d, 40)
    x[17] = 0.01     # base cell just past the middle
    f = inputs.samples_complex(N, 41)
    bad = f.copy()
    bad[17] = complex(value, 1.0)
    p, q = L.Plan(x, M, 2.0, m, "fp32"), L.Plan(x, M, 2.0, m, "fp32")
    fd, bd = to_dev(torch, f, torch.complex64), to_dev(torch, bad, torch.complex64)
    good = p.adjoint(fd).cpu().numpy()
    hs = [torch.empty((M,) * d, dtype=torch.complex64, device="cuda") for _ in range(2)]
    L.adjoint_batched([p, q], [bd, fd], hs, L.MODE_PLAIN)
    assert not np.isfinite(hs[0].cpu().numpy()).any()
    assert np.array_equal(hs[1].cpu().numpy(), good)
    g, clean = _grid(L, torch, p, bd), _grid(L, torch, p, fd)
    T = 16 if d == 2 else 8
    cells = [np.arange(-m, T + m) % (2 * M)] * d   # the tile of base cells 0 .. T - 1 and its padding
    inside = np.zeros(g.shape, bool)
    inside[np.ix_(*cells)] = True
    assert np.array_equal(g[~inside], clean[~inside])
    assert not np.isfinite(g[(0,) * d])


def test_persistent_and_staged_forms_share_the_spread(monkeypatch):
    """INFFT_SPREAD2D_PREFETCH=0 keeps a batch off the persistent kernel: two launches with it, the staged kernels'
    without, the same bits from both, and the oracle's Algorithm 2.4."""
    L, torch = lib_or_skip()
    specs = [(32, 4000), (64, 9001)]
    plans, fs = [], []
    for i, (M, N) in enumerate(specs):
        plans.append(L.Plan(inputs.random_points(N, 2, 45 + i), M, 2.0, 4, "fp32"))
        fs.append(to_dev(torch, inputs.samples_complex(N, 47 + i), torch.complex64))
    monkeypatch.setenv("INFFT_PERSISTENT", "1")
    out, launches = {}, {}
    for form in ("0", "1"):
        monkeypatch.setenv("INFFT_SPREAD2D_PREFETCH", form)
        hs = [torch.empty((M, M), dtype=torch.complex64, device="cuda") for M, _ in specs]
        L.launch_count_reset()
        L.adjoint_batched(plans, fs, hs, L.MODE_PLAIN)
        launches[form] = L.launch_count()
        out[form] = [h.cpu().numpy() for h in hs]
    assert launches["1"] == 2 and launches["0"] == 3
    for a, b in zip(out["0"], out["1"]):
        assert np.array_equal(a, b)
    M, N = specs[1]
    ref = NF.adjoint_nfft(inputs.random_points(N, 2, 46), inputs.samples_complex(N, 48), M, 2.0, 4)
    assert rel(out["1"][1].ravel(), ref) < 1e-5
