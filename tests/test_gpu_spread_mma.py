"""The float32 d = 2 spread on the tensor cores (Algorithm 2.4 step 1): its grids against the
float64 spread of the same points, at the edges of its bands, column windows and groups."""
import numpy as np
import pytest

import inputs
from tests.gpu_util import lib_or_skip, rel, to_dev

pytestmark = pytest.mark.gpu
U = 2.0 ** -24


def _grid(L, torch, p, f):
    g = torch.empty((p.Ms, p.Ms), dtype=torch.complex64 if p.precision == "fp32" else torch.complex128, device="cuda")
    st = L.load().infft_spread_grid(p.handle, L.MODE_PLAIN, f.data_ptr(), g.data_ptr(),
                                    torch.cuda.current_stream().cuda_stream)
    assert st == L.OK
    return g.cpu().numpy().astype(np.complex128)


def _points(gen, N, Ms, seed):
    x = inputs.random_points(N, 2, seed)
    if gen == "nodes":      # on grid nodes (2m + 1 taps) and just off them
        x = np.round(x * Ms) / Ms
        x[::3] += 1e-9
    if gen == "corners":    # first and last rows and columns of the tiles' bands and windows
        edge = np.array([0, 7, 8, 15])
        r = inputs.rng(seed + 1)
        cell = 16 * r.integers(0, Ms // 16, (N, 2)) + edge[r.integers(0, 4, (N, 2))]
        x = (cell + r.uniform(0.01, 0.99, (N, 2))) / Ms - 0.5
    return x


@pytest.mark.parametrize("m", [2, 3, 4, 5, 6, 7, 8])
@pytest.mark.parametrize("gen,N", [("random", 1), ("random", 33), ("random", 3001), ("nodes", 700), ("corners", 1500)])
@pytest.mark.parametrize("window", ["kb", "bspline"])
def test_grid_matches_float64(m, gen, N, window):
    """Largest error of a cell against the largest cell of the sum of absolute contributions.  Per
    contribution: two factors split to 2^-22 each, a sample and two taps with at most 16 u of the
    window's maximum each (polynomial or recursion), per group of 8 points two sums; a cell meets at
    most N points.  With u = 2^-24: (2 * 4 + 3 * 16 + N / 4) u."""
    L, torch = lib_or_skip()
    M = 32
    x = _points(gen, N, 2 * M, 70 + m)
    f = inputs.samples_complex(N, 71)
    p = L.Plan(x, M, 2.0, m, "fp32", window=window)
    q = L.Plan(x, M, 2.0, m, "fp64", window=window)
    f32 = to_dev(torch, f, torch.complex64)
    g = _grid(L, torch, p, f32)
    G = _grid(L, torch, q, f32.to(torch.complex128))
    S = _grid(L, torch, q, f32.abs().to(torch.complex128))
    assert np.max(np.abs(g - G)) <= (8 + 48 + N / 4) * U * np.max(np.abs(S))


@pytest.mark.parametrize("e", [-60, 60])
def test_scaled_samples_scale_the_grid(e):
    """Powers of two pass through exactly (the samples are brought to float16's range per chunk)."""
    L, torch = lib_or_skip()
    x = inputs.random_points(2000, 2, 5)
    f = to_dev(torch, inputs.samples_complex(2000, 6), torch.complex64)
    p = L.Plan(x, 32, 2.0, 4, "fp32")
    assert np.array_equal(_grid(L, torch, p, f * 2.0 ** e), _grid(L, torch, p, f) * 2.0 ** e)


def test_wide_range_of_samples():
    """Samples over 30 orders of magnitude: the error is bounded by the largest contributions."""
    L, torch = lib_or_skip()
    N = 4000
    x = inputs.random_points(N, 2, 7)
    f = inputs.samples_complex(N, 8) * 10.0 ** inputs.rng(9).uniform(-20, 10, N)
    p, q = L.Plan(x, 32, 2.0, 4, "fp32"), L.Plan(x, 32, 2.0, 4, "fp64")
    f32 = to_dev(torch, f, torch.complex64)
    g, G = _grid(L, torch, p, f32), _grid(L, torch, q, f32.to(torch.complex128))
    S = _grid(L, torch, q, f32.abs().to(torch.complex128))
    assert np.max(np.abs(g - G)) <= (8 + 48 + N / 4) * U * np.max(np.abs(S))


def test_batch_of_unlike_windows_equals_single_calls():
    """Plans of different oversampling have different window polynomials: the batch then reads them
    from shared memory and not from the parameter block, with the same results bit for bit."""
    L, torch = lib_or_skip()
    plans, fs, hs, alone = [], [], [], []
    for i, (M, sigma) in enumerate([(32, 2.0), (24, 63.5 / 24), (64, 2.0)]):
        p = L.Plan(inputs.random_points(3000 + i, 2, 20 + i), M, sigma, 4, "fp32")
        f = to_dev(torch, inputs.samples_complex(3000 + i, 30 + i), torch.complex64)
        plans.append(p)
        fs.append(f)
        hs.append(torch.empty((M, M), dtype=torch.complex64, device="cuda"))
        alone.append(p.adjoint(f).cpu().numpy())
    L.load()
    from paper_2302_00414_gb300.api import adjoint_batched
    adjoint_batched(plans, fs, hs)
    for h, a in zip(hs, alone):
        assert np.array_equal(h.cpu().numpy(), a)
