"""The default lengths of work items (float64: 128 points for d = 2, 16 for small d = 1 plans), on the GPU.

Shorter items mean more padded tiles.  A plan whose padded tiles then pass the fixed scratch of
infft_adjoint_noalloc, although those of long items do not, is still accepted there: it reconstructs from
a second list of long items.  The two lists add the same products in another order, so the results agree
to rounding: sums of at most 512 + 9 partial sums of N float64 terms, 1e-13 relative.
"""
import numpy as np
import pytest

import inputs
from tests.gpu_util import lib_or_skip, rel, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,M,N,m,items", [
    (2, 128, 300000, 8, "more"),      # 32 x 32 padded tiles: 768 items of 512 fit 32 MiB, 2,500 of 128 do not
    (2, 64, 20000, 8, "same"),        # both fit
    (1, 64, 700, 6, "same"),
    (1, 64, 20000, 6, "same"),        # past the range of 16-point items
])
def test_noalloc_accepts_plans_with_short_items(d, M, N, m, items):
    L, torch = lib_or_skip()
    from paper_2302_00414_gb300 import api
    x = inputs.random_points(N, d, 3)
    p = L.Plan(x, M, 2.0, m, "fp64")
    f = to_dev(torch, inputs.samples_complex(N, 5).astype(np.complex128))
    a = p.adjoint(f, mode=L.MODE_PLAIN).cpu().numpy().ravel()
    out = torch.empty(M ** d, dtype=torch.complex128, device="cuda")
    for _ in range(2):
        out.fill_(7.0)
        s = api.infft_adjoint_noalloc(p.handle, L.MODE_PLAIN, f.data_ptr(), out.data_ptr(),
                                      torch.cuda.current_stream().cuda_stream)
        torch.cuda.synchronize()
        assert s == 0
        b = out.cpu().numpy()
        if items == "same":
            assert np.array_equal(a, b)
        else:
            assert rel(b, a) < 1e-13


@pytest.mark.parametrize("prec,tol", [("fp64", 1e-12), ("fp32", 1e-5)])
@pytest.mark.parametrize("M,N,m,points,tune", [
    (64, 4000, 3, "random", None),            # one tile of 250 items
    (1024, 5000, 8, "random", None),          # eight tiles, past the range of 16-point items
    (64, 3001, 6, "cell", None),              # every point in two neighbouring cells, on a tile's edge
    (8, 300, 5, "random", {"item_cap": 1}),   # a window wider than half of the grid, an item per point
    (64, 2000, 4, "random", {"tile": 8, "item_cap": 3}),
])
def test_one_dimensional_merge_takes_the_items_of_a_cell(prec, tol, M, N, m, points, tune):
    """The d = 1 merge visits only the items of a tile that hold points near the cell; against the oracle's
    Algorithm 2.4 at the bounds of the other comparisons with it (float32: with exact sums of spreading)."""
    from oracle import nfft as NF
    L, torch = lib_or_skip()
    x = inputs.random_points(N, 1, 9)
    if points == "cell":
        x = x * (2.0 / (2 * M))   # offsets -1 .. 1 of cells around 0, the edge of the first and the last tile
    f = inputs.samples_complex(N, 10)
    p = L.Plan(x, M, 2.0, m, prec, tune=tune)
    h = p.adjoint(to_dev(torch, f, torch.complex64 if prec == "fp32" else torch.complex128), mode=L.MODE_PLAIN)
    assert rel(h.cpu().numpy().ravel(), NF.adjoint_nfft(x, f, M, 2.0, m).ravel()) < tol
