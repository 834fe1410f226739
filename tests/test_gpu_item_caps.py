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
