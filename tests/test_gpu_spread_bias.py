"""The tensor cores truncate their sums: the float32 spreads (Algorithm 2.4 step 1) must not come out small, on
sets with many points per group as on sets with one, and no further from float64 than float32 sums."""
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


@pytest.mark.parametrize("d,M,m", [(2, 64, 2), (2, 64, 3), (2, 64, 4), (2, 64, 5), (2, 64, 6), (2, 64, 8), (3, 16, 2),
                                   (3, 16, 3), (3, 16, 4)])
@pytest.mark.parametrize("density", [0.1, 0.5, 2, 8])
def test_least_squares_scale(d, M, m, density):
    """The scale that fits the float32 grid to the float64 one differs from 1 by less than u / 4 = 1.5e-8:
    the truncations' mean 3.7e-8 is made up to about a tenth (the mantissas' mean reciprocal varies by that much),
    the window's table carries its constant to twice the precision, and the cells' own roundings (1e-7, of either
    sign) average over thousands of cells."""
    L, torch = lib_or_skip()
    N = int(density * M ** d)
    x = inputs.random_points(N, d, 60 + m)
    f32 = to_dev(torch, inputs.samples_complex(N, 61), torch.complex64)
    g = _grid(L, torch, L.Plan(x, M, 2.0, m, "fp32"), f32)
    G = _grid(L, torch, L.Plan(x, M, 2.0, m, "fp64"), f32.to(torch.complex128))
    assert abs((np.vdot(G, g) / np.vdot(G, G)).real - 1) < U / 4
