"""FP64 reconstruction of data near the lower end of FP64's range (a state in
other units): the same relative accuracy as at size 1, against the oracle."""
import numpy as np
import pytest

import oracle
from paper_2201_12193_gb300 import hweno

pytestmark = pytest.mark.gpu

ADV = (1.0, 0.5)


@pytest.mark.parametrize("dim,nx,ny", [(1, 130, 1), (2, 37, 9)])
@pytest.mark.parametrize("base", [0.0, 1.0])
@pytest.mark.parametrize("scale", [1e-100, 1e-160, 1e-172, 1e-200, 1e-260])
def test_tiny_data_keep_their_accuracy(dim, nx, ny, scale, base):
    import torch
    g = np.random.default_rng(2)
    m = 0.1 * g.standard_normal((1, dim + 1, ny, nx))
    m[0, 0] += base
    m *= scale
    s = hweno.Solver(dim, nx, ny, x1=float(nx), y1=float(ny), eq="advection", adv=ADV, indicator="none",
                     bc=("periodic",) * 4)
    U = torch.from_numpy(m).cuda()
    L, Um = torch.empty_like(U), torch.empty_like(U)
    mask = torch.empty((s.ny, nx), dtype=torch.uint8, device="cuda")
    s.rhs(U, Um, L, mask)
    torch.cuda.synchronize()
    cfg = oracle.make_cfg(dim, nx, ny, dx=1.0, dy=1.0, eq="advection", adv=ADV, indicator="none",
                          bc=("periodic",) * 4)
    want = oracle.rhs(cfg, m)[1].reshape(m.shape)
    # sums of about 100 point values of size max|u|, each at the end of a chain of about 20
    # operations that round at 2^-53 of up to 10 max|u|: 1e-13 max|u| with dx = 1
    assert np.abs(L.cpu().numpy() - want).max() <= 1e-13 * np.abs(m).max()
