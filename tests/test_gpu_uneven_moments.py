"""First moments that are large against the averages: the weights discard q_4
(and q_3, which takes the cell's own), and what remains keeps the accuracy of the
averages.  Against the oracle's right-hand side, FP64 (1D, 2D, batched kernels'
shared cell routine) and double-float (2D)."""
import numpy as np
import pytest

import oracle
from paper_2201_12193_gb300 import hweno

pytestmark = pytest.mark.gpu

ADV = (1.0, 0.5)


def _data(dim, nx, ny, ratio, base, scale):
    """Averages base + 0.1 noise; the first moments of every ninth cell `ratio`, the others 0.01 noise."""
    g = np.random.default_rng(5)
    m = np.zeros((1, dim + 1, ny, nx))
    m[0, 0] = base + 0.1 * g.standard_normal((ny, nx))
    m[0, 1:] = 0.01 * g.standard_normal((dim, ny, nx))
    cell = np.arange(nx)[None, :] + 4 * np.arange(ny)[:, None]
    sign = np.where(g.random((dim, ny, nx)) < 0.5, -1.0, 1.0)
    m[0, 1:] = np.where(cell % 9 == 4, ratio * sign, m[0, 1:])
    return scale * m


def _rhs(dim, nx, ny, m, precision="fp64"):
    import torch
    s = hweno.Solver(dim, nx, ny, x1=float(nx), y1=float(ny), eq="advection", adv=ADV, indicator="none",
                     bc=("periodic",) * 4, precision=precision)
    U = torch.from_numpy(m).cuda()
    L, Um = torch.empty_like(U), torch.empty_like(U)
    mask = torch.empty((s.ny, nx), dtype=torch.uint8, device="cuda")
    s.rhs(U, Um, L, mask)
    torch.cuda.synchronize()
    return L.cpu().numpy()


def _compare(dim, nx, ny, m, precision, bound):
    cfg = oracle.make_cfg(dim, nx, ny, dx=1.0, dy=1.0, eq="advection", adv=ADV, indicator="none",
                          bc=("periodic",) * 4)
    want = oracle.rhs(cfg, m)[1]
    err = np.abs(_rhs(dim, nx, ny, m, precision) - want.reshape(m.shape)).max()
    assert err <= bound, f"{err:.2e} > {bound:.2e}"


# Sums of about 100 point values of the averages' size, each at the end of a chain of
# about 20 operations that round at 2^-53 (pairs: 2^-47) of up to 10 of it: 1e-13 (6.4e-12) of the
# largest average with dx = 1.  What a discarded q_l leaves is its weight, at most
# 1 / ratio^2, times the ratio.
@pytest.mark.parametrize("base", [1.0, 0.0])
@pytest.mark.parametrize("ratio", [0.3, 1.5, 3.0, 20.0, 1e3, 1e5, 1e8])
@pytest.mark.parametrize("dim,nx,ny,precision", [(1, 135, 1, "fp64"), (2, 36, 27, "fp64"), (2, 36, 27, "df64")])
def test_large_first_moments_leave_the_averages_their_accuracy(dim, nx, ny, precision, ratio, base):
    m = _data(dim, nx, ny, ratio, base, 1.0)
    unit = 1e-13 if precision == "fp64" else 6.4e-12
    _compare(dim, nx, ny, m, precision, unit * max(np.abs(m[0, 0]).max(), 1.0 if ratio < 1e3 else 0.0))


# Data so small that the weights are the linear ones: nothing is discarded, the result
# is of the largest first moment's size.
@pytest.mark.parametrize("dim,nx,ny", [(1, 135, 1), (2, 36, 27)])
def test_noise_keeps_the_linear_weights(dim, nx, ny):
    m = _data(dim, nx, ny, 100.0, 0.0, 1e-13)
    _compare(dim, nx, ny, m, "fp64", 1e-13 * np.abs(m).max())


# Which form a stencil takes is not seen by the others of its warp.
@pytest.mark.parametrize("precision", ["fp64", "df64"])
@pytest.mark.parametrize("dim,nx,ny", [(1, 135, 1), (2, 70, 11)])
def test_the_other_cells_keep_their_bits(dim, nx, ny, precision):
    m = _data(dim, nx, ny, 0.02, 1.0, 1.0)
    a = _rhs(dim, nx, ny, m, precision)
    i, j = 20, ny // 2
    m[0, 1:, j, i] = 1e5
    b = _rhs(dim, nx, ny, m, precision)
    far = (np.abs(np.arange(nx) - i)[None, :] > 2) | (np.abs(np.arange(ny) - j)[:, None] > 2)
    assert np.array_equal(a[..., far], b[..., far]) and not np.array_equal(a, b)


# 2D Euler: batches and single handles send the same stencils to the same form, in every
# kernel that reconstructs (first pass, troubled cells), at walls and periodic sides.
@pytest.mark.parametrize("bc", ["transmissive", "periodic", "reflective"])
@pytest.mark.parametrize("precision", ["fp64", "df64"])
def test_batches_agree_bit_for_bit(precision, bc):
    from types import SimpleNamespace
    g = np.random.default_rng(9)
    grids = [SimpleNamespace(nx=nx, ny=ny, x0=0.0, x1=nx / 64, y0=0.0, y1=ny / 64, bc=(bc,) * 4)
             for nx, ny in ((19, 33), (70, 36))]
    dt = 1e-6
    s = hweno.BatchSolver(grids, precision=precision)
    s.set_positivity_check(False)
    data = []
    for k, p in enumerate(grids):
        m = np.zeros((4, 3, p.ny, p.nx))
        m[0, 0], m[3, 0] = 1.0 + 0.2 * g.random((p.ny, p.nx)), 2.5
        m[1:3, 0] = 0.1 * g.standard_normal((2, p.ny, p.nx))
        m[1:3, 1:] = np.where(g.random((2, 2, p.ny, p.nx)) < 0.03, 1e4, 1e-3 * g.standard_normal((2, 2, p.ny, p.nx)))
        data.append(m)
        s.set_moments(k, m)
    import torch
    s.step(torch.full((2,), dt, dtype=torch.float64, device="cuda"))
    for k, p in enumerate(grids):
        one = hweno.Solver(2, p.nx, p.ny, x1=p.x1, y1=p.y1, bc=p.bc, precision=precision)
        one.set_positivity_check(False)
        one.set_moments(data[k])
        one.step(dt)
        a, b = one.get_moments(), s.get_moments(k)
        assert np.array_equal(a, b) and np.array_equal(one.troubled_mask(), s.troubled_mask(k))
        assert one.troubled_mask().any()
