"""FP64 reconstruction in block fixed point against the oracle where its integers
could go wrong: variations many orders below or above the value, jumps, zero
and constant data, all magnitudes, non-finite data, other linear weights."""
import numpy as np
import pytest

import oracle
from paper_2201_12193_gb300 import hweno

pytestmark = pytest.mark.gpu

ADV = (1.0, 0.5)


def _field(kind, dim, nx, ny, seed=3):
    g = np.random.default_rng(seed)
    shape = (dim + 1, ny, nx)
    m = np.zeros((1,) + shape)
    if kind == "constant":
        m[0, 0] = 1.7
    elif kind == "zero":
        pass
    elif kind == "smooth":
        x = 2 * np.pi * (np.arange(nx) + 0.5) / nx
        y = 2 * np.pi * (np.arange(ny) + 0.5) / ny
        m[0, 0] = 1.0 + 0.2 * np.sin(x)[None, :] + 0.1 * np.cos(y)[:, None]
        m[0, 1] = 0.2 * np.cos(x)[None, :] * (2 * np.pi / nx) / 12
    elif kind == "ripple":            # 1e-9 variations of 1
        m[0] = 1e-9 * g.standard_normal(shape)
        m[0, 0] += 1.0
    elif kind == "jump":              # a factor of 1e3 at random cells
        m[0, 0] = np.where(g.random((ny, nx)) < 0.5, 1e-3, 1.0)
        m[0, 1:] = 1e-2 * g.standard_normal((dim, ny, nx))
    elif kind == "moments_only":      # first moments without average variation
        m[0, 0] = 2.0
        m[0, 1:] = g.standard_normal((dim, ny, nx))
    else:                             # "noise"
        m[0] = g.standard_normal(shape)
    return m


def _rhs(dim, nx, ny, m, gbar=(1.0, 10.0, 100.0, 1000.0)):
    import torch
    s = hweno.Solver(dim, nx, ny, x1=float(nx), y1=float(ny), eq="advection", adv=ADV, indicator="none",
                     bc=("periodic",) * 4, gamma_bar=gbar)
    U = torch.from_numpy(m).cuda()
    L, Um = torch.empty_like(U), torch.empty_like(U)
    mask = torch.empty((s.ny, nx), dtype=torch.uint8, device="cuda")
    s.rhs(U, Um, L, mask)
    torch.cuda.synchronize()
    return L.cpu().numpy()


@pytest.mark.parametrize("dim,nx,ny", [(1, 130, 1), (2, 37, 9)])
@pytest.mark.parametrize("kind", ["constant", "zero", "smooth", "ripple", "jump", "moments_only", "noise"])
@pytest.mark.parametrize("scale", [1.0, 1e-30, 1e-6, 1e6, 1e25])
def test_fixed_point_reconstruction_matches_the_oracle(dim, nx, ny, kind, scale):
    m = scale * _field(kind, dim, nx, ny)
    got = _rhs(dim, nx, ny, m)
    cfg = oracle.make_cfg(dim, nx, ny, dx=1.0, dy=1.0, eq="advection", adv=ADV, indicator="none",
                          bc=("periodic",) * 4)
    want = oracle.rhs(cfg, m)[1]
    # both are sums of about 100 point values of size max|u|, each rounded at 2^-53 of up to
    # 10 max|u| per operation of a chain of about 20: 1e-13 max|u| with dx = 1
    top = np.abs(m).max()
    assert np.abs(got - want.reshape(got.shape)).max() <= 1e-13 * top if top else not got.any()


@pytest.mark.parametrize("gbar", [(1.0, 1.0, 1.0, 1.0), (1000.0, 1.0, 1.0, 1.0), (1e-3, 1.0, 1e3, 1e6)])
@pytest.mark.parametrize("dim,nx,ny", [(1, 64, 1), (2, 21, 14)])
def test_fixed_point_rows_of_other_linear_weights(dim, nx, ny, gbar):
    m = _field("smooth", dim, nx, ny)
    got = _rhs(dim, nx, ny, m, gbar)
    cfg = oracle.make_cfg(dim, nx, ny, dx=1.0, dy=1.0, eq="advection", adv=ADV, indicator="none",
                          gbar=gbar, bc=("periodic",) * 4)
    # c_k = (S_k/S_4)(n_k - n_{k+1}) / sum: the oracle's p_l carry up to S_l/g_l (1001 here) of rounding
    assert np.abs(got - oracle.rhs(cfg, m)[1].reshape(got.shape)).max() <= 1e-10


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
@pytest.mark.parametrize("mom", [0, 1])
@pytest.mark.parametrize("dim,nx,ny", [(1, 40, 1), (2, 16, 12)])
def test_non_finite_moments_stay_non_finite(dim, nx, ny, mom, bad):
    m = _field("smooth", dim, nx, ny)
    j, i = ny // 2, nx // 2
    m[0, mom, j, i] = bad
    got = _rhs(dim, nx, ny, m)
    assert not np.isfinite(got[0, 0, j, i])
    far = np.abs(np.arange(nx) - i) > 3
    assert np.isfinite(got[..., far]).all()
