"""The CFL maximum where its FP32 bounds have least room: gas so thin that squares
of its momentum leave FP32's range, and gamma near 1.  2D, 1D (grids above the
filter's size) and batches, against the FP64 maximum over all cells."""
from types import SimpleNamespace

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2201_12193_gb300 import hweno

pytestmark = pytest.mark.gpu


def _cells(kind, shape, gamma):
    """rho, u, v, p: many cells whose speed the bounds overstate, one faster cell."""
    r, u, v, p = (np.zeros(shape) for _ in range(4))
    one = tuple(n // 3 for n in shape)
    if kind == "thin":                       # moving at 10 and cold beside one hotter cell at rest
        r += 1e-24
        u += 10.0
        v += 10.0
        p += 1e-24
        u[one], v[one], p[one] = 0.0, 0.0, 15.0 ** 2 * 1e-24 / gamma
    elif kind == "thin at rest":             # momenta 0
        r += 1e-30
        p += r / gamma
        p[one] *= 1.5
    else:                                    # at rest, sound speed 1 beside |u| + c = 1.00002 of a moving cell
        r += 1.0
        p += 1.0 / gamma
        u[one], v[one], p[one] = 0.99, 0.99, 0.01002 ** 2 / gamma
    return r, u, v, p


def _speeds(r, u, v, p, gamma):
    c = np.sqrt(gamma * p / r)
    return (np.abs(u) + c).max(), (np.abs(v) + c).max()


CASES = [("thin", 1.4), ("thin", 3.0), ("thin at rest", 1.4), ("close", 1.0001), ("close", 1.01), ("close", 1.4)]


# the kernel's speeds: a few FP64 roundings of 2^-53, amplified by the pressure's cancellation: the
# kinetic energy over the pressure, at most 1e4 (1e2 where 1 / (gamma - 1) outweighs it), under a root
@pytest.mark.parametrize("kind,gamma", CASES)
@pytest.mark.parametrize("shape", [(203, 257), (60000,)])
def test_the_fastest_cell_is_found(kind, gamma, shape):
    r, u, v, p = _cells(kind, shape, gamma)
    dim = len(shape)
    v = v if dim == 2 else 0.0 * v
    nx, ny = shape[-1], shape[0] if dim == 2 else 1
    q = [r, r * u, r * v, p / (gamma - 1.0) + 0.5 * r * (u * u + v * v)]
    if dim == 1:
        q.pop(2)
    m = np.zeros((len(q), dim + 1, ny, nx))
    m[:, 0] = np.stack([x.reshape(ny, nx) for x in q])
    s = hweno.Solver(dim, nx, ny, x1=nx / 64, y1=ny / 64, gamma=gamma)
    s.set_moments(m)
    want = _speeds(r, u, v, p, gamma)
    got = s.wave_speeds()
    assert np.allclose(got[:dim], want[:dim], rtol=1e-10)


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("kind,gamma", CASES)
def test_batches_find_the_fastest_cell(kind, gamma, precision):
    grids = [SimpleNamespace(nx=n, ny=n, x0=0.0, x1=1.0, y0=0.0, y1=1.0, bc=("transmissive",) * 4) for n in (24, 70)]
    s = hweno.BatchSolver(grids, gamma=gamma, precision=precision)
    want = []
    for k, g in enumerate(grids):
        r, u, v, p = _cells(kind, (g.ny, g.nx), gamma)
        m = np.zeros((4, 3, g.ny, g.nx))
        m[:, 0] = np.stack([r, r * u, r * v, p / (gamma - 1.0) + 0.5 * r * (u * u + v * v)])
        s.set_moments(k, m)
        a, b = _speeds(r, u, v, p, gamma)
        want.append(0.5 / ((a + b) * g.nx))
    s.step(cfl=0.5)
    assert np.allclose(s.dts(), want, rtol=1e-10)
