"""The CFL maximum of large Euler grids (exact speeds only of the cells FP32
bounds leave) against the maximum over every cell in numpy, bit for bit of the
step length through hweno_max_dt_noalloc's rule: smooth, uniform (all cells tie),
one extreme cell, nearly vacuum pressure, non-physical cells."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2201_12193_gb300 import hweno
from paper_2201_12193_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _state(kind, ny, nx, g):
    r, u, v, p = (np.full((ny, nx), x) for x in (1.0, 0.3, -0.2, 1.0))
    if kind != "uniform":
        r = r + 0.5 * g.random((ny, nx))
        u = u + g.standard_normal((ny, nx))
        v = v + g.standard_normal((ny, nx))
        p = p + g.random((ny, nx))
    if kind == "one":
        p[ny // 2, nx // 3] = 1e4
    if kind == "cold":                  # Mach 1e4: the pressure is lost in FP32
        p = 1e-8 * p
    m = np.zeros((4, 3, ny, nx))
    m[:, 0] = W.prim_to_cons_2d(r, u, v, p)
    if kind == "negative":
        m[3, 0, 1, 2] = -1.0
    return m


@pytest.mark.parametrize("kind", ["uniform", "waves", "one", "cold", "negative"])
@pytest.mark.parametrize("nx,ny", [(257, 191), (1024, 39)])
def test_filtered_maximum_is_the_maximum(kind, nx, ny):
    m = _state(kind, ny, nx, np.random.default_rng(4))
    s = hweno.Solver(2, nx, ny, x1=nx / 64, y1=ny / 64)
    s.set_positivity_check(False)
    s.set_moments(m)
    r, a, b, E = m[:, 0]
    mu, nu = a / r, b / r
    c = np.sqrt(1.4 * np.maximum(0.4 * (E - 0.5 * r * (mu * mu + nu * nu)), 0.0) / r)
    want = (np.abs(mu) + c).max(), (np.abs(nu) + c).max()
    got = s.wave_speeds()
    # numpy rounds every operation, the kernel contracts some: a few units in the last place of
    # a sum whose pressure cancels by up to E / p (1e8 when cold, entering under a root)
    assert np.allclose(got, want, rtol=1e-7 if kind == "cold" else 1e-14)
    small = [s.wave_speeds() for _ in range(3)]
    assert all(x == got for x in small)
    # the same cells one row block at a time (below the size of the filter): the same maximum, exactly
    top = np.zeros(2)
    rows = 38912 // nx - 4
    for j in range(0, ny, rows):
        k = min(rows, ny - j)
        if k < 4:
            j, k = ny - 4, 4
        q = hweno.Solver(2, nx, k, x1=nx / 64, y1=k / 64)
        q.set_positivity_check(False)
        q.set_moments(np.ascontiguousarray(m[:, :, j:j + k]))
        top = np.maximum(top, q.wave_speeds())
        q.close()
    assert tuple(top) == got
