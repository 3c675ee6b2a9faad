"""The update kernel's sweep (one block does several tiles and reuses the faces
between them, on grids of more than about 7300 tiles) against row slabs of the
same grid, which are too small for it: bit for bit, ragged in both directions."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2201_12193_gb300 import decomp, hweno, workloads as W

pytestmark = pytest.mark.gpu


def _problem(eq, nx, ny):
    g = np.random.default_rng(5)
    shape = (3, ny, nx)
    if eq == "euler":
        r = 1.0 + 0.5 * (g.random((ny, nx)) < 0.1)
        m = np.zeros((4,) + shape)
        m[:, 0] = W.prim_to_cons_2d(r, 0.3 * g.standard_normal((ny, nx)), 0.2 * g.standard_normal((ny, nx)),
                                    1.0 + 0.2 * g.random((ny, nx)))
        m[:, 1:] = 1e-3 * g.standard_normal((4, 2, ny, nx))
    else:
        m = 0.1 * g.standard_normal((1,) + shape)
        m[:, 0] += 1.0
    bc = ("transmissive",) * 2 + ("periodic",) * 2
    return W.Problem("sweep", 2, nx, ny, 0.0, nx / 1024, 0.0, ny / 1024, eq, bc, m, adv=(1.0, 0.5))


@pytest.mark.parametrize("eq,prec", [("euler", "fp64"), ("euler", "df64"), ("burgers", "fp64")])
@pytest.mark.parametrize("nx,ny", [(1031, 1021), (97, 9803)])
def test_swept_tiles_equal_single_tiles(eq, prec, nx, ny):
    p = _problem(eq, nx, ny)
    s = hweno.Solver.from_problem(p, precision=prec)
    s.set_moments(p.m)
    dt = s.max_dt(0.4)
    s.step(dt)
    d = decomp.LocalSlabs(p, 4, precision=prec)
    d.set_moments(p.m)
    d.step(dt)
    assert np.array_equal(s.get_moments(), d.gather())
