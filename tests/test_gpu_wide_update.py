"""The two-threads-per-cell update of small FP64 grids (at most two 32 x 4 tiles per
SM) against the batched form, whose update is the one-thread kernel: bit for bit, at
ragged tiles, the smallest grid, and just below and above the line."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2201_12193_gb300 import hweno, workloads as W

pytestmark = pytest.mark.gpu


def _moments(nx, ny):
    g = np.random.default_rng(nx * 1000 + ny)
    m = np.zeros((4, 3, ny, nx))
    r = 1.0 + 0.5 * (g.random((ny, nx)) < 0.1)
    m[:, 0] = W.prim_to_cons_2d(r, 0.3 * g.standard_normal((ny, nx)), 0.2 * g.standard_normal((ny, nx)),
                                1.0 + 0.2 * g.random((ny, nx)))
    m[:, 1:] = 1e-3 * g.standard_normal((4, 2, ny, nx))
    return m


@pytest.mark.parametrize("nx,ny", [(4, 4), (31, 5), (33, 9), (128, 128), (96, 400), (97, 405), (64, 612)])
def test_small_grid_update_equals_the_batched_one(nx, ny):
    m = _moments(nx, ny)
    bc = ("transmissive",) * 2 + ("periodic",) * 2
    p = W.Problem("wide", 2, nx, ny, 0.0, nx / 64, 0.0, ny / 64, "euler", bc, m)
    s = hweno.Solver.from_problem(p)
    b = hweno.BatchSolver([p, p])
    s.set_moments(m)
    for _ in range(2):
        s.step(0.002)
    for k in range(2):
        b.set_moments(k, m)
    for _ in range(2):
        b.step(torch.full((2,), 0.002, dtype=torch.float64, device="cuda"))
    ref = s.get_moments()
    assert np.isfinite(ref).all()
    for k in range(2):
        assert np.array_equal(ref, b.get_moments(k))


def test_small_grid_update_reports_a_bad_state():
    nx, ny = 40, 22
    m = _moments(nx, ny)
    p = W.Problem("wide", 2, nx, ny, 0.0, nx / 64, 0.0, ny / 64, "euler", ("periodic",) * 4, m)
    s = hweno.Solver.from_problem(p)
    s.set_moments(m)
    s.step(5.0)                 # far beyond the stable step
    with pytest.raises(hweno.HwenoError):
        s.sync()
