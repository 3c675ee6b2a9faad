"""Calls for single-problem handles refuse a batch handle (it has none of the buffers
they work with) with ESTATE, and leave it usable."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2201_12193_gb300 import hweno, workloads as W

pytestmark = pytest.mark.gpu

ESTATE = -5


@pytest.mark.parametrize("call", ["max_dt", "wave_speeds", "totals", "step", "stage", "advance", "rhs"])
def test_single_problem_calls_refuse_batches(call):
    probs = [W.four_quadrant_2d(16, seed=1), W.vortex_2d(24, seed=2)]
    s = hweno.BatchSolver(probs)
    for k, p in enumerate(probs):
        s.set_moments(k, p.m)
    L, out, mask = hweno.lib(), (ctypes.c_double * 8)(), torch.zeros(16 * 16, dtype=torch.uint8, device="cuda")
    U = torch.from_numpy(probs[0].m).cuda()
    a, b = torch.empty_like(U), torch.empty_like(U)
    t, n = ctypes.c_double(), ctypes.c_longlong()
    got = {
        "max_dt": lambda: L.hweno_max_dt(s._h, 0.6, ctypes.cast(out, ctypes.POINTER(ctypes.c_double))),
        "wave_speeds": lambda: L.hweno_wave_speeds(s._h, ctypes.cast(out, ctypes.POINTER(ctypes.c_double))),
        "totals": lambda: L.hweno_totals(s._h, ctypes.cast(out, ctypes.POINTER(ctypes.c_double))),
        "step": lambda: L.hweno_step(s._h, 1e-3),
        "stage": lambda: L.hweno_stage(s._h, 0, 1e-3),
        "advance": lambda: L.hweno_advance(s._h, 1.0, 0.6, 1, ctypes.byref(t), ctypes.byref(n)),
        "rhs": lambda: L.hweno_rhs(s._h, U.data_ptr(), a.data_ptr(), b.data_ptr(), mask.data_ptr(), None),
    }[call]()
    assert got == ESTATE and "single-problem" in L.hweno_last_error(s._h).decode()
    s.step(cfl=0.6)
    s.sync()
    assert np.isfinite(s.get_moments(1)).all()
