"""Batched stages as one persistent launch each (set_barrier) against a launch per
phase: the same states, step lengths and flags, all precisions and tile shapes."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2201_12193_gb300 import hweno, workloads as W

pytestmark = pytest.mark.gpu


def _run(probs, precision, variant, persistent, dt):
    s = hweno.BatchSolver(probs, precision=precision)
    s.set_tile(variant)
    if persistent:
        s.set_barrier()
    for k, p in enumerate(probs):
        s.set_moments(k, p.m)
    given = torch.full((len(probs),), 1e-4, dtype=torch.float64, device="cuda") if dt else None
    dts = []
    for _ in range(2):
        s.step(given, cfl=0.6)
        dts.append(s.dts())
    s.sync()
    out = [s.get_moments(k) for k in range(len(probs))]
    masks = [s.troubled_mask(k) for k in range(len(probs))]
    s.close()
    return out, np.array(dts), masks


@pytest.mark.parametrize("dt", [False, True])
@pytest.mark.parametrize("variant", [0, 1, 2])
@pytest.mark.parametrize("precision", ["fp64", "df64", "fp32"])
def test_both_forms_agree(precision, variant, dt):
    probs = [W.four_quadrant_2d(16, seed=1), W.vortex_2d(32, seed=2), W.four_quadrant_2d(70, seed=6, ny=36)]
    a, ta, ma = _run(probs, precision, variant, False, dt)
    b, tb, mb = _run(probs, precision, variant, True, dt)
    assert np.array_equal(ta, tb)
    for k in range(len(probs)):
        if precision == "fp32":    # (two compilations of the same FP32 expressions: the bar of the FP32 form)
            assert np.abs(a[k] - b[k]).sum() <= 5e-6 * np.abs(a[k]).sum()
        else:
            assert np.array_equal(ma[k], mb[k]) and np.array_equal(a[k], b[k])


def test_the_persistent_form_waits_at_its_barrier():
    """A wait bounded to one poll gives up: the step is reported and rolled back."""
    probs = [W.four_quadrant_2d(70, seed=6, ny=36), W.vortex_2d(32, seed=2)]
    s = hweno.BatchSolver(probs)
    for k, p in enumerate(probs):
        s.set_moments(k, p.m)
    s.set_barrier(spin_limit=1)
    s.step(cfl=0.6)
    with pytest.raises(hweno.HwenoError) as e:
        s.sync()
    assert e.value.status == -4
    for k, p in enumerate(probs):
        assert np.array_equal(s.get_moments(k), p.m)
