"""The profiling launches of the fused kernel and what a context keeps by population
buffer (bonds, their decisions, the step counter, the force fields): an odd number of
launches advances the populations as an even one does and changes nothing else."""
import numpy as np
import pytest

from paper_1907_00080_gb300 import inputs, lbib

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,tiling", [("f64", None), ("f32", None), ("f32", (2, 0)), ("bf16", None)])
@pytest.mark.parametrize("steps", [20, 21])
def test_odd_numbers_of_launches(steps, precision, tiling):
    wl = inputs.capsule_128x32(bonds="stress")
    a, b = (lbib.Simulation(wl, precision=precision, tiling=tiling) for _ in range(2))
    for s in (a, b):
        s.step(steps)
    bonds, markers = a.bonds(), a.markers()
    assert (bonds >= 0).any()
    lbib.lbib_profile_fused(a.ctx, 1)
    assert np.array_equal(a.bonds(), bonds) and np.array_equal(a.markers(), markers)
    assert lbib.lbib_step_count(a.ctx) == steps
    lbib.lbib_profile_fused(a.ctx, 3)
    lbib.lbib_profile_fused(b.ctx, 4)
    assert np.array_equal(a.populations(), b.populations())
    # and the time steps go on from there
    for s in (a, b):
        s.step(9)
    assert np.array_equal(a.bonds(), b.bonds())
    assert np.array_equal(a.markers(), b.markers())
    assert np.array_equal(a.populations(), b.populations())
    a.close()
    b.close()
