"""The chained launches of a captured time step (a kernel's prologue runs beside
its predecessor): many steps in one call, whose kernels overlap across steps,
against the same steps taken one call at a time with a wait after each.  Every
sum of the time step has a fixed order or is over integers, so the state has to
be the same bits.  Sizes: capsule and odd lattices, both fused-kernel forms,
dynamic particles (four kernels), lattices without markers."""
import dataclasses

import numpy as np
import pytest

from paper_1907_00080_gb300 import inputs, lbib

pytestmark = pytest.mark.gpu


def state(sim):
    return sim.populations(), sim.markers(), sim.bonds()


def same(a, b):
    for x, y in zip(a, b):
        assert np.array_equal(x, y)


def together_and_apart(wl, precision, tiling, n):
    one, many = (lbib.Simulation(wl, precision=precision, tiling=tiling) for _ in range(2))
    many.step(n)
    many.sync()
    for _ in range(n):
        one.step(1)
        one.sync()
    same(state(one), state(many))
    one.close()
    many.close()


@pytest.mark.parametrize("precision", ["f64", "f32", "f16", "bf16"])
@pytest.mark.parametrize("case", ["capsule", "dynamic", "capillary", "persistent", "soft_ring"])
def test_steps_together_and_apart(case, precision):
    tiling = None
    if case == "capsule":
        wl = inputs.capsule_128x32(bonds="stress")
    elif case == "dynamic":
        wl = inputs.dynamic_carriers_128x48()
    elif case == "soft_ring":
        # one soft carrier of 210 vertices near the wall: several units per ring,
        # ligands on elements that straddle two of them
        wl = inputs.couette_cfl_600x200(carrier="soft")
        wl = dataclasses.replace(wl, bonds=dict(inputs.STRESS_BONDS, d_cut=wl.bonds["d_cut"]))
        wl.membranes[0].ligands = np.arange(210, dtype=np.int32)
        if precision == "f16":
            pytest.skip("the scaled FP16 range does not cover adhesion forces at this wall speed")
    else:
        wl = inputs.capillary(nx=200, ny=96, n_rbc=2, rbc_alpha=38.0, rbc_markers=120, n_carriers=2,
                              carrier_radius=5.0, carrier_markers=32, bonds="stress")
        if case == "persistent":
            tiling = (2 if precision != "f64" else 1, 0)
    together_and_apart(wl, precision, tiling, 37)


@pytest.mark.parametrize("walls", [0, 1, 2])
@pytest.mark.parametrize("nx,ny,tiling", [(33, 7, None), (64, 6, (1, 0)), (1032, 9, (2, 0))])
def test_lattice_steps_together_and_apart(walls, nx, ny, tiling):
    wl = inputs.Workload("lattice", nx, ny, body_force=(1e-6, 0.0), walls=walls, init="rest")
    f0 = inputs.random_populations(nx, ny, [4 / 9] + [1 / 9] * 4 + [1 / 36] * 4, seed=nx)
    sims = [lbib.Simulation(wl, precision="f32", tiling=tiling) for _ in range(2)]
    for s in sims:
        s.set_populations(f0)
    sims[0].step(35)
    for _ in range(35):
        sims[1].step(1)
        sims[1].sync()
    same((sims[0].populations(),), (sims[1].populations(),))
    for s in sims:
        s.close()


@pytest.mark.parametrize("precision,tiling", [("f32", (2, 0)), ("f32", (4, 1)), ("f16", (4, 0)), ("f64", (1, 2))])
def test_ensemble_steps_together_and_apart(precision, tiling):
    wls = [inputs.capillary(nx=nx, ny=64, n_rbc=1, rbc_alpha=25.6, rbc_markers=80, n_carriers=2, carrier_radius=4.0,
                            carrier_markers=32, ca_carrier=(ca,), seed=7 + nx, bonds="stress")
           for nx, ca in ((128, 0.0), (256, 1e-2), (192, 0.0))]
    one, many = (lbib.Ensemble(wls, precision=precision, tiling=tiling) for _ in range(2))
    many.step(37)
    many.sync()
    for _ in range(37):
        one.step(1)
        one.sync()
    for a, b in zip(one.members, many.members):
        same(state(a), state(b))
    one.close()
    many.close()


@pytest.mark.parametrize("n", [1, 2, 3, 7, 31, 32, 33, 63, 65])
def test_any_number_of_steps(n):
    """captured sequences of 1, 2, 4, .. 32 steps: any n, from either buffer"""
    wl = inputs.capsule_128x32(bonds="stress")
    a, b = (lbib.Simulation(wl, precision="f32") for _ in range(2))
    for s in (a, b):
        s.step(1)
    a.step(n)
    for _ in range(n):
        b.step(1)
    assert lbib.lbib_step_count(a.ctx) == lbib.lbib_step_count(b.ctx) == n + 1
    same(state(a), state(b))
    a.close()
    b.close()
