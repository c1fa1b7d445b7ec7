"""A context that joins an ensemble keeps working for what was made from it before:
its tangent, its recorded adjoint sweep and its slab group (joining drops the
captured time steps, which all three launch)."""
import numpy as np
import pytest

from paper_1907_00080_gb300 import inputs, lbib

pytestmark = pytest.mark.gpu


def join(*sims):
    """an ensemble of the simulations (it owns their contexts from here on)"""
    for s in sims:
        s.owned_by_ensemble = True
    return lbib.lbib_ensemble_create([s.ctx for s in sims])


@pytest.mark.parametrize("steps", [1, 4])
def test_tangent(steps):
    wl = inputs.capsule_128x32("f64", bonds="stress")
    dxy = np.random.default_rng(3).normal(size=(wl.n_vertices, 2))
    out = []
    for joins in (False, True):
        s = lbib.Simulation(wl)
        s.step(5 + steps % 2)
        t = lbib.lbib_tangent_create(s.ctx)
        lbib.lbib_tangent_seed(s.ctx, t, [0.0], [0.0], 0.0, dxy, None)
        ens = join(s) if joins else None
        lbib.lbib_tangent_step(s.ctx, t, steps)
        out.append((*lbib.lbib_tangent_read(s.ctx, t, wl.n_vertices), s.markers(), s.populations()))
        lbib.lbib_tangent_destroy(t)
        s.close()
        lbib.lbib_ensemble_destroy(ens)
    for x, y in zip(*out):
        assert np.array_equal(x, y)


def test_recorded_adjoint():
    wl = inputs.capsule_128x32("f64", bonds="stress")
    xb = np.random.default_rng(4).normal(size=(wl.n_vertices, 2))
    out = []
    for joins in (False, True):
        s = lbib.Simulation(wl)
        a = lbib.lbib_adjoint_create(s.ctx, 4)
        lbib.lbib_adjoint_record(s.ctx, a, 10)
        lbib.lbib_adjoint_seed(s.ctx, a, xb)
        ens = join(s) if joins else None
        lbib.lbib_adjoint_reverse(s.ctx, a)
        r = lbib.lbib_adjoint_read(s.ctx, a, wl.n_vertices, 1, wl.nx * wl.ny)
        out.append([np.asarray(r[k]) for k in ("xy", "xy_prev", "k_s", "k_b", "f")] + [s.markers()])
        lbib.lbib_adjoint_destroy(a)
        s.close()
        lbib.lbib_ensemble_destroy(ens)
    # the sweep adds with floating-point atomics, in any order: sums of up to 1e4 FP64
    # terms (1e-12 of the terms), which cancel to a thousandth at most
    for x, y in zip(*out):
        assert np.max(np.abs(x - y)) <= 1e-9 * np.max(np.abs(y))


def test_slabs():
    wl = inputs.Workload(name="lat", nx=48, ny=20, body_force=(2e-6, 0.0), walls=1, init="rest", precision="f32",
                         membranes=[], receptors=None)
    f0 = inputs.random_populations(48, 20, [4 / 9] + [1 / 9] * 4 + [1 / 36] * 4, seed=2)
    whole = lbib.Simulation(wl)
    whole.set_populations(f0)
    group = lbib.Slabs(wl, [20, 28], f0=f0)
    ens = join(*group.sims)
    whole.step(7)
    group.step(7)
    assert np.array_equal(whole.populations(), group.populations())
    group.close()
    lbib.lbib_ensemble_destroy(ens)
    whole.close()
