"""Markers many periods away from the lattice, in x and (without walls) in y: the
stencils, the forces of rings close to each other across periods and the interpolated
velocities are the oracle's. And the tallest lattices' default form with markers.

Tolerances. FP64: a position 1000 lattice units away carries 1.1e-13 of rounding, the
strain of an edge of 0.8 that of four such, 6e-13 of a largest strain of 0.05 or more:
1e-11 of the largest force. FP32 positions are pairs of floats (48 bits, 4e-12 at
1000): the parity tests' 1e-5."""
import numpy as np
import pytest

from helpers import make_oracle, rel_err, vel_err
from paper_1907_00080_gb300 import inputs, lbib

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["f64", "f32"])
@pytest.mark.parametrize("nx,ny,walls,px,py,qx,qy", [
    (48, 40, 1, 7, 0, 0, 0), (48, 40, 1, -20, 0, 3, 0),      # walls: periods in x alone
    (48, 40, 0, 0, 0, 0, 0), (48, 40, 0, 5, -9, 0, 0), (33, 37, 0, -11, 6, 0, 0),
    (48, 40, 0, 4, 3, 2, 0), (48, 40, 0, 2, -1, 0, 1), (48, 40, 0, 2, -1, 0, -4), (33, 37, 0, -3, 5, -2, 3)])
def test_rings_in_other_periods(nx, ny, walls, px, py, qx, qy, prec):
    """two rings 1.3 apart, moved by (px, py) periods, the second by (qx, qy) more"""
    wl = inputs.Workload(name="periods", nx=nx, ny=ny, body_force=(2e-6, 1e-6 * (not walls)), walls=walls, init="rest",
                         precision=prec, receptors=None)
    for cx, cy, ax, ay in ((8.3, 11.2, px, py), (16.9, 14.1, px + qx, py + qy)):
        wl.membranes.append(inputs.Membrane(xy=inputs.circle(cx + ax * nx, cy + ay * ny, 3.9, 32), ks=0.02, kb=0.002,
                                            ka=0.1))
    s, r = lbib.Simulation(wl), make_oracle(wl)
    xy = r.markers()
    xy[::5] += [0.05, -0.04]
    lbib.lbib_write_markers(s.ctx, xy)
    r.set_markers(xy, xy)
    tol = 1e-11 if prec == "f64" else 1e-5
    for n in (1, 5):
        s.step(n)
        r.step(n)
        assert rel_err(s.forces(), r.forces()) < (tol if n == 1 else 10 * tol)
    _, u, v = s.fields()
    _, u0, v0 = r.fields()
    assert vel_err(u, v, u0, v0) < 10 * tol
    s.close()


def test_repulsion_across_periods_is_there():
    """(the rings of the test above do repel each other)"""
    F = []
    for rep in (2.0, 0.0):
        wl = inputs.Workload(name="periods", nx=48, ny=40, walls=0, init="rest", precision="f64", receptors=None,
                             d_rep=rep)
        for cx, cy in ((8.3, 11.2), (16.9 + 96.0, 14.1 - 160.0)):
            wl.membranes.append(inputs.Membrane(xy=inputs.circle(cx, cy, 3.9, 32), ks=0.0, kb=0.0, ka=0.0))
        s = lbib.Simulation(wl)
        s.step(1)
        F.append(np.max(np.abs(s.forces())))
        s.close()
    assert F[0] > 0 and F[1] == 0


def test_tall_default_form_with_markers():
    """taller than two rows a block can cover: the persistent form, with markers"""
    wl = inputs.Workload("tall", 16, 140000, body_force=(1e-7, 0.0), walls=1, init="rest", precision="f32",
                         receptors=None)
    for y in (4.6, 70000.3, 139994.2):
        wl.membranes.append(inputs.Membrane(xy=inputs.circle(8.4, y, 3.5, 24), ks=0.02, kb=0.002, ka=0.1))
    a, b = lbib.Simulation(wl), lbib.Simulation(wl, tiling=(4, 4))
    xy = np.concatenate([m.xy for m in wl.membranes])
    xy[::5] += [0.1, -0.08]
    for s in (a, b):
        lbib.lbib_write_markers(s.ctx, xy)
        s.step(5)
    assert a.tiling == (2, 0)
    assert np.array_equal(a.markers(), b.markers())
    assert not np.array_equal(a.markers(), xy)
    assert np.array_equal(a.populations(), b.populations())
    a.close()
    b.close()
