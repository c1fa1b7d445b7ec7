"""Marker kernels where their plans change.

Rings of more than 256 vertices: the enclosed area comes from the chunks' sums,
which the advance kernel leaves behind, instead of a walk over the ring; after
set-up, after a write of the markers and after a load they are summed anew.

Repulsion candidates: found group by group; the first 48 segments of a block are
staged, up to 256 listed, beyond that every segment is walked.

Ligands at heights that no receptor is near: the receptor grid is not read.

Tolerances.  Forces of the first step, from equal positions: 1e-12 (FP64) and
1e-5 (FP32), as for short rings.  After further steps the positions differ by
roundings: an ulp at 300 lattice units is 5.7e-14; four of them over an edge's
strain (0.1 of 0.5) are 4.6e-12 of the largest force in FP64, taken as 1e-11.
In FP32 the marker velocities carry about 1e-7, 4e-7 in four steps, which is
1.6e-5 of the largest force, taken as 1e-4.  A chunk missing from the area
changes a force by its order of magnitude."""
import dataclasses

import numpy as np
import pytest

from helpers import make_oracle, rel_err
from paper_1907_00080_gb300 import inputs, lbib

pytestmark = pytest.mark.gpu


def ring_case(n, prec, kind=0):
    """one ring of n vertices, half a lattice unit apart, slightly blown up"""
    r = max(0.5 * n / (2 * np.pi), 6.0)
    nx = int(2 * r) + 30
    wl = inputs.Workload(name="ring", nx=nx, ny=nx, body_force=(1e-7, 0.0), walls=1, init="poiseuille",
                         precision=prec, receptors=None)
    wl.membranes = [inputs.Membrane(xy=inputs.circle(nx / 2 + 0.3, nx / 2 - 0.2, r, n), ks=0.02, kb=0.001, ka=0.3,
                                    kind=kind)]
    rng = np.random.default_rng(n)
    c = np.array([nx / 2 + 0.3, nx / 2 - 0.2])
    xy = c + 1.01 * (wl.membranes[0].xy - c)
    if kind in (0, 2):
        xy = xy + rng.normal(scale=0.02, size=(n, 2))
    return wl, xy


@pytest.mark.parametrize("prec", ["f64", "f32"])
@pytest.mark.parametrize("n", [64, 65, 255, 256, 257, 320, 321, 1700])
def test_ring_forces(n, prec):
    wl, xy = ring_case(n, prec)
    s, r = lbib.Simulation(wl), make_oracle(wl)
    lbib.lbib_write_markers(s.ctx, xy)
    r.set_markers(xy, xy)
    s.step(1)
    r.step(1)
    assert rel_err(s.forces(), r.forces()) < (1e-12 if prec == "f64" else 1e-5)
    s.step(4)
    r.step(4)
    assert rel_err(s.forces(), r.forces()) < (1e-11 if prec == "f64" else 1e-4)
    # a second write mid-run: the sums of the old positions are not used
    xy2 = xy + np.array([0.4, -0.3])
    lbib.lbib_write_markers(s.ctx, xy2)
    r.set_markers(xy2, xy2)
    s.step(1)
    r.step(1)
    assert rel_err(s.forces(), r.forces()) < (1e-11 if prec == "f64" else 1e-4)
    s.close()


@pytest.mark.parametrize("kind,n", [(0, 320), (1, 256), (2, 320), (3, 256)])  # rigid bodies have 256 vertices at most
@pytest.mark.parametrize("prec", ["f64", "f32", "f16"])
def test_ring_resumes(kind, n, prec, tmp_path):
    wl, _ = ring_case(n, prec, kind)
    a, b = lbib.Simulation(wl), lbib.Simulation(wl)
    a.step(7)
    path = str(tmp_path / "ring.lbib")
    a.save(path)
    b.load_state(path)
    a.step(9)
    for _ in range(9):
        b.step(1)
        b.sync()
    assert np.array_equal(a.markers(), b.markers())
    assert np.array_equal(a.populations(), b.populations())
    a.close()
    b.close()


@pytest.mark.parametrize("prec", ["f64", "f32"])
@pytest.mark.parametrize("n", [200, 1000, 3000])
def test_repulsion_of_a_dense_ring(n, prec):
    """a ring of 24 beside one of n vertices around a radius of 4: 25, 125 and
    375 segments, about 40 % of them near the first ring's box"""
    wl = inputs.Workload(name="dense", nx=64, ny=32, walls=1, init="rest", precision=prec, receptors=None)
    wl.membranes = [inputs.Membrane(xy=inputs.circle(20.0, 16.0, 4.0, 24), ks=0.0, kb=0.0, ka=0.0),
                    inputs.Membrane(xy=inputs.circle(29.4, 16.3, 4.0, n), ks=0.0, kb=0.0, ka=0.0),
                    # inside the second ring: its box meets all of that ring's groups
                    inputs.Membrane(xy=inputs.circle(29.4, 16.3, 2.3, 40), ks=0.0, kb=0.0, ka=0.0)]
    s, r = lbib.Simulation(wl), make_oracle(wl)
    s.step(1)
    r.step(1)
    F0 = r.forces()
    assert np.max(np.abs(F0[:24])) > 0
    assert rel_err(s.forces(), F0) < (1e-12 if prec == "f64" else 1e-5)
    s.close()


@pytest.mark.parametrize("prec", ["f64", "f32"])
@pytest.mark.parametrize("heights", [(0.0, 39.0), (3.0, 9.0, 9.5, 30.0), (20.0,)])
def test_bonds_at_all_heights(heights, prec):
    """rings at every height of the channel, receptors in a few rows: the bonds
    and their order of formation are the oracle's"""
    nx, ny = 160, 40
    wl = inputs.Workload(name="heights", nx=nx, ny=ny, walls=1, init="rest", precision=prec, sigma_lu=1e-4)
    rng = np.random.default_rng(5)
    wl.membranes = [inputs.Membrane(xy=inputs.circle(6.0 + 9.3 * k, 3.2 + 2.2 * k + rng.uniform(-0.2, 0.2), 2.5, 16),
                                    ks=0.05, kb=0.0, ka=0.0, ligands=np.arange(16, dtype=np.int32))
                    for k in range(16)]
    wl.receptors = np.array([(x, y) for y in heights for x in np.arange(0.0, nx, 1.0)])
    wl.bonds = dict(inputs.STRESS_BONDS, kf_dt=0.5)
    wl = dataclasses.replace(wl, seed=11)
    s, r = lbib.Simulation(wl), make_oracle(wl)
    seen = 0
    for _ in range(12):
        s.step(1)
        r.step(1)
        assert np.array_equal(s.bonds(), r.bonds())
        seen = max(seen, int((r.bonds() >= 0).sum()))
    assert seen > 3
    s.close()
