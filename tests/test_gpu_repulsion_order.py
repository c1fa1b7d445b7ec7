"""Repulsion of a block with 49 candidate segments and more, of which 48 are staged,
up to 256 listed, and all walked beyond that: a pair's force is the same bits on each
way, so that it does not matter in which order the segments were found.

A ring of 24 vertices, the first 40 vertices of a second ring within d_rep of it.
The other vertices of the second ring, out of range of every vertex of the first,
either lie inside the first ring (its block then has all of their segments as
candidates) or far away (the block has five candidates, all staged).  The pairs in
range are the same, so the first ring's forces have to be the same bits."""
import numpy as np
import pytest

from paper_1907_00080_gb300 import inputs, lbib

pytestmark = pytest.mark.gpu


def rings(n, prec, near, nx=80):
    wl = inputs.Workload(name="order", nx=nx, ny=32, walls=1, init="rest", precision=prec, receptors=None)
    t = np.linspace(-0.55, 0.55, 40)
    close = np.stack([20.0 + 5.31 * np.cos(t), 16.0 + 5.31 * np.sin(t)], axis=1)
    rest = inputs.circle(20.0 if near else 50.0, 16.0, 1.0, n - 40)
    wl.membranes = [inputs.Membrane(xy=inputs.circle(20.0, 16.0, 4.0, 24), ks=0.0, kb=0.0, ka=0.0),
                    inputs.Membrane(xy=np.concatenate([close, rest]), ks=0.0, kb=0.0, ka=0.0)]
    return wl


def first_forces(wl):
    s = lbib.Simulation(wl)
    s.step(1)
    F = s.forces()[:24]
    s.close()
    return F


@pytest.mark.parametrize("prec", ["f64", "f32"])
@pytest.mark.parametrize("n", [384, 400, 1000, 2048, 2056])  # 48, 50, 125, 256 and 257 candidates
def test_pairs_in_range(n, prec):
    far, near = (first_forces(rings(n, prec, k)) for k in (False, True))
    assert np.max(np.abs(far)) > 0
    assert np.array_equal(far, near)


@pytest.mark.parametrize("prec,tiling", [("f64", (2, 1)), ("f32", (2, 0)), ("f32", (4, 1))])
def test_batched_members_match_single_runs(prec, tiling):
    wls = [rings(n, prec, True, nx=128) for n in (400, 1000, 2056)]
    ens = lbib.Ensemble(wls, precision=prec, tiling=tiling)
    assert ens.form == 1
    ens.step(5)
    ens.sync()
    for wl, m in zip(wls, ens.members):
        s = lbib.Simulation(wl, precision=prec, tiling=tiling)
        s.step(5)
        assert np.array_equal(s.forces(), m.forces())
        assert np.array_equal(s.markers(), m.markers())
        s.close()
    ens.close()
