"""Row tiles of a batched ensemble: members of like sizes share one grid, members
of very different sizes and one-warp tiles of up to 64 nodes go through a list.
Either way every member computes the bits of its own single run."""
import numpy as np
import pytest

from paper_1907_00080_gb300 import inputs, lbib

pytestmark = pytest.mark.gpu

SIZES = {"one": [(128, 48)], "alike": [(128, 64), (200, 48), (136, 57)], "apart": [(64, 32), (512, 160), (72, 40), (64, 33)]}


@pytest.mark.parametrize("precision,tiling", [("f32", (4, 1)), ("f32", (2, 1)), ("f32", (1, 4)), ("f32", (2, 8)),
                                              ("f64", (2, 1)), ("f64", (1, 2)), ("bf16", (8, 1)), ("bf16", (4, 2)),
                                              ("f16", (2, 4))])
@pytest.mark.parametrize("sizes", ["one", "alike", "apart"])
def test_members_match_single_runs(sizes, precision, tiling):
    wls = [inputs.capillary(nx=nx, ny=ny, n_rbc=1, rbc_alpha=min(0.4 * ny, 25.6), rbc_markers=80, n_carriers=1,
                            carrier_radius=4.0, carrier_markers=32, ca_carrier=(0.0,), seed=3 + nx + ny)
           for nx, ny in SIZES[sizes]]
    ens = lbib.Ensemble(wls, precision=precision, tiling=tiling)
    assert ens.form == 1
    ens.step(21)
    ens.sync()
    for wl, m in zip(wls, ens.members):
        s = lbib.Simulation(wl, precision=precision, tiling=tiling)
        s.step(21)
        s.sync()
        assert np.array_equal(s.populations(), m.populations())
        assert np.array_equal(s.markers(), m.markers())
        s.close()
    ens.close()
