"""Force flags, one bit per node in words of 32: membranes placed across the ends
of rows whose last word holds 1, 2, 31 or 32 nodes (odd and even NX, every node
count per thread), against the FP64 oracle with the tolerances of the parity
tests (FP64 1e-12; FP32 1e-5 of the velocity scale over a few steps)."""
import numpy as np
import pytest

from helpers import f64_field_tol, make_oracle, rel_err, vel_err
from paper_1907_00080_gb300 import inputs, lbib

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,precision,tiling", [
    (33, "f64", (1, 2)), (33, "f32", (1, 1)), (34, "f64", (2, 1)), (63, "f32", (1, 4)), (64, "f32", (4, 2)),
    (65, "f64", (1, 1)), (64, "f32", (1, 0)), (516, "f32", (2, 0)), (1028, "f32", (4, 0)), (258, "f64", (1, 0))])
def test_membranes_across_row_ends(nx, precision, tiling):
    ny = 24
    wl = inputs.Workload("row_ends", nx, ny, body_force=(inputs.body_force_for(0.01, ny), 0.0), walls=1,
                         init="poiseuille", precision=precision)
    # one capsule around x = NX, one at a word's end inside the row, moved apart in y
    for x0, y0 in ((nx - 0.3, 6.3), (float(32 * (nx // 64)), 16.7)):
        wl.membranes.append(inputs.Membrane(xy=inputs.circle(x0, y0, 4.0, 32) * [1.0, 0.9] + [0.0, 0.1 * y0],
                                            ks=0.02, kb=0.002, ka=0.1))
    # pre-stretched by a moved vertex, so that forces act from the first step
    sim, ref = lbib.Simulation(wl, tiling=tiling), make_oracle(wl)
    xy = ref.markers()
    xy[3] += [0.2, 0.1]
    xy[40] += [-0.1, 0.2]
    lbib.lbib_write_markers(sim.ctx, xy)
    ref.set_markers(xy, xy)
    sim.step(6)
    ref.step(6)
    r, u, v = sim.fields()
    r0, u0, v0 = ref.fields()
    if precision == "f64":
        assert vel_err(u, v, u0, v0) < f64_field_tol(np.max(np.abs(u0)))
        assert rel_err(sim.markers(), ref.markers()) < 1e-12
    else:
        assert vel_err(u, v, u0, v0) < 1e-5
        assert np.max(np.abs(sim.markers() - ref.markers())) < 1e-5
    sim.close()
