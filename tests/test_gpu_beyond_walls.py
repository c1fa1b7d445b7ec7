"""A ring beyond a wall, whose stencils hold no fluid row: its velocity is zero,
whatever the velocity field holds from before. A step from populations that are not
finite leaves such velocities behind; a state loaded after it goes on as in a context
that never saw them."""
import numpy as np
import pytest

from paper_1907_00080_gb300 import inputs, lbib

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["f64", "f32", "f16"])
@pytest.mark.parametrize("y", [-5.2, 28.4])
def test_state_loaded_after_a_failure(y, prec, tmp_path):
    nx, ny = 64, 24
    wl = inputs.Workload(name="outside", nx=nx, ny=ny, body_force=(1e-6, 0.0), walls=1, init="poiseuille",
                         precision=prec, receptors=None)
    inside = 1.4 if y < 0 else ny - 2.4
    wl.membranes = [inputs.Membrane(xy=inputs.circle(20.0, 12.0, 3.0, 24), ks=0.01, kb=0.0, ka=0.1),
                    inputs.Membrane(xy=inputs.circle(40.3, inside, 2.0, 16), ks=0.01, kb=0.0, ka=0.1)]
    start = np.concatenate([m.xy for m in wl.membranes])
    moved = start.copy()
    moved[24:, 1] += y - inside
    path = str(tmp_path / "outside.lbib")
    a, b = lbib.Simulation(wl), lbib.Simulation(wl)
    lbib.lbib_write_markers(a.ctx, moved)
    a.step(2)
    a.save(path)
    # across the wall, in a flow that is not finite
    lbib.lbib_write_markers(a.ctx, start)
    a.set_populations(np.full((9, ny, nx), np.nan))
    a.step(1)
    with pytest.raises(lbib.LbibError) as e:
        a.sync()
    assert e.value.status == lbib.LBIB_E_NONFINITE
    for s in (a, b):
        s.load_state(path)
        s.step(3)
        s.sync()
    assert np.array_equal(a.markers(), b.markers())
    assert np.array_equal(a.populations(), b.populations())
    a.close()
    b.close()
