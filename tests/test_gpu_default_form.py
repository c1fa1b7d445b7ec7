"""The default form of the fused kernel over the sizes where it changes: the run
with it and runs in the other form give the same bits (the forms share the
collision), with and without markers, at rows that do and do not fill the
persistent form's segments."""
import numpy as np
import pytest

from paper_1907_00080_gb300 import inputs, lbib

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,nx,ny,default,other", [
    ("f32", 1504, 1000, "rows", (2, 0)),   # 108 MB in two buffers
    ("f32", 2000, 1000, (2, 0), (4, 2)),   # 144 MB
    ("f32", 2400, 1000, "rows", (2, 0)),   # 173 MB
    ("f32", 16, 140000, (2, 0), (4, 4)),   # taller than two rows a block
    ("bf16", 2000, 1000, "rows", (4, 0)),  # 2.0 M nodes
    ("bf16", 2400, 1000, (4, 0), (4, 2)),  # 2.4 M nodes, full rows
    ("bf16", 1032, 2400, (2, 0), (4, 1)),  # short rows
    ("bf16", 1032, 3600, (4, 0), (4, 2)),  # 134 MB
])
@pytest.mark.parametrize("markers", [False, True])
def test_default_form_and_the_other(markers, prec, nx, ny, default, other):
    if markers and nx > 1000:
        wl = inputs.probe_lattice(nx, ny, prec)
    else:
        # (a channel of 140000 rows has no Poiseuille state of finite Mach number at this force)
        wl = inputs.Workload("lattice", nx, ny, body_force=(1e-7, 0.0), walls=1,
                             init="poiseuille" if nx > 1000 else "rest", precision=prec)
    a, b = lbib.Simulation(wl, precision=prec), lbib.Simulation(wl, precision=prec, tiling=other)
    a.step(5)
    b.step(5)
    assert (a.tiling[1] > 0) if default == "rows" else (a.tiling == default)
    assert np.array_equal(a.populations(), b.populations())
    assert np.array_equal(a.markers(), b.markers())
    a.close()
    b.close()
