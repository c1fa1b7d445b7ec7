"""Bond decisions where the FP32 probability is not a number: a rupture rate of 1e-46
per step is 0 in FP32 while exp(beta_r z^2) overflows there, and the FP64 probability
decides (0 below z^2 = 17.6, near certainty above 18). The bonds are the oracle's."""
import numpy as np
import pytest

from helpers import make_oracle
from paper_1907_00080_gb300 import inputs, lbib

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["f64", "f32", "bf16"])
def test_rupture_probability_beyond_fp32(prec):
    nx, ny = 160, 40
    wl = inputs.Workload(name="stiff", nx=nx, ny=ny, walls=1, init="rest", precision=prec, sigma_lu=1e-6)
    wl.membranes = [inputs.Membrane(xy=inputs.circle(8.0 + 9.3 * k, 3.3 + 0.02 * k, 2.5, 16), ks=0.05, kb=0.0, ka=0.0,
                                    ligands=np.arange(16, dtype=np.int32)) for k in range(16)]
    wl.receptors = np.array([(x, y) for y in (-0.5, 0.5) for x in np.arange(0.25, nx, 1.0)])
    wl.bonds = dict(inputs.STRESS_BONDS, d_cut=1.5, y_eq=0.25, d_break=3.0, kf_dt=0.3, beta_f=0.0, kr0_dt=1e-46,
                    beta_r=6.0)
    s, r = lbib.Simulation(wl), make_oracle(wl)
    kept = broken = 0
    before = r.bonds()
    for _ in range(12):
        s.step(1)
        r.step(1)
        now = r.bonds()
        assert np.array_equal(s.bonds(), now)
        kept += int(((before >= 0) & (now == before)).sum())
        broken += int(((before >= 0) & (now != before)).sum())
        before = now
    assert kept > 20 and broken > 5
    s.close()
