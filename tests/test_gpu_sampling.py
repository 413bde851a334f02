"""The Fermi-Dirac sampling from the inverse table (csrc/pgc_fd.cuh) against the FP64 oracle, which
inverts the law per particle.  Parameters chosen where the table can go wrong: band minima near
zero (the branch point of eps^2 at the bottom of the law), far below and above the Fermi level,
low and high temperature, a range of band minima too wide for the table (the per-particle
inversion runs), ragged ensembles.  Tolerance: 1e-9 of the largest |k|, as for the FP64
trajectories (the sampled |k| is sqrt(eps^2 - eps0^2), which near the band minimum turns the
rounding of eps, 1e-16, into 1e-8 sqrt; uniforms are >= 2^-24, which bounds it by 1e-9)."""
import numpy as np
import pytest

import oracle as O
from paper_2404_19602_gb300 import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

LAWS = [dict(eps_F=0.4, T_K=300.0, eps0_lo=0.05, eps0_hi=0.15), dict(eps_F=0.4, T_K=300.0, eps0_lo=0.002, eps0_hi=0.9),
        dict(eps_F=0.2, T_K=300.0, eps0_lo=0.27, eps0_hi=0.32), dict(eps_F=-0.3, T_K=300.0, eps0_lo=0.05, eps0_hi=0.3),
        dict(eps_F=0.4, T_K=30.0, eps0_lo=0.05, eps0_hi=0.15), dict(eps_F=0.6, T_K=1500.0, eps0_lo=0.1, eps0_hi=0.2),
        dict(eps_F=0.4, T_K=300.0, eps0_lo=0.05, eps0_hi=2.4)]


@pytest.mark.parametrize("law", LAWS, ids=lambda d: "%g-%g-%g-%g" % tuple(d.values()))
@pytest.mark.parametrize("shape", ["1x1", "6x6", "21x36"])
def test_sampled_state_equals_oracle(law, shape):
    from paper_2404_19602_gb300 import build, pgc

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build.build()
    O.build()
    base = {"1x1": W.DET_FP64_1E4, "6x6": W.GAP_UQ_1E6, "21x36": W.GAP_FIELD_UQ_4E6}[shape]
    p = W.scaled(base, N=4099, precision="fp64", seed=7, **law)
    if shape == "1x1":
        p["eps0_hi"] = p["eps0_lo"]
    sim = pgc.Simulation(p, max_outputs=4)
    got, ref = sim.state(), O.Oracle(p).state()
    sim.close()
    assert np.abs(got - ref).max() <= 1e-9 * np.abs(ref).max()
