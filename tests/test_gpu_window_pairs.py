"""The histogram window's words hold two nodes of 16 bits each: an ensemble of which every streaming
block counts more than 2^16 particles, both nodes of the pair in the same cell, so that neither half may
carry into the other or wrap before the flush; a share of the particles lies outside the circle of
the window but inside its square (put aside, counted 32 at a time, also across a flush), a share outside
the window, and a share outside the grid.  All counts exact, in the fused and the two-launch form."""
import numpy as np
import pytest

from paper_2404_19602_gb300 import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("pipelined", [True, False])
def test_pair_counts_past_16_bits(pipelined):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2404_19602_gb300 import build, pgc

    build.build()
    N = 1 << 25          # ~74k particles per streaming block at 456 blocks
    p = W.scaled(W.GAP_UQ_1E6, N=N, M=1, Q1=2, mech_mask=0, Ex_lo=0.0, Ex_hi=0.0)
    Lk = p["Lk_hvF"] / 0.6582119569
    dk = 2 * Lk / p["Nk"]
    # cell offsets from the middle: one hot cell, the corner of the 48 x 48 window, beyond the window, outside the grid
    places = [(3, -2), (22, 22), (60, -40), (300, 0)]
    kind = np.zeros(N, dtype=np.int64)
    kind[7::61] = 1
    kind[11::97] = 2
    kind[13::101] = 3
    k = np.zeros((2, 2, N))
    for j, (r, l) in enumerate(places):
        k[0, 0, kind == j] = (r + 0.5) * dk
        k[1, 0, kind == j] = (l + 0.5) * dk
    sim = pgc.Simulation(p, init_khat=k, max_outputs=8)
    sim.set_pipeline(pipelined)
    count = np.bincount(kind, minlength=4)
    ref = np.zeros((2, p["Nk"], p["Nk"]), dtype=np.int64)
    for j, (r, l) in enumerate(places[:3]):
        ref[:, 120 + r, 120 + l] = count[j]
    for steps in (1, 3):
        before = sim.counters()["out_of_grid"]
        sim.step(steps, 0)
        assert np.array_equal(sim.hist()[0], ref)
        assert sim.counters()["out_of_grid"] - before == steps * 2 * count[3]
    sim.close()
