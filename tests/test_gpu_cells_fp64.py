"""The FP64 mode's histogram cells, taken in FP32 where FP32 is certain of them, against a numpy count of
the stored state: grids of one to many windows, odd sizes, node values outside the grid, both
splittings, and uploaded states of which every node value lies within the FP32 rounding of a cell edge
(1e-8 to 1e-7 of a cell on either side), so that each is decided by the FP64 path.

A value within 1e-9 cells of an edge may fall on either side: the node value carries ~30 FP64 roundings of
numbers of order one (1e-14 nm^-1, 1e-12 cells); everything else is exact."""
import numpy as np
import pytest

from paper_2404_19602_gb300 import workloads as W
from test_gpu_window_paths import BASE, _psi

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

EDGE = 1e-9
GRIDS = [(5, 5.0), (31, 5.0), (48, 2.0), (57, 1.5), (240, 5.0), (241, 0.45), (601, 5.0), (1000, 1.2)]


def _check(sim, p):
    H, _ = sim.hist()
    c = sim.state()
    psi, _ = _psi(p, sim.P)
    Lk = p["Lk_hvF"] / (6.582119569e-16 * 1e6 * 1e9)
    dk = 2 * Lk / p["Nk"]
    yx, yy = (psi @ c[0] + Lk) / dk, (psi @ c[1] + Lk) / dk
    for q in range(sim.Q):
        r, l = np.floor(yx[q]).astype(int), np.floor(yy[q]).astype(int)
        ok = (r >= 0) & (r < p["Nk"]) & (l >= 0) & (l < p["Nk"])
        ref = np.zeros((p["Nk"], p["Nk"]), dtype=np.int64)
        np.add.at(ref, (r[ok], l[ok]), 1)
        near = ((np.abs(yx[q] - np.rint(yx[q])) < EDGE) | (np.abs(yy[q] - np.rint(yy[q])) < EDGE)).sum()
        assert np.abs(H[q].astype(np.int64) - ref).sum() <= 2 * near, q


@pytest.mark.parametrize("Nk,Lk", GRIDS)
@pytest.mark.parametrize("shape", list(BASE))
@pytest.mark.parametrize("splitting", [0, 1])
def test_fp64_histogram_equals_count_of_the_state(shape, Nk, Lk, splitting):
    from paper_2404_19602_gb300 import build, pgc

    build.build()
    base, kw = BASE[shape]
    for N in (1, 1501):
        p = W.scaled(base, N=N, Nk=Nk, Lk_hvF=Lk, precision="fp64", splitting=splitting, seed=3, **kw)
        sim = pgc.Simulation(p, max_outputs=4)
        for steps in (1, 2):
            sim.step(steps, 0)
            _check(sim, p)
        sim.close()


@pytest.mark.parametrize("Nk", [48, 240, 1000])
@pytest.mark.parametrize("shape", list(BASE))
def test_fp64_values_next_to_cell_edges(shape, Nk):
    """Node values 1e-8 to 1e-7 of a cell beside an edge (below the resolution of FP32 at these grids)."""
    from paper_2404_19602_gb300 import build, pgc

    build.build()
    base, kw = BASE[shape]
    p = W.scaled(base, N=2003, Nk=Nk, precision="fp64", seed=3, mech_mask=0, Ex_lo=0.0, Ex_hi=0.0 if shape != "21x36" else 1e-9, **kw)
    if shape == "21x21":   # the field is this workload's random input
        p.update(W_lo=6.5, W_hi=7.5)
    sim = pgc.Simulation(p, max_outputs=4)
    Lk = p["Lk_hvF"] / (6.582119569e-16 * 1e6 * 1e9)
    dk = 2 * Lk / Nk
    rng = np.random.default_rng(Nk)
    k = np.zeros((2, sim.P, p["N"]))
    cells = rng.integers(-3, Nk + 4, (2, p["N"]))
    k[:, 0] = cells * dk - Lk + rng.choice([-1, 1], (2, p["N"])) * 10.0 ** rng.uniform(-8, -7, (2, p["N"])) * dk
    sim.set_state(k)
    sim.step(1, 0)
    _check(sim, p)
    sim.close()
