"""The streaming kernels' histogram paths (shared-memory window, particles put aside, global cells,
outside the grid) against a numpy count of the stored state: grids smaller than, equal to and
larger than the window, odd sizes, a grid so narrow that most particles leave the window's circle,
ragged ensembles, both splittings, the batched kernel.

A node value within 1e-3 cells of a cell edge may fall on either side in FP32 (the rounding of the
cell is below 1e-4 cells at these grid sizes), so the counts of a node may differ by at most two
per such value; everything else is exact, and counts plus particles outside the grid equal N."""
import numpy as np
import pytest

from paper_2404_19602_gb300 import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

BASE = {"1x1": (W.DET_FP64_1E4, {}), "6x6": (W.GAP_UQ_1E6, {}), "21x36": (W.GAP_FIELD_UQ_4E6, {}),
        "21x21": (W.TEST2_FIELD_1E6, dict(M=20, Q1=21)), "31x31": (W.TEST2_WIDTH_1E6, dict(M=30, Q1=31))}


def _psi(p, P):
    if p["M"] == 0:
        return np.ones((1, 1)), np.zeros(1)
    x, _ = np.polynomial.legendre.leggauss(p["Q1"])
    leg = np.stack([np.polynomial.legendre.Legendre.basis(h)(x) * np.sqrt(2 * h + 1) for h in range(p["M"] + 1)], -1)
    if P == p["M"] + 1:
        return leg, x
    psi = [[leg[a, t - j] * leg[b, j] for t in range(p["M"] + 1) for j in range(t + 1)] for a in range(len(x)) for b in range(len(x))]
    return np.array(psi), np.tile(x, len(x))


def _check(sim, p):
    H, _ = sim.hist()
    c = sim.state()   # at the step boundary
    psi, _ = _psi(p, sim.P)
    kx, ky = psi @ c[0], psi @ c[1]
    Lk = p["Lk_hvF"] / (6.582119569e-16 * 1e6 * 1e9)
    dk = 2 * Lk / p["Nk"]
    yx, yy = (kx + Lk) / dk, (ky + Lk) / dk
    out_total = 0
    for q in range(sim.Q):
        r, l = np.floor(yx[q]).astype(int), np.floor(yy[q]).astype(int)
        ok = (r >= 0) & (r < p["Nk"]) & (l >= 0) & (l < p["Nk"])
        ref = np.zeros((p["Nk"], p["Nk"]), dtype=np.int64)
        np.add.at(ref, (r[ok], l[ok]), 1)
        near = ((np.abs(yx[q] - np.rint(yx[q])) < 1e-3) | (np.abs(yy[q] - np.rint(yy[q])) < 1e-3)).sum()
        assert np.abs(H[q].astype(np.int64) - ref).sum() <= 2 * near, q
        assert H[q].sum() <= p["N"]
        out_total += p["N"] - int(H[q].sum())
    return out_total


GRIDS = [(240, 5.0), (241, 5.0), (47, 2.0), (48, 2.0), (57, 1.5), (240, 1.2), (64, 0.45)]


@pytest.mark.parametrize("Nk,Lk", GRIDS)
@pytest.mark.parametrize("shape", list(BASE))
@pytest.mark.parametrize("splitting", [0, 1])
def test_histogram_equals_count_of_the_state(shape, Nk, Lk, splitting):
    from paper_2404_19602_gb300 import build, pgc

    build.build()
    base, kw = BASE[shape]
    for N in (1, 517, 3001):
        p = W.scaled(base, N=N, Nk=Nk, Lk_hvF=Lk, precision="fp32", splitting=splitting, seed=3, **kw)
        sim = pgc.Simulation(p, max_outputs=4)
        out = 0
        for steps in (1, 3):
            before = sim.counters()["out_of_grid"]
            sim.step(steps, 0)
            if steps == 1:
                out = _check(sim, p)
                assert sim.counters()["out_of_grid"] - before == out
            else:
                _check(sim, p)
        sim.close()


@pytest.mark.parametrize("Nk,Lk", GRIDS)
@pytest.mark.parametrize("shape", ["1x1", "6x6", "21x36"])
def test_batched_histogram_equals_count_of_the_state(shape, Nk, Lk):
    from paper_2404_19602_gb300 import build, pgc

    build.build()
    base, kw = BASE[shape]
    cases = [W.scaled(base, N=N, Nk=Nk, Lk_hvF=Lk, precision="fp32", seed=3, stream_id=j, **kw) for j, N in enumerate((777, 1, 4099))]
    b = pgc.BatchSimulation(cases, max_outputs=4)
    b.step(3, 0, use_graph=False)
    for s, p in zip(b.sims, cases):
        _check(s, p)
    b.close()


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("shape", ["1x1", "6x6", "21x36", "21x21"])
def test_non_finite_and_huge_states_leave_the_others_alone(shape, precision):
    """NaN, infinite and huge coefficients (an uploaded state may hold any): every count of the finite
    particles is as without them, and a bad particle is counted at most once per node."""
    from paper_2404_19602_gb300 import build, pgc

    build.build()
    base, kw = BASE[shape]
    N = 700
    p = W.scaled(base, N=N, precision=precision, mech_mask=0, seed=3, **kw)
    sim = pgc.Simulation(p, max_outputs=4)
    good = sim.state()
    sim.close()
    far = good.copy()
    bad = np.arange(5, N, 61)
    far[:, :, bad] = 0.0
    far[0, 0, bad] = 1e3          # outside the grid, finite
    vals = [np.nan, np.inf, -np.inf, 1e30, -1e30, 3e38, -6.3e6, 6.3e6]
    ugly = far.copy()
    for j, i in enumerate(bad):
        ugly[j % 2, j % good.shape[1], i] = vals[j % len(vals)]
    hists = []
    for state in (far, ugly):
        s = pgc.Simulation(p, init_khat=good, max_outputs=4)
        s.set_state(state)
        s.step(1, 0)
        hists.append(s.hist()[0].astype(np.int64))
        s.close()
    extra = hists[1] - hists[0]
    assert extra.min() >= 0 and (extra.sum(axis=(1, 2)) <= len(bad)).all()
