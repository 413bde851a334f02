"""Grids of fewer cells than the shared-memory histogram window (which then holds the whole grid): the
histograms of the step, of the observation of an uploaded state and of the batched step against a numpy
count, most node values inside and some outside the grid, and the time of a step against that on a
grid larger than the window."""
import pytest

from paper_2404_19602_gb300 import workloads as W
from test_gpu_step_times import _step_us
from test_gpu_window_paths import BASE, _check

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

GRIDS = [(2, 5.0), (7, 1.0), (16, 5.0), (31, 0.9), (39, 5.0), (55, 5.0)]


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2404_19602_gb300 import build

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build.build()


@pytest.mark.parametrize("Nk,Lk", GRIDS)
@pytest.mark.parametrize("shape", list(BASE))
@pytest.mark.parametrize("splitting", [0, 1])
def test_histogram_on_small_grids(shape, Nk, Lk, splitting):
    from paper_2404_19602_gb300 import pgc

    base, kw = BASE[shape]
    for N in (1, 1501):
        p = W.scaled(base, N=N, Nk=Nk, Lk_hvF=Lk, precision="fp32", splitting=splitting, seed=3, **kw)
        sim = pgc.Simulation(p, max_outputs=4)
        _check(sim, p)
        sim.step(1, 0)
        _check(sim, p)
        sim.step(2, 0)
        _check(sim, p)
        sim.set_state(sim.state())
        _check(sim, p)
        sim.close()


@pytest.mark.parametrize("Nk,Lk", GRIDS)
@pytest.mark.parametrize("shape", ["1x1", "6x6", "21x36"])
def test_batched_histogram_on_small_grids(shape, Nk, Lk):
    from paper_2404_19602_gb300 import pgc

    base, kw = BASE[shape]
    cases = [W.scaled(base, N=N, Nk=Nk, Lk_hvF=Lk, precision="fp32", seed=3, stream_id=j, **kw) for j, N in enumerate((777, 1, 4099))]
    b = pgc.BatchSimulation(cases, max_outputs=4)
    b.step(3, 0, use_graph=False)
    for s, p in zip(b.sims, cases):
        _check(s, p)
    b.close()


@pytest.mark.parametrize("base,N", [(W.GAP_UQ_1E6, 1_000_000), (W.GAP_FIELD_UQ_4E6, 200_000)], ids=["6x6", "21x36"])
def test_step_time_on_a_small_grid(base, N):
    """40 cells against 64: at most half as long again (5 and 2.6 times without a window)."""
    from paper_2404_19602_gb300 import pgc

    us = []
    for Nk in (64, 40):
        sim = pgc.Simulation(W.scaled(base, N=N, Nk=Nk), max_outputs=4)
        us.append(_step_us(sim))
        sim.close()
    print(us)
    assert us[1] <= 1.5 * us[0]
