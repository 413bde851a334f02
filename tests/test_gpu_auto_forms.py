"""Launch forms and event counts that the library chooses by itself: the fused form that
unrecorded calls of the larger one-dimensional shapes take equals the two-launch form bit for bit
(states, histograms, counters), and the adjoint of particles with more events in a step than it
keeps equals the oracle's tangents.

Tolerances: the two forms do the same arithmetic per particle, so equality is exact.  The adjoint
case has about 35 events per particle in all; FP64 rounding is carried through them without growth
beyond the number of events, so the bounds of the short-step adjoint tests (1e-9 for the values,
1e-6 of the largest component for the gradients) hold here too."""
import numpy as np
import pytest

import oracle as O
from paper_2404_19602_gb300 import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2404_19602_gb300 import build

    build.build()
    O.build()


@pytest.mark.parametrize("M", [8, 12, 20, 30])
@pytest.mark.parametrize("N", [1, 517, 30001, 200000, 200001])
def test_unrecorded_steps_equal_two_launch_form(M, N):
    from paper_2404_19602_gb300 import pgc

    out = []
    for two_launches in (False, True):
        s = pgc.Simulation(W.scaled(W.TEST2_FIELD_1E6, M=M, Q1=M + 1, N=N), max_outputs=8)
        if two_launches:
            s.set_pipeline(False)
        for steps, every in ((7, 0), (1, 0), (4, 2), (6, 0)):   # unrecorded, single, recorded, unrecorded
            s.step(steps, every)
        out.append((s.state(), s.hist()[0], s.counters(), s.moments()["mean"]))
        s.close()
    a, b = out
    assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1]) and a[2] == b[2]
    assert np.allclose(a[3], b[3], rtol=1e-12, atol=1e-12 * np.abs(b[3]).max())   # FP64 sums of FP32 block partials


@pytest.mark.parametrize("name", ["det", "gap", "gap_field"])
def test_adjoint_with_many_events_per_step(name):
    from paper_2404_19602_gb300 import pgc

    base, N = {"det": (W.DET_FP64_1E4, 800), "gap": (W.GAP_UQ_1E6, 800), "gap_field": (W.GAP_FIELD_UQ_4E6, 150)}[name]
    p = W.scaled(base, N=N, precision="fp64", dt_fs=600.0)   # 2 to 6 events per particle and step on average
    val_o, grad_o = O.Oracle(p).tangent_run(6, 1, 3)
    val, grad = pgc.adjoint(p, 6, 4, 1, 3, weights=[1.0, 0.0])
    assert np.allclose(val, val_o, rtol=1e-9, atol=1e-9 * abs(val_o[0])), (val, val_o)
    assert np.abs(grad - grad_o[0]).max() <= 1e-6 * np.abs(grad_o[0]).max(), (grad, grad_o[0])
