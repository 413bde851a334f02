"""The rounding of an FP32 record is fixed (the contraction of the observables is written out, since the
compiler's choice follows the code around it): the record of the first step of small ensembles, whose
mean over a thousand particles shows it, equals golden values bit for bit
(tests/golden/record_rounding_fp32.txt)."""
import os

import numpy as np
import pytest

from paper_2404_19602_gb300 import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

BASE = {"width": W.TEST2_WIDTH_1E6, "field": W.TEST2_FIELD_1E6, "gap": W.GAP_UQ_1E6}
GOLDEN = [line.split() for line in open(os.path.join(os.path.dirname(__file__), "golden", "record_rounding_fp32.txt"))
          if not line.startswith("#")]


@pytest.mark.parametrize("row", GOLDEN, ids=lambda r: "-".join(r[:3]))
def test_record_bit_for_bit(row):
    from paper_2404_19602_gb300 import build, pgc

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build.build()
    M, N = int(row[1]), int(row[2])
    sim = pgc.Simulation(W.scaled(BASE[row[0]], N=N, M=M, Q1=M + 1, seed=7, precision="fp32"), max_outputs=4)
    sim.step(1, 1)
    m = sim.moments()
    sim.close()
    assert np.concatenate([m["mean"][1], m["var"][1]]).tolist() == [float.fromhex(v) for v in row[3:]]
