"""The sampled state and the record at t = 0 of an ensemble whose law does not depend on z: with the
field as the only random input every node has the same band minimum, so the coefficients above the
mean and the record's variance over z are the rounding of the sampler and of the sums alone.  They are
outputs all the same and are kept bit for bit: golden values of the node-by-node sampler
(tests/golden/sampled_field_fp64.txt), at a ragged size, one beyond the observation grid, a large
one-dimensional shape and the Strang splitting."""
import hashlib
import os

import numpy as np
import pytest

from paper_2404_19602_gb300 import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

GOLDEN = [line.split() for line in open(os.path.join(os.path.dirname(__file__), "golden", "sampled_field_fp64.txt"))
          if not line.startswith("#")]


@pytest.mark.parametrize("row", GOLDEN, ids=lambda r: "-".join(r[:3]))
def test_sampled_state_and_record_bit_for_bit(row):
    from paper_2404_19602_gb300 import build, pgc

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build.build()
    shape, N, splitting, state = row[0], int(row[1]), int(row[2]), row[3]
    values, nodes = [float.fromhex(v) for v in row[4:12]], row[12]
    M = int(shape.split("x")[0]) - 1
    p = W.scaled(W.TEST2_FIELD_1E6, N=N, precision="fp64", seed=7, splitting=splitting, M=M, Q1=M + 1)
    sim = pgc.Simulation(p, max_outputs=4)
    m, k = sim.moments(), sim.state()
    sim.close()
    assert hashlib.sha256(np.ascontiguousarray(k).tobytes()).hexdigest() == state
    assert np.concatenate([m["mean"][0], m["var"][0]]).tolist() == values
    assert hashlib.sha256(np.ascontiguousarray(m["nodes"][0]).tobytes()).hexdigest() == nodes


def test_fp32_record_is_accumulated_in_fp64():
    """The warp sums of an FP32 state's record are accumulated in FP64: two energies 2^24 apart, constant over
    each warp's 32 particles, whose sum of 51 bits comes out exactly (it does not from pairs of FP32
    numbers)."""
    from fractions import Fraction

    from paper_2404_19602_gb300 import build, pgc

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build.build()
    N, big = 1 << 20, 4.0e6   # nm^-1
    p = W.scaled(W.DET_FP64_1E4, precision="fp32")

    def energy(k):
        sim = pgc.Simulation(dict(p, N=k.shape[2]), init_khat=k, max_outputs=4)
        e = sim.moments()["nodes"][0, 0, 2]
        sim.close()
        return float(e)

    one = np.zeros((2, 1, 1))
    ea = energy(one)
    one[0] = big
    eb = energy(one)
    assert np.float32(ea) == ea and np.float32(eb) == eb and 2 ** 21 < eb < 2 ** 22
    chunks = np.random.default_rng(5).choice(N // 32, 8, replace=False)
    k = np.zeros((2, 1, N))
    k[0, 0].reshape(-1, 32)[chunks] = big
    exact = Fraction(ea) * (N - 8 * 32) + Fraction(eb) * (8 * 32)
    assert exact == Fraction(float(exact))   # 51 bits: FP64 holds it and every partial sum
    assert energy(k) == float(exact) / N
