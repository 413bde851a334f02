"""The work that users of this solver have it do, as measurable cases through its public entry points.

Every case is one of seven kinds of call, with the physical parameters of the workloads module:

  step     a running ensemble: Simulation.step (with moment records every `every` steps), then the
           records, the event counters and the state, as a program that follows a run reads them
  sweep    several ensembles of uneven size advanced together (BatchSimulation.step), then the same
  sample   a new ensemble: Simulation() samples the Fermi-Dirac state, counts its histogram and
           forms the record at t = 0
  observe  a sampled ensemble read at points z off the nodes: observables (observe_at) and the
           distribution (reconstruct_f)
  study    one degree of the stochastic-Galerkin error study (sg_error.energy_at_times, whole call)
  mcmc     Monte Carlo sampling of the random input (sg_error.mc_mc_samples, whole call)
  adjoint  the gradient of the steady current (pgc.adjoint, whole call)

`inputs` names the random inputs: det (none), gap (band gap U[0.1, 0.3] eV), width (ribbon width
6.5..7.5 nm), field (4..6 kV/cm at 7 nm) or gap_field (gap and field U[1, 10] kV/cm).
"""
import math

import numpy as np
import torch

from paper_2404_19602_gb300 import pgc, sg_error
from paper_2404_19602_gb300 import workloads as W

INPUTS = {"det": W.DET_FP64_1E4, "gap": W.GAP_UQ_1E6, "width": W.TEST2_WIDTH_1E6, "field": W.TEST2_FIELD_1E6,
          "gap_field": W.GAP_FIELD_UQ_4E6}
DEGREES = (1, 2, 3, 4, 6, 8, 10, 12, 15, 20, 25, 30)   # compiled one-dimensional degrees beside M = 5


def listed():
    return [
        # the smallest call: a few steps of a thousand particles (interactive use, unit-sized checks)
        dict(name="det_fp64_1e3", kind="step", inputs="det", M=0, N=1000, precision="fp64", splitting=0, steps=10, every=10),
        # deterministic inputs, 1e4 particles, FP64: the paper's Algorithm 1 at its smallest quoted size
        dict(name="det_fp64_1e4", kind="step", inputs="det", M=0, N=10_000, precision="fp64", splitting=0, steps=200, every=10),
        # one random input, the ordinary uncertainty run: 1e6 particles, degree 5, a record every 10 steps
        dict(name="gap_1e6", kind="step", inputs="gap", M=5, N=1_000_000, precision="fp32", splitting=0, steps=250, every=10),
        # two random inputs, the largest single run: 4e6 particles, 21 coefficients on 36 nodes
        dict(name="gap_field_4e6", kind="step", inputs="gap_field", M=5, N=4_000_000, precision="fp32", splitting=0, steps=50, every=10),
        # the FP64 reference mode of the one-input run, which results are checked against
        dict(name="gap_fp64_1e6", kind="step", inputs="gap", M=5, N=1_000_000, precision="fp64", splitting=0, steps=20, every=10),
        # ragged size, the width law with the Strang splitting, dt = 2.5 fs, dense output
        dict(name="width_strang_300007", kind="step", inputs="width", M=5, N=300_007, precision="fp32", splitting=1, steps=100, every=2),
        # the batched sweep: 32 cases, field 1..20 kV/cm x gap-interval width, uneven particle counts
        dict(name="sweep_32", kind="sweep", cases=32, n_lo=100_000, n_hi=1_000_000, steps=50, every=10),
        # a new two-input ensemble: what every run pays before its first step
        dict(name="sample_gap_field_5e5", kind="sample", inputs="gap_field", M=5, N=500_000, precision="fp32"),
        # bands over z: 400 points of the observables, and the distribution at a few z
        dict(name="observe_gap_1e6", kind="observe", inputs="gap", M=5, N=1_000_000, precision="fp32", points=400, recon=4),
        # one high degree of the error study: 1e4 particles on 21 nodes, energies at three times
        dict(name="study_width_M20", kind="study", inputs="width", M=20, N=10_000, steps=400, points=64),
        # sampling the random input: 64 deterministic ensembles of 5e4 particles, 200 steps
        dict(name="mcmc_64x5e4", kind="mcmc", inputs="width", samples=64, N=50_000, steps=200),
        # sensitivities of the steady current: forward with checkpoints and the reverse sweep
        dict(name="adjoint_gap_5e5", kind="adjoint", inputs="gap", M=5, N=500_000, precision="fp32", steps=500, ckpt=100, every=10, window=100),
    ]


def _log_int(rng, lo, hi):
    n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    return min(hi, max(lo, n | 1 if rng.random() < 0.5 else n))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "sweep", "sample", "observe", "study", "mcmc", "adjoint"])
    if kind == "step":
        inputs = rng.choice(["det", "gap", "gap", "width", "field", "gap_field", "gap_field"])
        fp64 = rng.random() < 0.3
        most = {"det": 100_000, "gap_field": 200_000 if fp64 else 4_000_000}.get(inputs, 1_000_000)
        N = _log_int(rng, 1000, most)
        M = 0 if inputs == "det" else 5
        if inputs in ("width", "field") and rng.random() < 0.4:   # the degrees of the error study, at its size
            M, N = rng.choice(DEGREES), _log_int(rng, 1000, 50_000)
        heavy = N * (36 if inputs == "gap_field" else M + 1) * (10 if fp64 else 1)
        steps = max(10, min(200, int(6e9 / heavy) // 10 * 10))
        return dict(kind=kind, inputs=inputs, M=M, N=N, precision="fp64" if fp64 else "fp32",
                    splitting=1 if rng.random() < 0.25 else 0, steps=steps, every=rng.choice([2, 5, 10]))
    if kind == "sweep":
        return dict(kind=kind, cases=rng.randint(2, 32), n_lo=_log_int(rng, 1000, 100_000), n_hi=_log_int(rng, 100_000, 1_000_000),
                    steps=rng.choice([20, 30, 50]), every=10)
    if kind == "sample":
        inputs = rng.choice(["det", "gap", "width", "field", "gap_field"])
        return dict(kind=kind, inputs=inputs, M=0 if inputs == "det" else 5, N=_log_int(rng, 1000, 500_000), precision=rng.choice(["fp32", "fp64"]))
    if kind == "observe":
        inputs = rng.choice(["gap", "width", "field", "gap_field"])
        return dict(kind=kind, inputs=inputs, M=5, N=_log_int(rng, 10_000, 500_000), precision=rng.choice(["fp32", "fp32", "fp64"]),
                    points=_log_int(rng, 8, 400), recon=rng.randint(1, 4))
    if kind == "study":
        return dict(kind=kind, inputs=rng.choice(["width", "field"]), M=rng.choice(DEGREES), N=_log_int(rng, 1000, 10_000),
                    steps=rng.choice([100, 200, 400]), points=64)
    if kind == "mcmc":
        return dict(kind=kind, inputs=rng.choice(["width", "field"]), samples=rng.randint(2, 64), N=_log_int(rng, 1000, 50_000),
                    steps=rng.choice([50, 100, 200]))
    return dict(kind=kind, inputs=rng.choice(["gap", "gap", "gap_field"]), M=5, N=_log_int(rng, 1000, 100_000), precision=rng.choice(["fp32", "fp32", "fp64"]),
                steps=rng.choice([50, 100]), ckpt=rng.choice([20, 25, 50]), every=10, window=50)


# ------------------------------------------------------------------------------------------
# the calls
# ------------------------------------------------------------------------------------------
def _params(case, seed):
    p = dict(INPUTS[case["inputs"]], N=case["N"], seed=1 + seed, precision=case.get("precision", "fp32"),
             splitting=case.get("splitting", 0))
    if "M" in case and case["inputs"] != "det":
        p.update(M=case["M"], Q1=case["M"] + 1)
    return p


def _sweep_params(case, seed):
    """Field 1..20 kV/cm x gap-interval width 0.02..0.2 eV around 0.2 eV; N log-uniform."""
    rng = np.random.default_rng(case["cases"])
    lo, hi = sorted((case["n_lo"], case["n_hi"]))
    out = []
    for j in range(case["cases"]):
        E, w = np.linspace(1000.0, 20000.0, 4)[j % 4], np.linspace(0.02, 0.2, 8)[(j // 4) % 8]
        n = int(round(float(np.exp(rng.uniform(np.log(lo), np.log(hi))))))
        out.append(W.scaled(W.GAP_UQ_1E6, eps0_lo=0.1 - w / 4.0, eps0_hi=0.1 + w / 4.0, Ex_lo=float(E), Ex_hi=float(E),
                            N=n, seed=1 + seed, stream_id=j))
    return out


def _state(sim):
    """The coefficients [2][P][N] of a Simulation, a view of its state buffer."""
    t = torch.float64 if sim.cfg.precision == pgc.PGC_FP64 else torch.float32
    return sim.state_buf.view(t).view(2, sim.P, -1)[:, :, :sim.N]


def prepare(case, seed):
    kind = case["kind"]
    st = dict(case=case, kind=kind)
    if kind == "step":
        st["sim"] = pgc.Simulation(_params(case, seed), max_outputs=20_000)
    elif kind == "sweep":
        st["batch"] = pgc.BatchSimulation(_sweep_params(case, seed), max_outputs=4_000)
    elif kind == "observe":
        st["sim"] = sim = pgc.Simulation(_params(case, seed), max_outputs=16)
        rng = np.random.default_rng(2000 + seed)
        st["z"] = rng.uniform(-1.0, 1.0, (case["points"], sim.d))
        st["zf"] = rng.uniform(-1.0, 1.0, (case["recon"], sim.d))
    else:
        st["params"] = _params(case, seed)
        st["seed"] = seed
    return st


def _records(m, sim):
    """The moment records; with deterministic inputs there is one node and no variance over z."""
    return dict(mean=m["mean"], nodes=m["nodes"]) if sim.Q == 1 else dict(mean=m["mean"], var=m["var"], nodes=m["nodes"])


def _followed(sim):
    m, c = sim.moments(), sim.counters()
    return dict(**_records(m, sim), counters=[c[k] for k in ("attempts", "changed", "rejected", "capped", "out_of_grid", "queued", "error")],
                state=_state(sim))


def run(st):
    case, kind = st["case"], st["kind"]
    if kind == "step":
        st["sim"].step(case["steps"], case["every"])
        return _followed(st["sim"])
    if kind == "sweep":
        st["batch"].step(case["steps"], case["every"])
        got = [_followed(s) for s in st["batch"].sims]
        return dict(mean=np.stack([g["mean"] for g in got]), var=np.stack([g["var"] for g in got]),
                    nodes=np.stack([g["nodes"] for g in got]), counters=np.array([g["counters"] for g in got]),
                    states=[g["state"] for g in got])
    if kind == "sample":
        sim = pgc.Simulation(st["params"], max_outputs=16)
        m = sim.moments()
        hist, nmax = sim.hist()
        state = _state(sim)
        sim.close()
        return dict(**_records(m, sim), hist=hist, nmax=nmax, state=state)
    if kind == "observe":
        obs = st["sim"].observe_at(st["z"])
        hist, top = st["sim"].reconstruct_f(st["zf"])
        return dict(obs=obs, hist=hist, top=top)
    if kind == "study":
        z, _ = sg_error.l2_rule(case["points"])
        n = case["steps"]
        return dict(energy=sg_error.energy_at_times(st["params"], case["M"], (n // 10, n // 2, n), z))
    if kind == "mcmc":
        return dict(vx=sg_error.mc_mc_samples(st["params"], case["samples"], case["N"], case["steps"], seed=1 + st["seed"]))
    value, grad = pgc.adjoint(st["params"], case["steps"], case["ckpt"], case["every"], case["window"], weights=(1.0, 0.5))
    return dict(value=value, grad=grad)


# ------------------------------------------------------------------------------------------
# what a pass cannot do without
# ------------------------------------------------------------------------------------------
def _shape(case):
    if case["inputs"] == "det" or case["kind"] == "mcmc":
        return 1, 1, 0
    if case["inputs"] == "gap_field":
        return 21, 36, 2
    return case["M"] + 1, case["M"] + 1, 1


def _per_particle_step(P, Q, d, esz, random_field):
    """One time step: the coefficients are read and the drifted ones written (each step needs the whole histogram
    of the one before); reconstruction at the nodes (sum factorisation in 2-D), cell and |k|^2 of a node, the bound."""
    recon = 4 * 342 if (P, Q) == (21, 36) else 4 * P * Q
    return (2 * P + (2 if random_field else 1)) * esz, recon + 9 * Q + 25


def work(case):
    kind = case["kind"]
    if kind == "sweep":
        n = sum(p["N"] for p in _sweep_params(case, 0))
        b, f = _per_particle_step(6, 6, 1, 4, False)
        return dict(bytes=b * n * case["steps"], flops=f * n * case["steps"])
    P, Q, d = _shape(case)
    N, esz = case["N"], 8 if case.get("precision") == "fp64" else 4
    rf = case["inputs"] in ("field", "gap_field")
    sb, sf = _per_particle_step(P, Q, d, esz, rf)
    init = 400 * Q + 4 * P * Q   # inversion of the Fermi-Dirac law per node (two evaluations of its integral), projection
    if kind == "step":
        return dict(bytes=sb * N * case["steps"], flops=sf * N * case["steps"])
    if kind == "sample":
        return dict(bytes=(2 * P * esz) * N + 4 * Q * 240 * 240, flops=(init + 4 * P * Q + 20 * Q) * N)
    if kind == "observe":
        return dict(bytes=2 * P * esz * N, flops=N * (case["points"] * (4 * P + 16) + case["recon"] * (4 * P + 6)))
    if kind == "study":
        return dict(bytes=(sb * case["steps"] + 3 * 2 * P * esz) * N, flops=N * (init + sf * case["steps"] + 3 * case["points"] * (4 * P + 16)))
    if kind == "mcmc":
        n = N * case["samples"]
        return dict(bytes=sb * n * case["steps"], flops=n * (init + sf * case["steps"]))
    # adjoint: the forward step, its replay and the reverse step (the adjoint state read and written)
    return dict(bytes=N * case["steps"] * (2 * sb + 4 * P * esz + 2 * P * esz), flops=N * (2 * init + case["steps"] * 4 * sf))


# ------------------------------------------------------------------------------------------
# the same computations in 64 bits, from the paper's formulas in plain torch
# ------------------------------------------------------------------------------------------
_C = dict(e=1.602176634e-19, hbar=6.582119569e-16, kB=8.617333262e-5, vF=1.0e6, hwO=0.1646, hwK=0.124)


def _dev():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _mulhilo(a, b):
    """High and low words of the 32-bit product a * b (int64 tensors or ints holding uint32)."""
    lo = a * (b & 0xFFFF)
    hi = a * (b >> 16) + (lo >> 16)
    return hi >> 16, ((hi & 0xFFFF) << 16) | (lo & 0xFFFF)


def _uniforms(i, stream, step, word, seed):
    """The four 24-bit uniforms of the Philox4x32-10 counter (i, stream, step, word)."""
    c = [i & 0xFFFFFFFF, torch.full_like(i, stream), torch.full_like(i, step), word if torch.is_tensor(word) else torch.full_like(i, word)]
    k0, k1 = seed & 0xFFFFFFFF, seed >> 32
    for _ in range(10):
        h0, l0 = _mulhilo(c[0], 0xD2511F53)
        h1, l1 = _mulhilo(c[2], 0xCD9E8D57)
        c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return [((x >> 8) | 1) for x in c]   # odd multiples of 2^-24


def _fd_integral(e, mu, kT):
    """int_e^inf x / (1 + exp((x - mu)/kT)) dx = kT^2 [ (e/kT) F0 + F1 ], with the Fermi-Dirac integrals F0 and F1 of
    eta = (mu - e)/kT; F1 for eta <= 0 from its alternating series (Cohen, Rodriguez Villegas and Zagier's
    acceleration), for eta > 0 by the reflection F1(eta) + F1(-eta) = pi^2/6 + eta^2/2."""
    eta = (mu - e) / kT
    x = torch.exp(-eta.abs())
    n = 40
    d = (3.0 + math.sqrt(8.0)) ** n
    d = (d + 1.0 / d) / 2.0
    b, c, s = -1.0, -d, torch.zeros_like(x)
    t = x.clone()
    for k in range(n):
        c = b - c
        s = s + c * t / float((k + 1) ** 2)
        t = t * x
        b = b * (k + n) * (k - n) / ((k + 0.5) * (k + 1))
    f1 = s / d
    f1 = torch.where(eta > 0, math.pi ** 2 / 6.0 + eta * eta / 2.0 - f1, f1)
    f0 = torch.clamp(eta, min=0.0) + torch.log1p(x)
    return kT * (e * f0 + kT * f1)


class _Exact:
    """One ensemble in FP64: Fermi-Dirac sampling, time steps, observables."""

    def __init__(self, p):
        dev = self.dev = _dev()
        t64 = dict(dtype=torch.float64, device=dev)
        self.p = p
        kT = self.kT = _C["kB"] * p["T_K"]
        self.mu, self.hvF = p["eps_F"], _C["hbar"] * _C["vF"] * 1e9
        width = (p.get("W_lo") or 0.0) > 0.0
        er = p["W_lo"] != p["W_hi"] if width else p["eps0_lo"] != p["eps0_hi"]
        fr = p["Ex_lo"] != p["Ex_hi"]
        self.d, self.M = int(er) + int(fr), p["M"]
        x, w = np.polynomial.legendre.leggauss(p["Q1"]) if self.d else (np.zeros(1), np.ones(1) * 2.0)
        w = w / 2.0
        if self.d == 2:
            z = np.array([(a, b) for a in x for b in x])
            wq = np.array([a * b for a in w for b in w])
        else:
            z, wq = x.reshape(-1, 1), w
        self.z, self.wq, self.er, self.fr, self.width = z, torch.tensor(wq, **t64), er, fr, width
        self.psi = torch.tensor(self.basis(z), **t64)                 # [Q][P]
        self.wpsi = self.psi * self.wq[:, None]
        self.eps0 = torch.tensor(self.eps0_of(z), **t64)
        E = np.full(len(z), p["Ex_lo"])
        if fr:
            E = p["Ex_lo"] + 0.5 * (p["Ex_hi"] - p["Ex_lo"]) * (z[:, -1] + 1.0)
        self.dt = p["dt_fs"]
        self.dq = torch.tensor(E * 1e-7 * self.dt / (_C["hbar"] * 1e15), **t64)
        dhat = self.wpsi.T @ self.dq
        self.dhat = torch.where(dhat.abs() > 1e-13 * dhat.abs().max(), dhat, torch.zeros_like(dhat))
        self.half = 0.5 if p["splitting"] == 1 else 0.0                # the stored state leads by half a drift
        self.Lk = p["Lk_hvF"] / self.hvF
        self.Nk = p["Nk"]
        self.dk = 2.0 * self.Lk / self.Nk
        self.nq = self.density(self.eps0)
        self.constants(kT, t64)
        self.i = torch.arange(p["N"], device=dev, dtype=torch.int64)
        self.sample()
        self.n = 0
        self.H = self.hist(self.nodes())
        self.nmax = self.H.amax(dim=1)

    def basis(self, z):
        def legendre(v):
            return np.stack([np.polynomial.legendre.Legendre.basis(h)(v) * math.sqrt(2 * h + 1) for h in range(self.M + 1)], -1)
        if self.d == 0:
            return np.ones((len(z), 1))
        if self.d == 1:
            return legendre(z[:, 0])
        a, b = legendre(z[:, 0]), legendre(z[:, 1])
        return np.stack([a[:, t - j] * b[:, j] for t in range(self.M + 1) for j in range(t + 1)], -1)

    def eps0_of(self, z):
        p, v = self.p, (z[:, 0] + 1.0) / 2.0 if self.er else np.zeros(len(z))
        if self.width:
            return math.pi * self.hvF / (p["W_lo"] + (p["W_hi"] - p["W_lo"]) * v)
        return p["eps0_lo"] + (p["eps0_hi"] - p["eps0_lo"]) * v

    def density(self, e0):
        return 2.0 / (math.pi * self.hvF ** 2) * _fd_integral(e0, self.mu, self.kT) * 1e18

    def constants(self, kT, t64):
        e, hbar = _C["e"], _C["hbar"] * _C["e"]
        sig, vp, vF = 7.6e-7, 2.0e4, _C["vF"]
        n = [1.0 / math.expm1(_C[k] / kT) for k in ("hwO", "hwK")]
        self.Cac = (6.8 * e) ** 2 * kT * e / (4 * hbar ** 3 * vF ** 2 * sig * vp ** 2) * e * 1e-15
        D = [1.0e11 * e, 3.5e10 * e]
        C = [D[k] ** 2 / (hbar ** 2 * vF ** 2 * sig * (_C[h] / _C["hbar"])) * e * 1e-15 for k, h in enumerate(("hwO", "hwK"))]
        self.COm, self.COp, self.CKm, self.CKp = C[0] * (n[0] + 1), C[0] * n[0], C[1] * (n[1] + 1), C[1] * n[1]
        V0 = 4.56e-14 * e * 1e-4
        self.Cedg = 1.0e6 * V0 ** 2 / (2 * math.pi ** 2 * hbar * (hbar * vF) ** 3) * e * e * 1e-15
        nth = self.p["n_theta"]
        self.th = torch.arange(nth + 1, **t64) * (2 * math.pi / nth)

    def sample(self):
        p, N = self.p, self.p["N"]
        u = _uniforms(self.i, p["stream_id"], 0, 0x10000, p["seed"])
        ue, ut = u[0].double() * 2.0 ** -24, u[1].double() * 2.0 ** -24
        kx, ky = [], []
        for e0 in self.eps0.tolist():
            e0t = torch.tensor([e0], dtype=torch.float64, device=self.dev)
            tot = _fd_integral(e0t, self.mu, self.kT)
            lo, hi = torch.full((N,), e0, dtype=torch.float64, device=self.dev), torch.full((N,), max(self.mu, e0) + 80 * self.kT, dtype=torch.float64, device=self.dev)
            x = torch.where(ue < 0.9, torch.sqrt(e0 * e0 + ue * 2 * tot), torch.full_like(ue, max(self.mu, e0)))
            for _ in range(100):   # safeguarded Newton on the upper tail
                r = (1.0 - ue) - _fd_integral(x, self.mu, self.kT) / tot
                lo, hi = torch.where(r < 0, x, lo), torch.where(r < 0, hi, x)
                dens = x / (1.0 + torch.exp((x - self.mu) / self.kT)) / tot
                y = x - r / dens
                y = torch.where((y >= lo) & (y <= hi), y, 0.5 * (lo + hi))
                small = (y - x).abs() <= 2e-16 * x
                x = y
                if bool(small.all()):
                    break
            km = torch.sqrt(torch.clamp(x * x - e0 * e0, min=0.0)) / self.hvF
            kx.append(km * torch.cos(2 * math.pi * ut))
            ky.append(km * torch.sin(2 * math.pi * ut))
        self.c = torch.stack([self.wpsi.T @ torch.stack(kx), self.wpsi.T @ torch.stack(ky)])   # [2][P][N]
        self.c[0] += self.half * self.dhat[:, None]

    def nodes(self, sel=None):
        c = self.c if sel is None else self.c[:, :, sel]
        return self.psi @ c[0], self.psi @ c[1]                        # [Q][n] each

    def cells(self, kx, ky, shift):
        """Cell of the node values on the grid moved by `shift` along x; -1 outside."""
        r = torch.floor((kx + (self.Lk - shift)[:, None]) / self.dk).long()
        l = torch.floor((ky + self.Lk) / self.dk).long()
        ok = (r >= 0) & (r < self.Nk) & (l >= 0) & (l < self.Nk)
        return torch.where(ok, r * self.Nk + l, torch.full_like(r, -1))

    def hist(self, k):
        H = []
        cl = self.cells(*k, self.half * self.dq)
        for q in range(len(self.eps0)):
            H.append(torch.bincount(cl[q] + 1, minlength=self.Nk ** 2 + 1)[1:])
        return torch.stack(H)

    def observables(self, k, e0, shift, n):
        kx = k[0] - shift[:, None]
        eps = torch.sqrt(self.hvF ** 2 * (kx * kx + k[1] * k[1]) + (e0 * e0)[:, None])
        vx, vy = (self.hvF * kx / eps).mean(1) * _C["vF"], (self.hvF * k[1] / eps).mean(1) * _C["vF"]
        return torch.stack([vx, vy, eps.mean(1), -_C["e"] * n * vx], 1)   # [Q][4]

    def record(self):
        v = self.observables(self.nodes(), self.eps0, self.half * self.dq, self.nq)
        m = self.wq @ v
        return v, m, self.wq @ (v * v) - m * m

    def at(self, z, chunk=8):
        out = []
        for j in range(0, len(z), chunk):
            zz = z[j:j + chunk]
            psi = torch.tensor(self.basis(zz), dtype=torch.float64, device=self.dev)
            e0 = torch.tensor(self.eps0_of(zz), dtype=torch.float64, device=self.dev)
            out.append(self.observables((psi @ self.c[0], psi @ self.c[1]), e0, self.half * (psi @ self.dhat), self.density(e0)))
        return torch.cat(out)

    def edge(self, kx, ky):
        """exp(-beta (cos th' - c)^2) on the trapezoid grid, and the rule's integral."""
        kk = kx * kx + ky * ky
        km = torch.sqrt(kk)
        c = torch.where(km > 0, kx / km, torch.ones_like(km))
        beta = 2.0 * (1.0e-10 * 1e9) ** 2 * kk
        g = torch.exp(-beta[..., None] * (torch.cos(self.th) - c[..., None]) ** 2)
        return g, torch.trapezoid(g, dx=2 * math.pi / self.p["n_theta"], dim=-1)

    def rates(self, kx, ky, e0):
        eps = torch.sqrt(self.hvF ** 2 * (kx * kx + ky * ky) + e0 * e0)
        zero = torch.zeros_like(eps)
        T = self.edge(kx, ky)[1]
        hO, hK = _C["hwO"], _C["hwK"]
        return torch.stack([self.Cac * eps, torch.where(eps - hO - e0 > 0, self.COm * (eps - hO), zero), self.COp * (eps + hO),
                            torch.where(eps - hK - e0 > 0, self.CKm * (eps - hK), zero), self.CKp * (eps + hK),
                            self.Cedg * e0 * eps * T])

    def angle(self, u, sgn):
        lo, hi, t = torch.zeros_like(u), torch.full_like(u, 2 * math.pi), 2 * math.pi * u
        for _ in range(56):
            mid = 0.5 * (lo + hi)
            up = mid + sgn * torch.sin(mid) < t
            lo, hi = torch.where(up, mid, lo), torch.where(up, hi, mid)
        return 0.5 * (lo + hi)

    def final(self, l, kx, ky, u):
        """Final states h^l of the node values, every mechanism evaluated and selected."""
        km = torch.sqrt(kx * kx + ky * ky)
        ci = torch.where(km > 0, kx / km, torch.ones_like(km))
        si = torch.where(km > 0, ky / km, torch.zeros_like(km))
        ub = u.expand_as(km)
        th = torch.where(l == 0, self.angle(u, 1.0).expand_as(km),
                         torch.where((l == 1) | (l == 2), 2 * math.pi * ub, self.angle(u, -1.0).expand_as(km)))
        dO, dK = _C["hwO"] / self.hvF, _C["hwK"] / self.hvF
        kn = km + torch.tensor([0.0, -dO, dO, -dK, dK, 0.0, 0.0], dtype=torch.float64, device=self.dev)[l]
        nx, ny = kn * (torch.cos(th) * ci - torch.sin(th) * si), kn * (torch.sin(th) * ci + torch.cos(th) * si)
        ed = l == 5
        if bool(ed.any()):
            g, _ = self.edge(kx[ed], ky[ed])
            h = 2 * math.pi / self.p["n_theta"]
            C = torch.cat([torch.zeros_like(g[:, :1]), torch.cumsum(0.5 * h * (g[:, 1:] + g[:, :-1]), 1)], 1)
            target = ub[ed] * C[:, -1]
            j = torch.searchsorted(C, target[:, None], right=True).clamp(1, g.shape[1] - 1)
            a, b = C.gather(1, j - 1)[:, 0], C.gather(1, j)[:, 0]
            phi = ((j[:, 0] - 1).double() + ((target - a) / (b - a)).clamp(0.0, 1.0)) * h
            nx[ed], ny[ed] = km[ed] * torch.cos(phi), km[ed] * torch.sin(phi)
        return nx, ny

    def step(self):
        p, a1, dt = self.p, 1.0 + self.p["alpha"], self.dt
        self.c[0] -= self.dhat[:, None]
        kx, ky = self.nodes()
        e = torch.sqrt(self.hvF ** 2 * (kx * kx + ky * ky).amax(0) + float(self.eps0.max()) ** 2)
        hO, hK = _C["hwO"], _C["hwK"]
        top = (self.Cac * e + self.COm * (e - hO).clamp(min=0) + self.COp * (e + hO) + self.CKm * (e - hK).clamp(min=0) + self.CKp * (e + hK)
               + self.Cedg * float(self.eps0.max()) * e * 2 * math.pi * 1.0001) * a1 * 1.001
        u0 = _uniforms(self.i, p["stream_id"], self.n, 0, p["seed"])[0].double() * 2.0 ** -24
        act = torch.nonzero(-torch.log(u0) < top * dt)[:, 0]
        e0, tc, cnt = self.eps0[:, None], torch.zeros(len(act), dtype=torch.float64, device=self.dev), 0
        while len(act) and cnt < p["max_coll"]:
            x, y = kx[:, act], ky[:, act]
            g = self.rates(x, y, e0.expand_as(x))                      # [6][Q][n]
            cum = torch.cumsum(g, 0)
            Gt = a1 * cum[5].amax(0)
            u = _uniforms(self.i[act], p["stream_id"], self.n, cnt, p["seed"])
            dtc = -torch.log(u[0].double() * 2.0 ** -24) / Gt
            hit = tc + dtc < dt
            act, x, y, cum, Gt, tc = act[hit], x[:, hit], y[:, hit], cum[:, :, hit], Gt[hit], (tc + dtc)[hit]
            if not len(act):
                break
            u = [v[hit] for v in u]
            target = u[1].double() * 2.0 ** -24 * Gt
            l = (target >= cum).sum(0)                                 # 6: self scattering
            nx, ny = self.final(l, x, y, u[3].double() * 2.0 ** -24)
            cl = self.cells(nx + self.dq[:, None], ny, self.half * self.dq)
            Hc = self.H.gather(1, cl.clamp(min=0))
            free = (cl < 0) | (self.nmax[:, None] == 0) | (Hc * 2 ** 24 < u[2] * self.nmax[:, None])
            ch = (l < 6) & (free if p["pauli_norm"] != 2 else torch.ones_like(free))
            x, y = torch.where(ch, nx, x), torch.where(ch, ny, y)
            any_ = ch.any(0)
            ia, xa, ya = act[any_], x[:, any_], y[:, any_]
            if len(ia):
                self.c[0][:, ia], self.c[1][:, ia] = self.wpsi.T @ xa, self.wpsi.T @ ya
                kx[:, ia], ky[:, ia] = self.nodes(ia)
            cnt += 1
        self.H = self.hist((kx, ky))
        self.n += 1

    def run(self, steps, every):
        rec = [self.record()]
        for _ in range(steps):
            self.step()
            if every and self.n % every == 0:
                rec.append(self.record())
        v, m, s = (torch.stack(x).cpu().numpy() for x in zip(*rec))
        return dict(mean=m, var=s, nodes=v)


def exact(case, seed):
    """The floating outputs of run() in 64 bits; None where they take too long (many ensembles, many nodes and steps)."""
    kind = case["kind"]
    if kind in ("sweep", "mcmc"):
        return None
    P, Q, _ = _shape(case)
    steps = 0 if kind in ("sample", "observe") else case["steps"]
    if case["N"] * Q * steps > 8e9 or (steps > 0 and steps * 0.03 > 20):
        return None
    if kind == "study":
        s, z = _Exact(_params(case, seed)), sg_error.l2_rule(case["points"])[0][:, None]
        out = []
        for k in range(steps):
            s.step()
            if k + 1 in (steps // 10, steps // 2, steps):
                out.append(s.at(z)[:, 2].cpu().numpy())
        return dict(energy=np.array(out))
    s = _Exact(_params(case, seed))
    if kind == "observe":
        rng = np.random.default_rng(2000 + seed)
        return dict(obs=s.at(rng.uniform(-1.0, 1.0, (case["points"], s.d))).cpu().numpy(), hist=None, top=None)
    got = s.run(steps, case.get("every", 0))
    if kind == "adjoint":
        at = [n for n in range(0, steps + 1, case["every"]) if n > steps - case["window"]]
        J = got["mean"][[n // case["every"] for n in at], 3].mean(), got["var"][[n // case["every"] for n in at], 3].mean()
        return dict(value=np.array(J), grad=None)
    # FP32 rounding now and then flips a decision at a node, and such a particle goes its own way: after many
    # node decisions the coefficients say no more about accuracy (the moments do)
    decisions = steps * Q * s.dt if case["precision"] == "fp32" else 0
    got["state"] = s.c if decisions <= 2000 else None
    if Q == 1:
        del got["var"]
    if kind == "step":
        got["counters"] = None
    else:
        got.update(hist=None, nmax=None)
    return got
