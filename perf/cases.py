"""The work whose speed this repository is measured by: Krotov iterations, gradients and their variants.

Each case is one pass of a user's program through the public entry points.  A Krotov pass sets a
guess pulse, propagates it (the guess sweep) and runs Krotov iterations (backward co-state sweep and
updating forward sweep); a gradient pass evaluates J_T and its gradient through torch.autograd.  The
models, time steps, precisions and trajectory counts are those of the workloads in synth_inputs.py
(d = 36 ... 6561, 1 ... 1024 trajectories); the time windows of the larger ones are cut to what a
pass can take, with the workload's own time step.  Windows start from the chain's initial state
|e g..g> with a share ``upper`` of the first atom in its upper level (the e-r coherence that a pulse
leaves when it is not followed adiabatically; without it the update nearly cancels) and, where
trajectories jump, a photon in flight in the second cavity.  A share ``jumps`` of the trajectories
draws a threshold that the photon's decay crosses: a few per cent jump inside the window, as in the
middle of a run.  Or they start from random states of the full space (``random_init``), where every
trajectory jumps, some several times.

FP32-mixed problems hold their states in complex64; their results are handed on as 32-bit values.
"""
from __future__ import annotations

import math

import numpy as np
import torch

DELTA = 100.0          # detuning of the atoms' upper level, units of the cavity coupling


# ----------------------------------------------------------------------------------- the cases
def _case(kind, n_nodes, n_cav, m, nt, dt, precision, **more):
    c = dict(kind=kind, n_nodes=n_nodes, n_cav=n_cav, m=m, nt=nt, dt=dt, precision=precision, amp=1.0, kappa=1.0,
             jumps=0.0, upper=0.1, random_init=False, local=False, first_order=False, ckpt=0, iters=1)
    c.update(more)
    return c


def listed():
    return [
        # the smallest workload in full: two nodes, one photon, 32 trajectories, FP64, T = 50
        dict(_case("krotov", 2, 1, 32, 500, 0.1, "fp64"), name="krotov_d36_m32_fp64"),
        # one trajectory of the two-photon chain in full: latency alone
        dict(_case("krotov", 2, 2, 1, 1000, 0.05, "fp64", jumps=1.0), name="krotov_d81_m1_fp64"),
        # the two-photon chain with 128 trajectories, FP32-mixed, two iterations
        dict(_case("krotov", 2, 2, 128, 100, 0.05, "fp32", jumps=0.05, iters=2), name="krotov_d81_m128_fp32"),
        # the same in FP64 from random states with a detector on each cavity: several jumps per trajectory
        dict(_case("krotov", 2, 2, 128, 80, 0.05, "fp64", amp=30.0, random_init=True, local=True),
             name="krotov_d81_m128_fp64_jumps"),
        # three nodes, one photon, an odd number of trajectories, co-states checkpointed
        dict(_case("krotov", 3, 1, 333, 101, 0.025, "fp32", jumps=0.05, ckpt=12), name="krotov_d216_m333_fp32_ckpt"),
        # three nodes, two photons: the differentiation workload's model under Krotov iterations
        dict(_case("krotov", 3, 2, 1024, 100, 0.025, "fp32", jumps=0.03), name="krotov_d729_m1024_fp32"),
        # the same model in FP64
        dict(_case("krotov", 3, 2, 100, 40, 0.025, "fp64", jumps=0.05), name="krotov_d729_m100_fp64"),
        # the largest workload: four nodes, two photons, 1024 trajectories
        dict(_case("krotov", 4, 2, 1024, 80, 0.01, "fp32", jumps=0.02), name="krotov_d6561_m1024_fp32"),
        # J_T and its gradient through torch.autograd, the differentiation workload
        dict(_case("gradient", 3, 2, 1024, 60, 0.025, "fp32", jumps=0.03), name="gradient_d729_m1024_fp32"),
        # the cross-trajectory update (all pairs of trajectories)
        dict(_case("cross", 2, 2, 128, 100, 0.05, "fp32", jumps=0.05), name="cross_d81_m128_fp32"),
        # the density matrix the trajectory results are compared with
        dict(_case("density", 2, 2, 1, 60, 0.05, "fp32", jumps=0.03), name="density_d81_fp32"),
        # independent problems of mixed sizes iterated together
        dict(_case("batch", 4, 2, 512, 60, 0.025, "fp32", jumps=0.02, problems=12), name="batch_mix12_fp32"),
    ]


# time step of the workload with this many nodes
_DT = {1: 0.1, 2: 0.05, 3: 0.025, 4: 0.01}
_MODELS = [(1, 2), (2, 1), (2, 2), (2, 2), (2, 3), (3, 1), (3, 2), (3, 2), (4, 1), (4, 2)]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    for _ in range(1000):
        kind = rng.choice(["krotov"] * 6 + ["gradient"] * 2 + ["cross", "density", "batch"])
        n, nc = rng.choice(_MODELS)
        prec = rng.choice(["fp32", "fp32", "fp64"])
        m, nt = _log_int(rng, 1, 1024), _log_int(rng, 20, 250 if prec == "fp64" else 100)
        more = dict(amp=rng.choice([1.0, 5.0, 20.0] if prec == "fp64" else [1.0, 2.0, 5.0]), kappa=round(rng.uniform(0.5, 2.0), 3),
                    jumps=rng.choice([0.0, 0.02, 0.05] if m > 8 else [0.0, 1.0]),
                    upper=rng.choice([0.1, 0.2]), iters=rng.choice([1, 1, 2]))
        if kind == "krotov":
            more.update(random_init=n <= 2 and prec == "fp64" and rng.random() < 0.25, local=rng.random() < 0.25,
                        first_order=rng.random() < 0.2, ckpt=rng.choice([0, 0, 0, 7, 16]))
        elif kind == "gradient":
            more.update(ckpt=rng.choice([0, 0, 11]), iters=1)
            n, nc = rng.choice([(2, 1), (2, 2), (3, 1), (3, 2)])
        elif kind == "cross":
            n, nc = rng.choice([(2, 1), (2, 2), (3, 1)])
            m = min(m, 300)
        elif kind == "density":
            n, nc, m = rng.choice([(1, 2, 1), (2, 1, 1), (2, 2, 1)])
        else:
            n, nc, m, nt, prec = 4, 2, min(m, 512), max(20, nt // 4), "fp32"
            more.update(problems=rng.randint(3, 10), iters=1)
        c = _case(kind, n, nc, m, nt, _DT[n], prec, **more)
        if _cost(c) <= _cost(listed()[7]):
            return c
    raise RuntimeError("no case within the cost bound")


def _cost(c):
    """What a pass takes, roughly: flops, FP64 ones weighted by their rate, and an interval's latency."""
    if c["kind"] == "batch":
        return sum(_cost(s) for s in _subproblems(c, 0))
    weight = 30.0 if c["precision"] == "fp64" else 1.0
    jumps = 4.0 if c["random_init"] else 1.0
    wide = 40.0 if c["kind"] == "density" else 1.0          # a density matrix is one state
    return c["iters"] * (jumps * weight * wide * work(c)["flops"] + 2e8 * c["nt"])


# ---------------------------------------------------------------------------------- the inputs
def _sweeps(c):
    return 1 + 2 * c["iters"] if c["kind"] != "gradient" else 4


def _draws(c):
    return 1 + 2 * (c["n_nodes"] * (1 + c["n_cav"]) + 1)


def _pulse(c, seed):
    rng = np.random.default_rng(seed + 1)
    x = (np.arange(c["nt"]) + 0.5) / c["nt"]
    shape = np.tile(np.sin(np.pi * x) ** 2, (c["n_nodes"], 1))
    wave = np.zeros_like(shape)
    for i in range(c["n_nodes"]):
        for k in range(1, 4):
            wave[i] += 0.2 * rng.normal() * np.sin(math.pi * k * x)
    return c["amp"] * (shape + 0.5 * np.tanh(wave)), shape


def _uniforms(c, seed):
    """Thresholds and channel draws.  A threshold that equals the norm at which a trajectory has lost its
    photons and decays no further leaves its jump time to the last bits of that norm; the first thresholds
    keep clear of it: a share ``jumps`` lies in the first 60 % of the photon's decay, the others a tenth
    below what is left of the norm (random states: above 0.15); the later thresholds, for the freshly
    normalised state, lie below 0.98."""
    u = np.random.default_rng(seed).random((1 + c["iters"], c["m"], _draws(c)))
    u[:, :, 2::2] *= 0.98
    if c["random_init"]:
        u[:, :, 0] = 0.15 + 0.85 * u[:, :, 0]
    else:
        q, w, r = c["jumps"], _photon(c), u[:, :, 0]
        u[:, :, 0] = np.where(r < q, 1.0 - 0.6 * w * r / max(q, 1e-9), 0.9 * (1.0 - w) * (r - q) / max(1.0 - q, 1e-9))
    return u


def _photon(c):
    return 0.3 if c["jumps"] > 0.0 else 0.0


def _psi0(c):
    """The first atom in e and (share ``upper``) r, the others in g, no photon; where trajectories jump,
    weight 0.3 on the first atom in e and one photon in the second cavity."""
    n, nl = c["n_nodes"], 3 * (c["n_cav"] + 1)
    v = np.zeros(nl ** n, dtype=np.complex128)
    e = (c["n_cav"] + 1) * nl ** (n - 1)
    v[e] = math.sqrt((1.0 - _photon(c)) * (1.0 - c["upper"]))
    v[2 * e] = math.sqrt((1.0 - _photon(c)) * c["upper"])
    v[e + (nl ** (n - 2) if n > 1 else 1)] = math.sqrt(_photon(c))
    return v


def _random_states(c, seed):
    rng = np.random.default_rng(seed + 2)
    shape = (c["m"], (3 * (c["n_cav"] + 1)) ** c["n_nodes"])
    z = rng.normal(size=shape) + 1j * rng.normal(size=shape)
    return z / np.linalg.norm(z, axis=1, keepdims=True)


def _subproblems(c, seed):
    """The problems of a batch: networks of two to four nodes, trajectory counts over a factor of eight."""
    rng = np.random.default_rng(77)
    out = []
    for i in range(c["problems"]):
        n = (2, 3, 4)[i % 3]
        m = max(1, c["m"] >> int(rng.integers(0, 4)))
        m = min(m, 256) if n == 4 else m
        out.append(_case("krotov", n, 2, m, c["nt"] * int(rng.integers(1, 3)), _DT[n], c["precision"], amp=c["amp"],
                         kappa=round(float(rng.uniform(0.5, 2.0)), 3), jumps=c["jumps"], upper=c["upper"]))
    return out


def _spec(c, seed):
    from paper_1801_04382_gb300 import cascaded_chain
    eps, shape = _pulse(c, seed)
    net = cascaded_chain(c["n_nodes"], c["n_cav"], kappa=c["kappa"], lindblad="local" if c["local"] else "collective")
    net.psi0 = _psi0(c)
    spec = dict(net=net, T=c["nt"] * c["dt"], nt=c["nt"], eps_guess=eps, shape=shape, lam=np.full(c["n_nodes"], 10.0),
                precision=c["precision"], ckpt_interval=c["ckpt"])
    if c["kind"] != "density":
        spec.update(M=c["m"], uniforms=_uniforms(c, seed), jump_scheme="first_order" if c["first_order"] else "bisection",
                    update_rule="cross" if c["kind"] == "cross" else "independent")
        if c["random_init"]:
            spec["psi0_batch"] = _random_states(c, seed)
    return spec


def prepare(case, seed):
    from paper_1801_04382_gb300 import Batch, DensityProblem, Problem
    if case["kind"] == "batch":
        specs = [_spec(s, seed + 101 * i) for i, s in enumerate(_subproblems(case, seed))]
        return dict(case=case, batch=Batch(specs), eps=[s["eps_guess"] for s in specs])
    spec = _spec(case, seed)
    p = DensityProblem(**spec) if case["kind"] == "density" else Problem(**spec)
    eps = spec["eps_guess"]
    if case["kind"] == "gradient":
        eps = torch.tensor(eps, dtype=torch.float64, device="cuda", requires_grad=True)
    return dict(case=case, problem=p, eps=eps)


def _hand_on(case, out):
    """Results of an FP32-mixed problem as 32-bit values."""
    if case["precision"] == "fp64":
        return out
    return {k: v.astype(np.complex64 if np.iscomplexobj(v) else np.float32) if isinstance(v, np.ndarray) else v.float()
            for k, v in out.items()}


def run(state):
    case = state["case"]
    if case["kind"] == "batch":
        b = state["batch"]
        for p, e in zip(b.problems, state["eps"]):
            p.set_pulses(e)
        jt = b.update(case["iters"])
        return {"JT": jt.astype(np.float32), "pulses": [p.pulses().astype(np.float32) for p in b.problems]}
    p, eps = state["problem"], state["eps"]
    if case["kind"] == "gradient":
        from paper_1801_04382_gb300 import trajectory_functional
        eps.grad = None
        jt = trajectory_functional(eps, p)
        jt.backward()
        return _hand_on(case, {"JT": jt.detach(), "grad": eps.grad})
    p.set_pulses(eps)
    jt, j = p.update(case["iters"])
    return _hand_on(case, {"JT": jt, "J": j, "pulses": p.pulses(), "deps": p.deps(),
                           "fidelities": np.abs(p.fidelity()[1]) ** 2})


# ------------------------------------------------------------------------------------ the work
def _terms(c):
    """Terms of the Chebyshev series of one interval: the Bessel functions J_k(r dt) of the spectral
    half width r, cut at the roundoff of the state's type."""
    r = 0.5 * c["n_nodes"] * DELTA + 2.0
    if c["kind"] == "density":
        r *= 2.0
    x, tol = r * c["dt"], 1e-16 if c["precision"] == "fp64" else 2.0 ** -24
    th = (np.arange(512) + 0.5) * (math.pi / 512)
    for k in range(1, 250):
        if k > x and abs(np.mean(np.cos(k * th - x * np.sin(th)))) < tol:
            return k
    return 250


def work(case):
    """Bytes: pulses and uniforms in, pulses out, and each co-state written by the backward sweep and
    read by the updating one.  Flops: the generator once per Chebyshev term and sweep, two FMAs per
    (real or imaginary) coupling, four for the diagonal and two for the sum."""
    c = case
    if c["kind"] == "batch":
        parts = [work(s) for s in _subproblems(c, 0)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    n, nl = c["n_nodes"], 3 * (c["n_cav"] + 1)
    s = 16 if c["precision"] == "fp64" else 8
    d, m = nl ** n, c["m"]
    hop = (c["n_cav"] / (c["n_cav"] + 1.0)) ** 2
    couplings = n * (2.0 * c["n_cav"] + 2.0 * (c["n_cav"] + 1)) / nl + 0.5 * n * (n - 1) * hop
    if c["kind"] == "density":
        d, couplings = d * d, 2.0 * couplings + n * n * hop
    per = 2.0 * (2.0 * couplings + 4.0 + 2.0) * (_terms(c) - 1)
    flops = _sweeps(c) * c["nt"] * float(m) * d * per
    if c["kind"] == "cross":
        flops += c["iters"] * c["nt"] * 8.0 * m * m * d * (1 + n)
    pulses = 8.0 * n * c["nt"]
    nbytes = (2 + c["iters"]) * pulses + 8.0 * (1 + c["iters"]) * m
    if c["kind"] != "gradient":
        nbytes += c["iters"] * 2.0 * s * d * m * c["nt"]
    else:
        nbytes += 2.0 * s * d * m * c["nt"]
    return {"bytes": nbytes, "flops": flops}


# ----------------------------------------------------------------- the same in plain 64-bit torch
# Operators as (column, value) lists per row, propagators as Taylor series, jump times by bisection
# of the norm through the Gram matrix of the series' terms.  Trajectories that share their state
# (no jump yet, or the same random start) share a column.
class _Op:
    """Sum of shifted diagonals: (A v)[x] = sum_o val_o[x] v[x + o]."""

    def __init__(self, d):
        self.d, self.parts = d, {}

    def add(self, rows, off, vals):
        v = self.parts.setdefault(off, np.zeros(self.d, dtype=np.complex128))
        v[rows] += vals

    def dagger(self):
        out = _Op(self.d)
        for o, v in self.parts.items():
            x = np.nonzero(v)[0]
            out.add(x + o, -o, v[x].conj())
        return out

    def plus(self, other, w):
        for o, v in other.parts.items():
            x = np.nonzero(v)[0]
            self.add(x, o, w * v[x])
        return self

    def tables(self, offs, dev):
        x = np.arange(self.d)
        cols = torch.tensor(np.stack([np.clip(x + o, 0, self.d - 1) for o in offs]), device=dev)
        vals = torch.tensor(np.stack([self.parts.get(o, np.zeros(self.d, dtype=np.complex128)) for o in offs]), device=dev)
        return cols, vals


def _mul(cols, vals, v):
    """A v for a block of columns v [d, R]; ``vals`` [S, d], or [S, d] per use."""
    return torch.einsum("sd,sdr->dr", vals, v[cols])


class _Model:
    def __init__(self, c, dev):
        n, nc, kap = c["n_nodes"], c["n_cav"], c["kappa"]
        npn, nl = nc + 1, 3 * (nc + 1)
        d = nl ** n
        self.d, self.n, self.dt, self.dev = d, n, c["dt"], dev
        x = np.arange(d)
        stride = [nl ** (n - 1 - i) for i in range(n)]
        dig = [(x // s) % nl for s in stride]
        atom, num = [g // npn for g in dig], [g % npn for g in dig]
        h, self.hc, low = _Op(d), [], []
        for i in range(n):
            s = stride[i]
            h.add(x, 0, -DELTA * (atom[i] == 2) - num[i] / DELTA)
            up = x[(atom[i] == 2) & (num[i] < nc)]                       # (r, k) <- (g, k + 1)
            dn = x[(atom[i] == 0) & (num[i] >= 1)]                       # (g, k) <- (r, k - 1)
            h.add(up, (1 - 2 * npn) * s, np.sqrt(num[i][up] + 1.0))
            h.add(dn, (2 * npn - 1) * s, np.sqrt(1.0 * num[i][dn]))
            hc = _Op(d)
            hc.add(x[atom[i] == 2], -npn * s, 0.5j)                      # (r, k) <- (e, k)
            hc.add(x[atom[i] == 1], npn * s, -0.5j)
            self.hc.append(hc)
            a = _Op(d)
            k = x[num[i] < nc]
            a.add(k, s, np.sqrt(num[i][k] + 1.0))
            low.append(a)

        def prod(a, b, w):                                               # w a^dag b, added to h
            ad = a.dagger()
            for o1, v1 in ad.parts.items():
                for o2, v2 in b.parts.items():
                    r = np.nonzero(v1)[0]
                    h.add(r, o1 + o2, w * v1[r] * v2[r + o1])

        for i in range(n):
            for j in range(i + 1, n):
                prod(low[i], low[j], 1j * kap)
                prod(low[j], low[i], -1j * kap)
        g = math.sqrt(2.0 * kap)
        groups = [[i] for i in range(n)] if c["local"] else [list(range(n))]
        self.lind = [_Op(d) for _ in groups]
        for op, grp in zip(self.lind, groups):
            for i in grp:
                op.plus(low[i], g)
            for i in grp:
                for j in grp:
                    prod(low[i], low[j], -0.5j * g * g)
        offs = sorted(set(o for op in [h] + self.hc for o, v in op.parts.items() if np.any(v)))
        self.cols, self.h0 = h.tables(offs, dev)
        self.hct = [op.tables(offs, dev)[1] for op in self.hc]
        hd = h.dagger()
        offd = sorted(set(o for op in [hd] + self.hc for o, v in op.parts.items() if np.any(v)))
        self.cols_d, self.h0_d = hd.tables(offd, dev)
        self.hct_d = [op.tables(offd, dev)[1] for op in self.hc]
        self.lin = [op.tables(sorted(op.parts), dev) for op in self.lind]
        self.lin_d = [op.dagger().tables(sorted(op.dagger().parts), dev) for op in self.lind]
        self.shift = -0.5 * n * DELTA                                    # centre of the spectrum
        v = np.zeros(d, dtype=np.complex128)
        for i in range(n):
            v[sum(0 if q != i else npn * stride[i] for q in range(n))] = 1.0 / math.sqrt(n)
        self.tgt = torch.tensor(v, device=dev)
        alpha = self.dt * (0.5 * n * DELTA + 12.0 * n)
        self.order = 8
        while alpha ** self.order / math.factorial(self.order) > 1e-19:
            self.order += 1

    def gen(self, eps, adj=False):
        """(columns, values) of -i (H_eff - shift), or of its adjoint's partner +i (H_eff^dag - shift)."""
        base, hct = (self.h0_d, self.hct_d) if adj else (self.h0, self.hct)
        v = base.clone()
        for e, hc in zip(eps, hct):
            v += float(e) * hc
        return (self.cols_d if adj else self.cols), v * (1j if adj else -1j)

    def terms(self, g, v, adj=False):
        """A^k v / k! for k = 0 .. order, A = -i (H - shift) (adj: +i (H^dag - shift)), no time factor."""
        cols, vals = g
        sh = (-1j if adj else 1j) * self.shift
        out = [v]
        for k in range(1, self.order + 1):
            t = (_mul(cols, vals, out[-1]) + sh * out[-1]) * (1.0 / k)
            out.append(t)
        return out

    def sum(self, terms, s, adj=False):
        """exp(A s) v for times s (a number, or one per column), with the shift's phase."""
        s = torch.as_tensor(s, dtype=torch.float64, device=self.dev)
        out = terms[-1] * s
        for t in terms[-2:0:-1]:
            out = (out + t) * s
        return (out + terms[0]) * torch.exp((1j if adj else -1j) * self.shift * s)

    def expm(self, g, v, s, adj=False):
        """exp(A s) v without keeping the series' terms."""
        cols, vals = g
        s = torch.as_tensor(s, dtype=torch.float64, device=self.dev)
        sh = (-1j if adj else 1j) * self.shift
        out, t = v.clone(), v
        for k in range(1, self.order + 1):
            t = (_mul(cols, vals, t) + sh * t) * (s / k)
            out += t
        return out * torch.exp((1j if adj else -1j) * self.shift * s)

    def lower(self, l, v, adj=False):
        return _mul(*(self.lin_d if adj else self.lin)[l], v)


def _crossing(md, terms, r, length):
    """Times at which the columns' norms fall to r: bisection of sum_kl s^(k+l) <t_k|t_l> = r."""
    v = torch.stack(terms)                                               # [order + 1, d, J]
    gram = torch.einsum("adj,bdj->jab", v.conj(), v).real
    n = len(terms)
    coef = torch.zeros(gram.shape[0], 2 * n - 1, dtype=torch.float64, device=md.dev)
    for a in range(n):
        coef[:, a:a + n] += gram[:, a]
    lo, hi = torch.zeros_like(length), length.clone()
    for _ in range(54):
        mid = 0.5 * (lo + hi)
        f = torch.zeros_like(mid)
        for q in range(2 * n - 2, -1, -1):
            f = f * mid + coef[:, q]
        down = f <= r
        hi, lo = torch.where(down, mid, hi), torch.where(down, lo, mid)
    return hi


def _forward(md, c, eps, U, psi, row, chi=None, keep=False):
    """A forward sweep.  psi [d, R] and row [M] (the column of each trajectory); chi = (list of co-states,
    rows, shape, rule) for an updating one.  Returns the final columns, rows, records, pulse, kept states."""
    M, dev, dt = c["m"], md.dev, md.dt
    r = U[:, 0].copy()
    rec = [[] for _ in range(M)]
    eps = eps.copy()
    kept = []
    for j in range(c["nt"]):
        if chi is not None:
            cj, crow, shape, cross = chi[0][j], chi[1], chi[2], chi[3]
            for i in range(md.n):
                a = cj.conj().T @ _mul(md.cols, md.hct[i], psi)          # <chi|h_i|psi> by column pair
                if cross:
                    g = cj.conj().T @ psi
                    wa = torch.tensor(np.bincount(crow, minlength=cj.shape[1]), device=dev, dtype=torch.float64)
                    wb = torch.tensor(np.bincount(row, minlength=psi.shape[1]), device=dev, dtype=torch.float64)
                    s = float(((a * g.conj()).imag * wa[:, None] * wb[None, :]).sum()) / M
                else:
                    s = float(a.imag[torch.tensor(crow, device=dev), torch.tensor(row, device=dev)].sum())
                eps[i, j] += shape[i, j] / (10.0 * M) * s
        if keep:
            kept.append((psi, row.copy()))
        g = md.gen(eps[:, j])
        new = md.expm(g, psi, dt)
        nrm = (new.abs() ** 2).sum(0).cpu().numpy()
        todo = np.nonzero(nrm[row] <= r)[0]
        if len(todo) and c["first_order"]:
            start, s0 = new[:, torch.tensor(row[todo], device=dev)], np.full(len(todo), dt)
        elif len(todo):
            start, s0 = psi[:, torch.tensor(row[todo], device=dev)], np.zeros(len(todo))
        cols, at = [new], psi.shape[1]
        while len(todo):
            left = torch.tensor(dt - s0, device=dev)
            if c["first_order"]:
                phi, s = start, s0
            else:
                terms = md.terms(g, start)
                step = _crossing(md, terms, torch.tensor(r[todo], device=dev), left)
                phi, s = md.sum(terms, step), s0 + step.cpu().numpy()
            ys = [md.lower(l, phi) for l in range(len(md.lin))]
            pl = torch.stack([(y.abs() ** 2).sum(0) for y in ys]).cpu().numpy()
            cum = np.cumsum(pl, axis=0)
            nj = np.array([len(rec[k]) + 1 for k in todo])
            ch = np.argmax(cum >= U[todo, 2 * nj - 1] * cum[-1], axis=0)
            cn = 1.0 / np.sqrt(pl[ch, np.arange(len(todo))])
            start = torch.stack([ys[l][:, i] for i, l in enumerate(ch)], dim=1) * torch.tensor(cn, device=dev)
            for i, k in enumerate(todo):
                rec[k].append((j, float(s[i]), int(ch[i]), float(cn[i])))
            r[todo] = U[todo, 2 * nj]
            s0 = s
            if c["first_order"]:
                end, again = start, np.zeros(len(todo), dtype=bool)
            else:
                end = md.expm(g, start, torch.tensor(dt - s0, device=dev))
                again = (end.abs() ** 2).sum(0).cpu().numpy() <= r[todo]
            done = np.nonzero(~again)[0]
            cols.append(end[:, torch.tensor(done, device=dev)])
            row[todo[done]] = at + np.arange(len(done))
            at += len(done)
            sel = np.nonzero(again)[0]
            todo, s0, start = todo[sel], s0[sel], start[:, torch.tensor(sel, device=dev)]
        psi = torch.cat(cols, dim=1)
        used, row = np.unique(row, return_inverse=True)                  # drop columns nobody holds
        if len(used) < psi.shape[1]:
            psi = psi[:, torch.tensor(used, device=dev)]
    return psi, row, rec, eps, kept


def _backward(md, c, eps, rec, chiT, row):
    """Co-states at t_0 .. t_nt along each column's record (columns share a record)."""
    R = chiT.shape[1]
    of = [None] * R
    for k, q in enumerate(row):
        of[q] = rec[k]
    out = [None] * c["nt"] + [chiT]
    for j in range(c["nt"] - 1, -1, -1):
        g = md.gen(eps[:, j], adj=True)
        v = md.expm(g, out[j + 1], md.dt, adj=True)
        for q in range(R):
            js = [x for x in of[q] if x[0] == j]
            if js:
                w, hi = out[j + 1][:, q:q + 1], md.dt
                for (_, s, l, cn) in reversed(js):
                    w = md.lower(l, md.expm(g, w, hi - s, adj=True), adj=True) * cn
                    hi = s
                v[:, q:q + 1] = md.expm(g, w, hi, adj=True)
        out[j] = v
    return out


def _regroup(rec, row):
    """Columns by record: a trajectory's co-state is shared only with those of the same column and record."""
    seen, out, first = {}, np.zeros(len(row), dtype=int), []
    for k, q in enumerate(row):
        key = (int(q), tuple(rec[k]))
        if key not in seen:
            seen[key] = len(first)
            first.append(k)
        out[k] = seen[key]
    return out, first


def _exact_trajectories(c, seed, dev):
    md = _Model(c, dev)
    eps, shape = _pulse(c, seed)
    U = _uniforms(c, seed)
    M = c["m"]

    def start():
        if c["random_init"]:
            return torch.tensor(_random_states(c, seed).T.copy(), device=dev), np.arange(M)
        return torch.tensor(_psi0(c), device=dev)[:, None], np.zeros(M, dtype=int)

    def overlaps(psi):
        return (md.tgt.conj()[:, None] * psi).sum(0) / torch.sqrt((psi.abs() ** 2).sum(0))

    if c["kind"] == "gradient":
        psi, row, rec, _, kept = _forward(md, c, eps, U[0], *start(), keep=True)
        tau = overlaps(psi)
        nrm = torch.sqrt((psi.abs() ** 2).sum(0))
        crow, first = _regroup(rec, row)
        sel = torch.tensor(row[first], device=dev)
        chiT = (tau * md.tgt[:, None] - (tau.abs() ** 2) * psi / nrm)[:, sel] / nrm[sel]
        mult = np.bincount(crow)
        grad = _exact_gradient(md, c, eps, rec, crow, first, chiT, mult, kept)
        jt = 1.0 - float((tau.abs() ** 2)[torch.tensor(row, device=dev)].sum()) / M
        return {"JT": torch.tensor(jt, dtype=torch.float64), "grad": torch.tensor(grad)}
    psi, row, rec, _, _ = _forward(md, c, eps, U[0], *start())
    jts, js = [], []
    for it in range(c["iters"]):
        tau = overlaps(psi)
        crow, first = _regroup(rec, row)
        sel = torch.tensor(row[first], device=dev)
        cross = c["kind"] == "cross"
        chiT = md.tgt[:, None].expand(-1, len(first)).clone() if cross else tau[sel][None, :] * md.tgt[:, None]
        chi = _backward(md, c, eps, [rec[k] for k in range(M)], chiT, crow)
        psi, row, rec, new, _ = _forward(md, c, eps, U[1 + it], *start(), chi=(chi, crow, shape, cross))
        tau = overlaps(psi)
        jt = 1.0 - float((tau.abs() ** 2)[torch.tensor(row, device=dev)].sum()) / M
        jts.append(jt)
        js.append(jt + float((10.0 * (new - eps) ** 2 * c["dt"] / shape).sum()))
        deps, eps = new - eps, new
    return {"JT": np.array(jts), "J": np.array(js), "pulses": eps, "deps": deps,
            "fidelities": (tau.abs() ** 2)[torch.tensor(row, device=dev)].cpu().numpy()}


def _exact_gradient(md, c, eps, rec, crow, first, chi, mult, kept):
    """dJ_T/deps of the frozen records: reverse differentiation of each interval's Taylor series."""
    grad = np.zeros_like(eps)
    w = torch.tensor(mult, dtype=torch.float64, device=md.dev)

    def piece(j, z, v, s, weight):
        """Adds <v| d exp(A s) |z> to the gradient of interval j; returns exp(A s)^dag v."""
        g, gd = md.gen(eps[:, j]), md.gen(eps[:, j], adj=True)
        N = md.order
        ph = torch.exp(torch.tensor(-1j * md.shift * s, dtype=torch.complex128, device=md.dev))
        ys = [None] * (N + 1)
        ys[N] = z
        for n in range(N, 0, -1):
            ys[n - 1] = z + (_mul(*g, ys[n]) + 1j * md.shift * ys[n]) * (s / n)
        b = v * ph.conj()
        out = b.clone()
        for n in range(1, N + 1):
            for i in range(md.n):
                x = (b.conj() * (-1j) * _mul(md.cols, md.hct[i], ys[n])).sum(0) * (s / n)
                grad[i, j] += float((x.real * weight).sum())
            b = (_mul(*gd, b) - 1j * md.shift * b) * (s / n)
            out += b
        return out

    for j in range(c["nt"] - 1, -1, -1):
        psi, prow = kept[j]
        z = psi[:, torch.tensor(prow[first], device=md.dev)]
        jumps = [[x for x in rec[k] if x[0] == j] for k in first]
        sel = np.nonzero([not x for x in jumps])[0]
        new = chi.clone()
        if len(sel):
            st = torch.tensor(sel, device=md.dev)
            new[:, st] = piece(j, z[:, st], chi[:, st], md.dt, w[st])
        for q in np.nonzero([bool(x) for x in jumps])[0]:
            zs, at, cur = [], 0.0, z[:, q:q + 1]
            g = md.gen(eps[:, j])
            for (_, s, l, cn) in jumps[q]:
                zs.append((cur, s - at))
                cur = md.lower(l, md.expm(g, cur, s - at)) * cn
                at = s
            v = piece(j, cur, chi[:, q:q + 1], md.dt - at, w[q:q + 1])
            for (cur, ln), (_, s, l, cn) in zip(reversed(zs), reversed(jumps[q])):
                v = piece(j, cur, md.lower(l, v, adj=True) * cn, ln, w[q:q + 1])
            new[:, q:q + 1] = v
        chi = new
    return -2.0 / c["m"] * grad


def _exact_density(c, seed, dev):
    md = _Model(c, dev)
    eps, shape = _pulse(c, seed)
    eye = torch.eye(md.d, dtype=torch.complex128, device=dev)
    h0, hc = _mul(md.cols, md.h0, eye), [_mul(md.cols, t, eye) for t in md.hct]
    L = [md.lower(l, eye) for l in range(len(md.lin))]
    order = 2 * md.order

    def step(e, rho, adj):
        h = h0 + sum(float(x) * m for x, m in zip(e, hc))
        out, t = rho.clone(), rho
        for k in range(1, order + 1):
            if adj:
                t = 1j * (h.conj().T @ t - t @ h) + sum(l.conj().T @ t @ l for l in L)
            else:
                t = -1j * (h @ t - t @ h.conj().T) + sum(l @ t @ l.conj().T for l in L)
            t = t * (md.dt / k)
            out += t
        return out

    v = torch.tensor(_psi0(c), device=dev)
    rho0, tgt = torch.outer(v, v.conj()), torch.outer(md.tgt, md.tgt.conj())
    jts, js = [], []
    for _ in range(c["iters"]):
        P = [None] * c["nt"] + [tgt]
        for j in range(c["nt"] - 1, -1, -1):
            P[j] = step(eps[:, j], P[j + 1], True)
        rho, new = rho0, eps.copy()
        for j in range(c["nt"]):
            for i in range(md.n):
                s = float(((P[j].conj() * (hc[i] @ rho - rho @ hc[i])).sum()).imag)
                new[i, j] += shape[i, j] / 10.0 * s
            rho = step(new[:, j], rho, False)
        tau = (tgt.conj() * rho).sum()
        jts.append(1.0 - float(tau.real))
        js.append(jts[-1] + float((10.0 * (new - eps) ** 2 * c["dt"] / shape).sum()))
        deps, eps = new - eps, new
    return {"JT": np.array(jts), "J": np.array(js), "pulses": eps, "deps": deps, "fidelities": np.array([abs(complex(tau)) ** 2])}


def exact(case, seed):
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    if case["kind"] == "batch":
        parts = [_exact_trajectories(s, seed + 101 * i, dev) for i, s in enumerate(_subproblems(case, seed))]
        return {"JT": np.stack([p["JT"] for p in parts], axis=1), "pulses": [p["pulses"] for p in parts]}
    if case["kind"] == "density":
        return _exact_density(case, seed, dev)
    return _exact_trajectories(case, seed, dev)
