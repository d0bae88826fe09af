"""Performance cases: what a user of this library has it do, through its public calls.

Every case is a plain dict.  `prepare` builds what a program holds before the call (a
lowered circuit, a context with its terms, strings, chains' start strings, a network),
`run` is one pass through the public entry points, `work` counts the bytes and
floating-point operations a pass cannot do without, and `exact` gives the same outputs
from plain 64-bit torch, independently of the library.

Kinds of pass:
  amplitude   <x|psi> of a batch of strings, with or without the per-result error bound
  circuit     the circuit from the start: terms re-initialised, all gates, a few amplitudes
  norm        equatorial norm estimates eta_l
  median      the median-of-means norm estimate (a host number)
  chains      Metropolis chains: start from given strings, then single-flip steps
  batch       several circuits of uneven chi: gates and amplitudes in batched calls
  logits      the learned proposal's forward pass (logits and log q)
  gradient    one backward pass of the learned proposal (loss and gradients)
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1808_00128_gb300 import lrstab, workloads

DEV = "cuda:0"


def listed():
    return [
        # every amplitude of a 10-qubit Clifford+T circuit, exact 2-term T: the smallest use
        dict(name="amplitude_n10", kind="amplitude", circuit="clifford_t", n=10, gates=200, slots=6, chi=64,
             batch=1024, bound=False),
        # a batch of 40-bit strings with the error bound of every result
        dict(name="amplitude_n40_bound", kind="amplitude", circuit="clifford_t", n=40, gates=2000, slots=24,
             chi=1 << 16, batch=4096, bound=True),
        # the same batch on the n = 50 QAOA state at chi = 2^20
        dict(name="amplitude_n50", kind="amplitude", circuit="qaoa", n=50, gates=0, slots=0, chi=1 << 20, batch=4096,
             bound=False),
        # a QAOA circuit pushed through from its initial terms, a handful of amplitudes read:
        # the gate updates dominate; chi is no multiple of any tile
        dict(name="circuit_n50", kind="circuit", circuit="qaoa", n=50, gates=0, slots=0, chi=300001, batch=100),
        # one norm estimate of the 40-qubit single-qubit-marginal workload (6 CCZ, 497 terms)
        dict(name="median_n40", kind="median", circuit="hidden_shift", n=40, gates=0, slots=6, chi=497, L=256, K=3),
        # norm estimates of a random Clifford+T state
        dict(name="norm_n40", kind="norm", circuit="clifford_t", n=40, gates=2000, slots=24, chi=1 << 16, L=256),
        # the full-size norm estimate of the n = 50 QAOA state: the largest use
        dict(name="norm_n50", kind="norm", circuit="qaoa", n=50, gates=0, slots=0, chi=1 << 20, L=512),
        # many chains on the 40-qubit state
        dict(name="chains_n40", kind="chains", circuit="clifford_t", n=40, gates=2000, slots=24, chi=1 << 16,
             chains=1024, steps=32),
        # 256 chains of the n = 50 QAOA sampler
        dict(name="chains_n50", kind="chains", circuit="qaoa", n=50, gates=0, slots=0, chi=1 << 20, chains=256,
             steps=64),
        # four QAOA circuits of uneven chi in batched calls
        dict(name="batch_n50", kind="batch", circuit="qaoa", n=50, gates=0, slots=0, chi=1 << 17, batch=1000,
             circuits=4),
        # the 50 -> 512 -> 512 -> 50 proposal network: log q of 16384 strings
        dict(name="logits_n50", kind="logits", n=50, hidden=512, rows=16384),
        # its gradients on a training batch
        dict(name="gradient_n50", kind="gradient", n=50, hidden=512, rows=1024),
    ]


def _between(rng, lo, hi):
    """A whole number between lo and hi, spread evenly over its logarithm."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_circuit(rng, n_max):
    name = rng.choice(["clifford_t", "clifford_t", "qaoa", "hidden_shift"])
    if name == "clifford_t":
        n = rng.randint(10, n_max)
        return dict(circuit=name, n=n, gates=_between(rng, 10 * n, 50 * n), slots=rng.randint(6, 40))
    if name == "qaoa":
        return dict(circuit=name, n=rng.randint(20, n_max), gates=0, slots=0)
    return dict(circuit=name, n=2 * rng.randint(10, n_max // 2), gates=0, slots=2 * rng.randint(1, 8))


def draw(rng):
    kind = rng.choice(["amplitude", "amplitude", "circuit", "norm", "norm", "median", "chains", "chains", "batch",
                       "logits", "gradient"])
    if kind in ("logits", "gradient"):
        return dict(kind=kind, n=rng.randint(10, 62), hidden=64 * _between(rng, 2, 16), rows=_between(rng, 100, 20000))
    if kind == "batch":
        return dict(kind=kind, circuit="qaoa", n=rng.randint(20, 62), gates=0, slots=0, chi=_between(rng, 500, 1 << 17),
                    batch=_between(rng, 16, 2000), circuits=rng.randint(2, 5))
    c = _draw_circuit(rng, 62 if kind == "chains" else 64)
    c["kind"] = kind
    chi = c["chi"] = _between(rng, 64, 1 << 19)
    if kind == "amplitude":
        c.update(batch=_between(rng, 1, min(10000, (1 << 32) // chi)), bound=rng.random() < 0.5)
    elif kind == "circuit":
        c["chi"] = min(chi, 1 << 17)
        c["batch"] = _between(rng, 1, 300)
    elif kind == "norm":
        c["L"] = _between(rng, 16, max(17, min(2000, (1 << 25) // chi)))
    elif kind == "median":
        c["chi"] = min(chi, 1 << 14)
        c.update(L=_between(rng, 16, 512), K=rng.choice([1, 3, 5]))
    else:
        if c["circuit"] == "hidden_shift":   # its chains see P = 0 all around: a walk on rounding noise
            c.update(circuit="qaoa", gates=0, slots=0, n=max(20, c["n"]))
        c.update(chains=_between(rng, 8, max(9, min(1500, (1 << 27) // chi))), steps=rng.randint(5, 70))
    return c


# ---- inputs ------------------------------------------------------------------------------
def _ops(case, seed):
    """The seeded circuit of a case and the string it is about (the hidden shift), if any."""
    n = case["n"]
    if case["circuit"] == "clifford_t":
        return workloads.random_clifford_t(n, case["gates"], case["slots"], 1000 + seed), None
    if case["circuit"] == "qaoa":
        return workloads.qaoa_e3lin2_circuit(n, 4, 0.3, 0.2, 1000 + seed)[0], None
    return workloads.hidden_shift_circuit(n, case["slots"], 1000 + seed)


def _mode(case, slots):
    """Exact enumeration where chi is the exact term count (two choices a slot), else sparsified."""
    return "exact" if case["circuit"] == "clifford_t" and case["chi"] == 1 << slots else "sparsify"


def _ccz(case):
    return "sum8" if case["circuit"] == "hidden_shift" else "proj"


def _strings(n, count, seed, shift=None):
    """Uniform n-bit strings as int64 words; half of a hidden-shift batch is the shift and its neighbourhood."""
    x = workloads.random_bitstrings(n, count, 77 + seed)
    if shift is not None:
        rng = np.random.default_rng(7 + seed)
        near = np.uint64(shift) ^ (np.uint64(1) << rng.integers(0, n, count).astype(np.uint64))
        near[0] = np.uint64(shift)
        x[::2] = near[: len(x[::2])]
    return x.view(np.int64)


def _terms(case, seed):
    ops, shift = _ops(case, seed)
    low = lrstab.lower_circuit(case["n"], ops, _ccz(case))
    sim = lrstab.Simulator(case["n"], 0)
    sim.init_terms(low, case["chi"], _mode(case, len(low.slots)), seed=500 + seed)
    return sim, low, shift


def _params(case, seed):
    n, H = case["n"], case["hidden"]
    rng = np.random.default_rng(900 + seed)
    r1, r2 = 1 / math.sqrt(n), 1 / math.sqrt(H)
    shapes = dict(W1=((H, n), r1), b1=((H,), r1), W2=((H, H), r2), b2=((H,), r2), W3=((n, H), r2), b3=((n,), r2))
    return {k: rng.uniform(-r, r, s).astype(np.float32) for k, (s, r) in shapes.items()}


def _uneven(case):
    """chi of each circuit of a batch: chi, then falling by about 1.6."""
    return [max(64, int(case["chi"] / 1.6 ** i)) for i in range(case["circuits"])]


def prepare(case, seed):
    kind, n = case["kind"], case["n"]
    if kind in ("logits", "gradient"):
        net = lrstab.MLP(n, case["hidden"], 0)
        net.set_params(_params(case, seed))
        return dict(kind=kind, net=net, x=torch.from_numpy(_strings(n, case["rows"], seed)).to(DEV))
    if kind == "batch":
        parts = [_terms(dict(case, chi=chi), seed + 31 * i) for i, chi in enumerate(_uneven(case))]
        return dict(kind=kind, sims=[p[0] for p in parts], gates=[p[1].gates for p in parts],
                    seeds=[500 + seed + 31 * i for i in range(len(parts))],
                    xs=[torch.from_numpy(_strings(n, case["batch"], seed + i)).to(DEV) for i in range(len(parts))])
    sim, low, shift = _terms(case, seed)
    st = dict(kind=kind, sim=sim, gates=low.gates, seed=500 + seed, case=case)
    if kind != "circuit":
        sim.apply_clifford(low.gates)
    if kind in ("amplitude", "circuit"):
        st["x"] = torch.from_numpy(_strings(n, case["batch"], seed, shift)).to(DEV)
    elif kind == "chains":
        st["x"] = sim.sample_terms(case["chains"], seed=600 + seed)
    return st


# ---- one pass ------------------------------------------------------------------------------
def run(st):
    kind = st["kind"]
    if kind == "amplitude":
        x = st["x"]
        if not st["case"]["bound"]:
            return st["sim"].amplitude(x)
        err = torch.empty(x.numel(), dtype=torch.float32, device=x.device)
        return st["sim"].amplitude(x, err=err), err
    if kind == "circuit":
        st["sim"].reinit_terms(st["seed"])
        st["sim"].apply_clifford(st["gates"])
        return st["sim"].amplitude(st["x"])
    if kind == "norm":
        return st["sim"].norm_estimate(st["case"]["L"], st["seed"])
    if kind == "median":
        return st["sim"].norm_median_of_means(st["case"]["L"], st["case"]["K"], st["seed"])
    if kind == "chains":
        x = torch.empty_like(st["x"])
        p = torch.empty(x.numel(), dtype=torch.float64, device=x.device)
        st["sim"].chains_init(st["x"])
        st["sim"].metropolis(st["case"]["steps"], st["seed"], x_out=x, p_out=p)
        return x, p
    if kind == "batch":
        for sim, seed in zip(st["sims"], st["seeds"]):
            sim.reinit_terms(seed)
        lrstab.apply_clifford_batch(st["sims"], st["gates"])
        return lrstab.amplitude_batch(st["sims"], st["xs"])
    if kind == "logits":
        return st["net"].forward(st["x"])
    loss = st["net"].backward(st["x"])
    return loss, st["net"].get_params()[1]


def work(case):
    """Bytes read and written once (a term's tableau is 3n rows, five scalars and its choices) and
    floating-point operations (one complex addition per (string or equatorial state, term); the
    network's multiply-adds).  The bit operations of the tableaux are in neither."""
    kind, n = case["kind"], case["n"]
    if kind in ("logits", "gradient"):
        H, r = case["hidden"], case["rows"]
        mults = 2 * n * H + H * H
        if kind == "logits":
            return dict(bytes=4 * mults + r * (8 + 4 * n + 4), flops=2 * mults * r)
        return dict(bytes=8 * mults + 8 * r, flops=6 * mults * r)
    term = 24 * n + 44
    if kind == "batch":
        chis, B = _uneven(case), case["batch"]
        return dict(bytes=sum(chis) * term + 24 * B * len(chis), flops=2 * B * sum(chis))
    chi = case["chi"]
    if kind in ("amplitude", "circuit"):
        return dict(bytes=chi * term + case["batch"] * (28 if case.get("bound") else 24), flops=2 * case["batch"] * chi)
    if kind == "chains":
        return dict(bytes=chi * term + 24 * case["chains"], flops=2 * case["chains"] * (case["steps"] + 1) * chi)
    L = case["L"] * case.get("K", 1)
    return dict(bytes=chi * term + 8 * L, flops=2 * L * chi)


# ---- the same outputs in 64 bits, by plain torch ---------------------------------------------
_GOLDEN = 0x9E3779B97F4A7C15


def _i64(x):
    """A 64-bit pattern as a signed word."""
    x &= (1 << 64) - 1
    return x - (1 << 64) if x >> 63 else x


def _shr(x, k):
    return (x >> k) & ((1 << (64 - k)) - 1)


def _mix(z):
    """The SplitMix64 finaliser on int64 tensors."""
    z = (z ^ _shr(z, 30)) * _i64(0xBF58476D1CE4E5B9)
    z = (z ^ _shr(z, 27)) * _i64(0x94D049BB133111EB)
    return z ^ _shr(z, 31)


def _stream(seed, stream):
    return _mix(_mix(stream + _i64(_GOLDEN)) ^ _i64(seed))


def _word(key, i):
    return _mix(key + _i64((i + 1) * _GOLDEN))


def _par(x):
    """Parity of 64-bit words, as 0/1 words."""
    for k in (32, 16, 8, 4, 2, 1):
        x = x ^ (x >> k)
    return x & 1


def _slot(op, ccz):
    """Choices of a non-Clifford gate: [(coefficient, [Clifford gates])]."""
    if op[0] == "CCZ":
        a, b, c = op[1:]
        ab, ac, bc = ("CZ", a, b), ("CZ", a, c), ("CZ", b, c)
        za, zb, zc = ("Z", a), ("Z", b), ("Z", c)
        if ccz == "proj":
            return [(1, []), (-2, [("P1", a), ("P1", b), ("P1", c)])]
        w = 1 / 6
        return [(w, []), (w, [ab]), (w, [ac]), (w, [bc]), (w, [ab, ac, za]), (w, [ab, bc, zb]), (w, [ac, bc, zc]),
                (-w, [ab, ac, bc, za, zb, zc])]
    theta = math.pi / 4 if op[0] == "T" else op[2]
    g = complex(math.cos(math.pi / 8), math.sin(math.pi / 8)) if op[0] == "T" else 1.0
    c, s = math.cos(abs(theta) / 2), math.sin(abs(theta) / 2)
    return [(g * (c - s), []), (g * complex(s, -s if theta >= 0 else s), [("S" if theta >= 0 else "SDG", op[1])])]


class _Terms:
    """All terms of a decomposed circuit in CH form, one tensor entry per term: U_C |s> after
    Hadamards on v, phase omega = e^{i pi k/4} 2^{-h/2}, coefficient b (Sec. 4.1 of the paper)."""

    def __init__(self, case, chi, seed, circuit_seed, dev):
        n = self.n = case["n"]
        ops, _ = _ops(case, circuit_seed)
        slots = [_slot(op, _ccz(case)) for op in ops if op[0] in workloads.NON_CLIFFORD]
        z = lambda: torch.zeros(chi, dtype=torch.int64, device=dev)  # noqa: E731
        eye = torch.ones(chi, dtype=torch.int64, device=dev) << torch.arange(n, device=dev)[:, None]
        self.F, self.G, self.M = eye.clone(), eye.clone(), torch.zeros_like(eye)
        self.g = torch.zeros((n, chi), dtype=torch.int8, device=dev)
        self.v, self.s, self.k, self.h = z(), z(), z(), z()
        self.dead = torch.zeros(chi, dtype=torch.bool, device=dev)
        self.mask = _i64((1 << n) - 1)
        alpha = torch.arange(chi, device=dev)
        self.b = torch.ones(chi, dtype=torch.complex128, device=dev)
        exact = _mode(dict(case, chi=chi), len(slots)) == "exact"
        choice, key = [], _stream(seed, alpha)
        for p, sl in enumerate(slots):
            c = torch.tensor([x for x, _ in sl], dtype=torch.complex128, device=dev)
            if exact:
                j = (alpha >> p) & 1
                self.b = self.b * c[j]
            else:
                cdf = torch.cumsum(c.abs() / c.abs().sum(), 0)
                u = _shr(_word(key, p), 11).double() * 2.0 ** -53
                j = (u[:, None] >= cdf).sum(1).clamp(max=len(sl) - 1)
                self.b = self.b * (c / c.abs())[j] * c.abs().sum()
            choice.append(j)
        if not exact:
            self.b = self.b / chi
        p = 0
        for op in ops:
            if op[0] not in workloads.NON_CLIFFORD:
                self.gate(op, None)
                continue
            for j, (_, gates) in enumerate(slots[p]):
                for gate in gates:
                    self.gate(gate, choice[p] == j)
            p += 1
        self.g = self.g & 3

    def gate(self, op, on):
        name, q = op[0], op[1]
        keep = -1 if on is None else -on.long()
        one = 1 if on is None else on.to(torch.int8)
        F, G, M, g = self.F, self.G, self.M, self.g
        if name in ("S", "SDG"):
            M[q] ^= G[q] & keep
            g[q] += (3 if name == "S" else 1) * one
        elif name == "Z":
            g[q] += 2 * one
        elif name == "CZ":
            r = op[2]
            M[q], M[r] = M[q] ^ (G[r] & keep), M[r] ^ (G[q] & keep)
        elif name == "CX":   # Clifford gates of the circuit only: on every term
            r = op[2]
            g[q] += g[r] + 2 * _par(M[q] & F[r]).to(torch.int8)
            G[r] ^= G[q]
            F[q] ^= F[r]
            M[q] ^= M[r]
        elif name == "H":
            nv = ~self.v & self.mask
            t = self.s ^ (G[q] & self.v)
            u = self.s ^ (F[q] & nv) ^ (M[q] & self.v)
            alpha = _par(G[q] & nv & self.s)
            beta = _par((M[q] & nv & self.s) ^ (F[q] & self.v & (M[q] ^ self.s)))
            self.superpose(t, u, (g[q].long() + 2 * (alpha + beta)) & 3, ~self.dead, 4 * alpha, 0)
        else:   # P1: (I - Z_q)/2
            nv = ~self.v & self.mask
            t = self.s ^ (G[q] & self.v)
            sg = 1 ^ _par(G[q] & nv & self.s)
            on = ~self.dead & (True if on is None else on)
            self.dead |= on & (t == self.s) & (sg == 1)
            self.superpose(self.s, t, 2 * sg, on & (t != self.s), 0, 1)

    def superpose(self, t, u, delta, on, dk, dh):
        """U_H(|t> + i^delta |u>) back to CH form on the terms `on` (Prop. of Sec. 4.1)."""
        self.k = self.k + torch.where(on, dk, 0)
        same = on & (t == u)     # 2^{-1/2}(1 + i^delta) with delta odd
        self.k = self.k + torch.where(same, torch.where(delta == 1, 1, 7), 0)
        self.s = torch.where(same, t, self.s)
        on = on & (t != u)
        d = torch.where(on, t ^ u, 1)
        v0, v1 = d & ~self.v, d & self.v
        first = v0 != 0
        pick = torch.where(first, v0, v1)
        q = pick & -pick                      # one-bit mask of the qubit that carries the superposition
        m = torch.where(on, pick & ~q, 0)
        m1 = torch.where(on & first, v1, 0)
        tq, vq = (t & q) != 0, (self.v & q) != 0
        y = torch.where(tq, u ^ q, t)
        flip = (y & q) != 0
        self.k = self.k + torch.where(on & flip, 2 * delta, 0)
        dd = torch.where(flip, (4 - delta) & 3, delta)
        # H^{vq}(|0> + i^dd |1>) = sqrt2 e^{i pi dk/4} S^a H^b |c>
        a = dd & 1
        b = torch.where(vq, a, 1)
        c = torch.where(vq, torch.tensor([0, 1, 1, 0], device=d.device)[dd], dd >> 1)
        self.k = self.k + torch.where(on & vq, torch.tensor([0, 1, 0, 7], device=d.device)[dd], 0)
        a = torch.where(on, a, 0)
        F, G, M = self.F, self.G, self.M
        for p in range(self.n):
            Fp, Gp, Mp = F[p], G[p], M[p]
            fq, gq, mq = -((Fp & q) != 0).long(), -((Gp & q) != 0).long(), -((Mp & q) != 0).long()
            cz = _par(Fp & m1)
            Gn = torch.where(first, Gp ^ (q * _par(Gp & m)), Gp ^ (m & gq))
            Fn = torch.where(first, Fp ^ (m & fq), Fp ^ (q * _par(Fp & m)))
            Mn = torch.where(first, Mp ^ (q * (_par(Mp & m) ^ cz)) ^ (m1 & fq), Mp ^ (m & mq))
            fa = ((Fn & q) != 0).long() * a
            F[p], G[p], M[p] = Fn, Gn, Mn ^ (q * fa)
            self.g[p] += (2 * (cz & -fq) - fa).to(torch.int8)
        self.v = torch.where(on, (self.v & ~q) | (q * b), self.v)
        self.s = torch.where(on, (y & ~q) | (q * c), self.s)
        self.h = self.h + torch.where(on, dh, 0)

    def bits(self, rows, lo, hi):
        """[terms][row][column] of a matrix of words, as 0/1 floats."""
        w = rows[:, lo:hi].t()
        return ((w[:, :, None] >> torch.arange(self.n, device=w.device)) & 1).float()

    def prefactor(self, lo, hi):
        """b omega 2^{-|v|/2} of each term."""
        vw = ((self.v[lo:hi, None] >> torch.arange(self.n, device=self.v.device)) & 1).sum(1)
        size = torch.where(self.dead[lo:hi], 0.0, 2.0 ** (-0.5 * (self.h[lo:hi] + vw).double()))
        return self.b[lo:hi] * size * torch.exp(0.25j * math.pi * (self.k[lo:hi] & 7).double())


def _phases(z):
    return torch.tensor([1, 1j, -1, -1j], dtype=torch.complex128, device=z.device)[z & 3]


def _amplitudes(T, x):
    """Eqs. (amplitude), (amplitude1): <x|phi> is zero unless F^T x = s off v, and else a Z4
    form of x: diagonal gamma_p + 2 F_p.M_p + 2 F_p.(s & v), off the diagonal (M F^T)_pq."""
    n, dev = T.n, T.v.device
    X = ((x[:, None] >> torch.arange(n, device=dev)) & 1).float()
    pq = torch.triu_indices(n, n, 1, device=dev)
    feat = torch.cat([X, X[:, pq[0]] * X[:, pq[1]]], 1)
    out = torch.zeros(len(x), dtype=torch.complex128, device=dev)
    step = max(16, min(1 << 14, (1 << 28) // (len(x) + n * n)))
    for lo in range(0, len(T.v), step):
        hi = min(len(T.v), lo + step)
        F, M = T.bits(T.F, lo, hi), T.bits(T.M, lo, hi)
        J = torch.bmm(M, F.transpose(1, 2))
        vs = T.bits((T.v & T.s)[None], lo, hi)[:, 0]
        diag = T.g[:, lo:hi].t().float() + 2 * (F * M).sum(2) + 2 * torch.bmm(F, vs[:, :, None])[:, :, 0]
        form = torch.cat([diag, 2 * J[:, pq[0], pq[1]]], 1)
        z = (feat @ form.t()).round().long()
        free = T.bits(T.v[None], lo, hi)[:, 0]
        want = T.bits(T.s[None], lo, hi)[:, 0]
        live = torch.ones(z.shape, dtype=torch.bool, device=dev)
        for k in range(n):
            on = (free[:, k] == 0).nonzero()[:, 0]
            if len(on):
                live[:, on] &= ((X @ F[on, :, k].t()).round().long() & 1) == want[on, k].long()
        out += (torch.where(live, _phases(z), 0) * T.prefactor(lo, hi)).sum(1)
    return torch.view_as_real(out)


def _forms(n, L, seed, dev):
    """The equatorial states: symmetric A_l with Z4 diagonals, from their counter streams."""
    key = _stream(seed, torch.arange(L, device=dev))
    pairs = n * (n - 1) // 2
    words = torch.stack([_word(key, i) for i in range(2 + (pairs + 63) // 64)], 1)
    b = (words[:, :, None] >> torch.arange(64, device=dev)) & 1
    pq = torch.triu_indices(n, n, 1, device=dev)
    A = torch.zeros((L, n, n), device=dev)
    A[:, pq[0], pq[1]] = b[:, 2:].reshape(L, -1)[:, :pairs].float()
    A = A + A.transpose(1, 2)
    A.diagonal(dim1=1, dim2=2).copy_((b[:, 0, :n] + 2 * b[:, 1, :n]).float())
    return A


def _sums(S, active, lin):
    """sum over x in Z2^active of (-1)^(x^T S x / 2 + lin . x) of each form (S alternating), by
    eliminating pairs of joined variables.  Returns the sum as (sign or 0, power of two)."""
    P, m = active.shape
    dev = S.device
    sign = torch.zeros(P, dtype=torch.uint8, device=dev)
    e = torch.zeros(P, dtype=torch.int64, device=dev)
    idx = torch.arange(P, device=dev)
    for a in range(m):
        row = S[:, a] * active
        has = (row.amax(1) * active[:, a]).bool()
        b = row.argmax(1)
        r1, r2 = row * has[:, None], S[idx, b] * active * has[:, None]
        r1[idx, b] = 0
        r2[:, a] = 0
        la, lb = lin[:, a] * has, lin[idx, b] * has
        sign ^= la & lb
        lin ^= (r1 & r2) ^ (r1 * lb[:, None]) ^ (r2 * la[:, None])
        S ^= (r1[:, :, None] & r2[:, None, :]) ^ (r2[:, :, None] & r1[:, None, :])
        active[:, a] &= ~has
        active[idx, b] &= ~has
        e += has
    e += active.sum(1)
    return torch.where((lin & active).amax(1) > 0, 0.0, 1.0 - 2.0 * sign.double()), e


def _etas(T, L, seed):
    """eta_l = 2^n |<phi_{A_l}|psi>|^2 by Lemma (Inner Product) on every (l, term)."""
    n, dev = T.n, T.v.device
    A = _forms(n, L, seed, dev)
    total = torch.zeros(L, dtype=torch.complex128, device=dev)
    step = max(1, (1 << 29) // (L * n * n * 4))
    for lo in range(0, len(T.v), step):
        hi = min(len(T.v), lo + step)
        F, G, M = (T.bits(w, lo, hi) for w in (T.F, T.G, T.M))
        v, s = T.bits(T.v[None], lo, hi)[:, 0], T.bits(T.s[None], lo, hi)[:, 0]
        J = torch.bmm(M, F.transpose(1, 2)) % 2
        J.diagonal(dim1=1, dim2=2).copy_(T.g[:, lo:hi].t().float())
        D = (A[None] + J[:, None]).reshape(-1, n, n)            # [term * l]
        Gt = G[:, None].expand(-1, L, -1, -1).reshape(-1, n, n)
        K = torch.bmm(Gt.transpose(1, 2), torch.bmm(D, Gt)).round().long() & 3
        sv = s[:, None].expand(-1, L, -1).reshape(-1, n).long()
        vv = v[:, None].expand(-1, L, -1).reshape(-1, n).bool()
        sK = (sv[:, :, None] * K).sum(1)
        sKs = (sK * sv).sum(1)
        diag = (K.diagonal(dim1=1, dim2=2) + 2 * (sv + sK)) & 3
        # lift of the Z4 form to Z2 with one more variable X joined to the odd diagonals
        odd = ((diag & 1).bool() & vv).to(torch.uint8)
        S = torch.zeros((len(odd), n + 1, n + 1), dtype=torch.uint8, device=dev)
        S[:, :n, :n] = (K & 1).to(torch.uint8) ^ (odd[:, :, None] & odd[:, None, :])
        S[:, :n, n] = odd
        S[:, n, :n] = odd
        S.diagonal(dim1=1, dim2=2).zero_()
        act = torch.cat([vv, torch.ones_like(vv[:, :1])], 1).to(torch.uint8)
        lin = torch.cat([(diag >> 1) & 1, torch.zeros_like(diag[:, :1])], 1).to(torch.uint8)
        S &= act[:, :, None] & act[:, None, :]
        lin &= act
        re, e = _sums(S.clone(), act.clone(), lin.clone())
        lin[:, n] = 1
        im, _ = _sums(S, act, lin)
        z = torch.complex(re, im).conj() * 2.0 ** (e - 1).double()
        sign = 1.0 - 2.0 * ((sv * vv).sum(1) & 1).double()
        val = z * sign * _phases(-sKs)
        total += (val.reshape(-1, L) * T.prefactor(lo, hi)[:, None]).sum(0)
    return total.abs() ** 2


def _network(case, seed, dev):
    """Masked weights of the proposal network and its input bits, in 64 bits."""
    n, H = case["n"], case["hidden"]
    p = {k: torch.from_numpy(v).double().to(dev) for k, v in _params(case, seed).items()}
    x = torch.from_numpy(_strings(n, case["rows"], seed)).to(dev)
    X = ((x[:, None] >> torch.arange(n, device=dev)) & 1).double()
    d, m = torch.arange(1, n + 1, device=dev), torch.arange(H, device=dev) % (n - 1) + 1
    keep = dict(W1=m[:, None] >= d, W2=m[:, None] >= m, W3=d[:, None] > m)
    return p, {k: v.double() for k, v in keep.items()}, X


def exact(case, seed):
    kind = case["kind"]
    dev = DEV if torch.cuda.is_available() else "cpu"
    if kind in ("logits", "gradient"):
        p, keep, X = _network(case, seed, dev)
        for t in p.values():
            t.requires_grad_(kind == "gradient")
        h1 = torch.relu(X @ (p["W1"] * keep["W1"]).t() + p["b1"])
        h2 = torch.relu(h1 @ (p["W2"] * keep["W2"]).t() + p["b2"])
        z = h2 @ (p["W3"] * keep["W3"]).t() + p["b3"]
        nll = (torch.nn.functional.softplus(z) - X * z).sum(1)
        if kind == "logits":
            return z, -nll
        nll.mean().backward()
        return nll.mean().detach().reshape(1), {k: t.grad for k, t in p.items()}
    if kind == "chains":
        return None   # every step needs every chain's amplitude of another string: minutes
    if kind == "batch":
        return [_amplitudes(_Terms(case, chi, 500 + seed + 31 * i, seed + 31 * i, dev),
                            torch.from_numpy(_strings(case["n"], case["batch"], seed + i)).to(dev))
                for i, chi in enumerate(_uneven(case))]
    if kind in ("norm", "median"):
        L = case["L"] * case.get("K", 1)
        if L * case["chi"] * case["n"] ** 3 > 2 ** 41:
            return None   # beyond some ten seconds
        eta = _etas(_Terms(case, case["chi"], 500 + seed, seed, dev), L, 500 + seed)
        return eta if kind == "norm" else float(eta.reshape(-1, case["L"]).mean(1).median())
    x = torch.from_numpy(_strings(case["n"], case["batch"], seed, _ops(case, seed)[1])).to(dev)
    amp = _amplitudes(_Terms(case, case["chi"], 500 + seed, seed, dev), x)
    return (amp, None) if case.get("bound") else amp   # the error bound has no other value
