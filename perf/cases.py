"""The work that a user of this package has it do, as cases to be timed and compared.

A case is one call (or one short sequence) of the public entry points in
paper_2111_00050_gb300: time evolution of a prepared state, a coupling sweep, the
observables of a state, a run observed at intervals, H psi, and gradients by the
adjoint.  Every size comes from the toy models of the workloads, the tests and the
benchmark, or from the same ranges.

exact() restates the mathematics in 64-bit torch, from the occupation vectors on: no
part of the package is used there.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2111_00050_gb300 as qb
from paper_2111_00050_gb300 import api

DEV = "cuda"


# ------------------------------------------------------------------ the cases


def listed():
    return [
        # the smallest call: one number state of a 42-ket sector, a few of its 10^4 steps
        dict(name="number_m5", op="evolve", M=5, coupling="contact", strength=-0.1, exact=False, state="number",
             n_tot=6, p0=True, dt=1e-3, steps=100),
        # a breaktime run: a coherent state observed at intervals, one sample per 20 steps
        dict(name="series_m5", op="series", M=5, coupling="long_range", strength=0.1, exact=False, state="coherent",
             n_tot=5, p0=False, dt=5e-3, steps=200, every=20),
        # the ordinary evolution between two samples of a squeezing run (0.25M kets)
        dict(name="squeezing_m7", op="evolve", M=7, coupling="long_range", strength=0.1, exact=False, state="coherent",
             n_tot=4, p0=False, dt=2e-3, steps=100),
        # the largest state: every sector of a Poisson-weighted coherent state (62.9M kets)
        dict(name="coherent_m7", op="evolve", M=7, coupling="contact", strength=-0.05 / 16, exact=False,
             state="coherent", n_tot=16, p0=False, dt=1e-3, steps=1),
        # gravity-like long range from a field number state, one particle number (23.5M kets)
        dict(name="long_range_m9", op="evolve", M=9, coupling="long_range", strength=0.1 / 27, exact=False,
             state="field", n_tot=27, p0=False, dt=1e-3, steps=1),
        # eight couplings of one large sector evolved side by side (8 x 2.7M kets)
        dict(name="sweep_m11", op="sweep", M=11, coupling="contact", strength=-0.02, exact=False, state="field",
             n_tot=20, p0=True, dt=5e-4, steps=1, batch=8),
        # momentum conserved exactly: many more, smaller sectors (2.6M kets)
        dict(name="exact_m7", op="evolve", M=7, coupling="contact", strength=-0.05 / 8, exact=True, state="coherent",
             n_tot=8, p0=False, dt=1e-3, steps=4),
        # an even number of modes with a complex Hermitian coupling (0.23M kets)
        dict(name="hermitian_m6", op="evolve", M=6, coupling="hermitian", strength=0.02, exact=False, state="coherent",
             n_tot=6, p0=False, dt=1e-3, steps=10),
        # every observable of one state between two stretches of evolution (15.4M kets)
        dict(name="observables_m7", op="observables", M=7, coupling="contact", strength=-0.05 / 12, exact=False,
             state="coherent", n_tot=12, p0=False),
        # gradient of a breaktime loss from stored checkpoints (2.3M kets)
        dict(name="adjoint_m5", op="adjoint", M=5, coupling="contact", strength=-0.1, exact=False, state="coherent",
             n_tot=20, p0=False, dt=2e-3, steps=20, ckpt=10, loss="Q"),
        # forward and backward through the autograd function, the coupling tensor among its inputs
        dict(name="autograd_m5", op="autograd", M=5, coupling="contact", strength=-0.1, exact=False, state="coherent",
             n_tot=12, p0=False, dt=5e-3, steps=10, ckpt=0, loss="PO"),
        # one double-precision H psi of the large sector, as for an energy variance (2.7M kets)
        dict(name="hpsi_m11", op="hpsi", M=11, coupling="contact", strength=-0.02, exact=False, state="field",
             n_tot=20, p0=True),
    ]


def draw(rng):
    """One more case of the same ranges: the work of a pass stays below the largest listed one's."""
    op = rng.choice(["evolve"] * 5 + ["sweep", "observables", "observables", "series", "adjoint", "autograd", "hpsi"])
    M = rng.choice([5, 5, 7, 7, 9, 11, 4, 6, 8])
    exact = op == "evolve" and rng.random() < 0.2
    coupling = rng.choice(["contact", "contact", "long_range", "long_range", "hermitian"])
    if op in ("sweep", "autograd") and coupling == "hermitian":
        coupling = "contact"
    if op in ("adjoint", "autograd"):
        M = rng.choice([5, 5, 7, 4])
    most = {"evolve": 8e6, "sweep": 1e6, "observables": 2e7, "series": 3e5, "adjoint": 2e6, "autograd": 4e5,
            "hpsi": 4e6}[op]
    state = "coherent" if op in ("adjoint", "autograd", "series") else rng.choice(["coherent", "coherent", "field"])
    p0 = state == "field" and rng.random() < 0.5
    if op == "evolve" and state == "field" and rng.random() < 0.3:
        state = "number"
    # the mean particle number: its kets spread over the logarithm of the range
    want = math.exp(rng.uniform(math.log(60.0), math.log(most)))
    top = 31 if M >= 9 else 90
    n_tot = 1
    for n in range(1, top + 1):
        if _kets(M, state, n, p0) > want or _nmax(state, n) > top:
            break
        n_tot = n
    strength = {"contact": -0.05, "long_range": 0.1, "hermitian": 0.1}[coupling] * rng.uniform(0.5, 2.0) / n_tot
    case = dict(op=op, M=M, coupling=coupling, strength=strength, exact=exact, state=state, n_tot=n_tot, p0=p0)
    if op in ("observables", "hpsi"):
        return case
    if op == "sweep":
        case["batch"] = rng.choice([2, 4, 8])
    per_step = 4.0 * _terms(case) * case.get("batch", 1)
    steps = int(min(math.exp(rng.uniform(0.0, math.log(200.0))), 2e9 / per_step))
    case.update(dt=rng.choice([5e-4, 1e-3, 2e-3]), steps=max(1, steps))
    if op == "series":
        every = rng.choice([5, 10, 20])
        case.update(every=every, steps=every * rng.randint(2, 8))
    if op in ("adjoint", "autograd"):  # runs long enough for the loss to leave its initial value
        case.update(strength=-0.1 * rng.uniform(0.5, 1.5), dt=rng.choice([2e-3, 5e-3]), steps=rng.randint(8, 16),
                    ckpt=rng.choice([0, 1, 5]) if op == "adjoint" else 0, loss=rng.choice(["Q", "PO"]))
    return case


def _nmax(state, n_tot):
    return int(math.floor(n_tot + 6.0 * math.sqrt(n_tot))) if state == "coherent" else n_tot


def _kets(M, state, n_tot, p0):
    """Kets of the space (one momentum of M: about 1 / M of a layer)."""
    if state == "coherent":
        return math.comb(_nmax(state, n_tot) + M, M)
    layer = math.comb(n_tot + M - 1, M - 1)
    return layer / M if p0 else layer


def _terms(case):
    """Matrix elements of one H psi, diagonal included: each active pair of a ket has a partner for
    every pair of its momentum class, and (ket, pair) matches a ket with two particles fewer."""
    M, exact = case["M"], case["exact"]
    lab = _labels(M)
    pairs = [(r, s) for r in range(M) for s in range(r, M)]
    tot = [lab[r] + lab[s] for r, s in pairs]
    partners = sum((a - b) == 0 if exact else (a - b) % M == 0 for a in tot for b in tot) - len(pairs)
    if case["state"] == "coherent":
        below = math.comb(max(0, _nmax("coherent", case["n_tot"]) - 2) + M, M)
    else:
        below = math.comb(max(0, case["n_tot"] - 2) + M - 1, M - 1) / (M if case["p0"] else 1)
    return _kets(M, case["state"], case["n_tot"], case["p0"]) + partners * below


def work(case):
    """Bytes: the state read and written once (H psi, observables: as their inputs and outputs
    are).  Flops: two multiply-adds a matrix element (four for a complex coupling), for every
    H psi that the scheme takes: four a Runge-Kutta step; the adjoint's backward step four
    costate stages beside the forward ones; the moments one element a ket and operator."""
    op, M = case["op"], case["M"]
    kets, terms = _kets(M, case["state"], case["n_tot"], case["p0"]), _terms(case)
    flop = 8.0 if case["coupling"] == "hermitian" else 4.0
    moments = flop * terms / 2 + 8.0 * kets * (M + M * M)
    if op == "evolve":
        return {"bytes": 32.0 * kets, "flops": 4 * case["steps"] * flop * terms}
    if op == "sweep":
        return {"bytes": 32.0 * kets * case["batch"], "flops": 4 * case["steps"] * flop * terms * case["batch"]}
    if op == "hpsi":
        return {"bytes": 32.0 * kets, "flops": flop * terms}
    if op == "observables":
        return {"bytes": 16.0 * kets, "flops": moments}
    if op == "series":
        return {"bytes": 32.0 * kets,
                "flops": 4 * case["steps"] * flop * terms + moments * (case["steps"] // case["every"] + 1)}
    grad_l = 8.0 * terms if op == "autograd" else 0.0
    return {"bytes": 16.0 * kets * (case["steps"] + 2),
            "flops": case["steps"] * (8 * flop * terms + 4 * grad_l) + 2 * moments}


# ------------------------------------------------------------------ the models


def _labels(M):
    return [i - (M - 1) // 2 if M % 2 else i for i in range(M)]


def _dispersion(M):
    lab = np.array(_labels(M), dtype=np.float64)
    return np.abs(lab) if M == 11 else lab ** 2 / 2


def _conserving(case):
    M = case["M"]
    lab = np.array(_labels(M))
    s = lab[:, None, None, None] + lab[None, :, None, None] - lab[None, None, :, None] - lab[None, None, None, :]
    return s == 0 if case["exact"] else s % M == 0


def _coupling(case):
    M, x = case["M"], case["strength"]
    cons = _conserving(case)
    if case["coupling"] == "contact":
        return np.where(cons, x / M, 0.0).astype(np.complex128)
    if case["coupling"] == "long_range":
        lab = np.array(_labels(M), dtype=np.float64)
        d = np.broadcast_to(lab[:, None, None, None] - lab[None, None, :, None], (M, M, M, M))
        val = np.where(d != 0, -x / (M * np.where(d != 0, d, 1.0) ** 2), 0.0)
        return np.where(cons, val, 0.0).astype(np.complex128)
    # a Hermitian coupling without further symmetry: the model is fixed, the states vary
    rng = np.random.default_rng(7)
    L = rng.standard_normal((M, M, M, M)) + 1j * rng.standard_normal((M, M, M, M))
    L = 0.25 * (L + L.transpose(1, 0, 2, 3) + L.transpose(0, 1, 3, 2) + L.transpose(1, 0, 3, 2))
    L = 0.5 * (L + L.transpose(2, 3, 0, 1).conj())
    return np.where(cons, x * L / M, 0.0)


def _range(case):
    n = _nmax(case["state"], case["n_tot"])
    return (0, n) if case["state"] == "coherent" else (n, n)


def _amplitudes(case, seed):
    """A Gaussian momentum profile with n_tot particles and phases from the seed."""
    M = case["M"]
    lab = np.array([i - (M - 1) / 2 for i in range(M)])
    rng = np.random.default_rng(seed)
    z = np.exp(-lab ** 2 / 8) * np.exp(1j * rng.uniform(0.0, 2 * math.pi, M))
    return z * math.sqrt(case["n_tot"] / float(np.sum(np.abs(z) ** 2)))


def _twist(seed):
    """The strength of the interaction phases that an observed state has picked up."""
    return 0.02 + 0.03 * np.random.default_rng([seed, 1]).random()


def _number(case, seed):
    """An occupation vector of n_tot particles (total momentum 0 where only that sector is held)."""
    M, n = case["M"], case["n_tot"]
    rng = np.random.default_rng(seed)
    while True:
        occ = np.bincount(rng.integers(0, M, n), minlength=M)
        if not case["p0"] or _momentum(case, occ) == 0:
            return occ.astype(np.int32)


def _momentum(case, occ):
    p = int(np.dot(_labels(case["M"]), occ))
    return p if case["exact"] else p % case["M"]


# ------------------------------------------------------------------ prepare, run


class State:
    pass


def prepare(case, seed):
    s = State()
    s.case, s.op = case, case["op"]
    M = case["M"]
    s.w, s.L = _dispersion(M), _coupling(case)
    lo, hi = _range(case)
    s.z = _amplitudes(case, seed)
    if s.op == "autograd":
        s.scale = torch.tensor(1.0, dtype=torch.float64, requires_grad=True)
        s.wt = torch.tensor(s.w, dtype=torch.float64, requires_grad=True)
        s.zt = torch.tensor(s.z, dtype=torch.complex128, requires_grad=True)
        s.Lt = torch.tensor(s.L, dtype=torch.complex128, requires_grad=True)
        s.spec = dict(M=M, n_min=lo, n_max=hi, dt=case["dt"], steps=case["steps"], ckpt_every=case["ckpt"],
                      loss=case["loss"])
        return s
    s.space = qb.Space(M, s.w, s.L, lo, hi, [0] if case["p0"] else None, exact=case["exact"])
    if s.op == "adjoint":
        n = int(api.lib().qb_adjoint_workspace_bytes(s.space._h, case["steps"], case["ckpt"]))
        s.work = torch.empty(n, dtype=torch.uint8, device=DEV)
        return s
    psi = torch.empty(s.space.total, dtype=torch.complex128, device=DEV)
    if case["state"] == "number":
        s.space.init_number(_number(case, seed), psi)
    elif case["state"] == "field":
        s.space.init_field_number(s.z, case["n_tot"], psi)
    else:
        s.space.init_coherent(s.z, psi)
    if s.op in ("observables", "hpsi"):
        n = s.space.basis()
        psi *= torch.exp(-1j * _twist(seed) * (n * (n - 1)).sum(1).to(torch.float64))
        s.out = torch.empty_like(psi) if s.op == "hpsi" else None
    elif s.op == "sweep":
        s.scale = [0.25 * (k + 1) for k in range(case["batch"])]
        psi = psi.repeat(case["batch"], 1)
        s.work = s.space.workspace(case["batch"])
    else:
        s.work = s.space.workspace(1)
    s.psi = psi
    return s


_OBS = ("norm", "N", "H", "n_tot", "Q", "lam_p", "PO", "gap", "Vminus_p", "a", "Mij", "aa", "eigvals", "Vminus_modes")


def _observed(rows):
    """The observables of the samples as arrays; the principal mode, whose phase is free, as its projector."""
    out = {k: np.stack([np.asarray(r[k]) for r in rows]) for k in _OBS}
    out["principal"] = np.stack([np.outer(r["xi"], np.conj(r["xi"])) for r in rows])
    return out


def run(s):
    case = s.case
    if s.op == "evolve":
        s.space.evolve(s.psi, case["dt"], case["steps"], s.work)
        return {"psi": s.psi}
    if s.op == "sweep":
        s.space.evolve_batch(s.psi, s.scale, case["dt"], case["steps"], s.work)
        return {"psi": s.psi}
    if s.op == "hpsi":
        s.space.hpsi(s.psi, s.out)
        return {"hpsi": s.out}
    if s.op == "observables":
        return _observed([s.space.observables(s.psi)])
    if s.op == "series":
        rows = s.space.evolve_observe(s.psi, case["dt"], case["steps"], case["every"], s.work)
        return {**_observed(rows), "psi": s.psi}
    if s.op == "adjoint":
        return s.space.adjoint(s.z, 1.0, case["dt"], case["steps"], case["ckpt"], case["loss"], s.work)
    for t in (s.scale, s.wt, s.zt, s.Lt):
        t.grad = None
    loss = qb.adjoint_loss(s.scale, s.wt, s.zt, s.Lt, **s.spec)
    loss.backward()
    return {"loss": loss.detach(), "grad_scale": s.scale.grad, "grad_w": s.wt.grad, "grad_z": s.zt.grad,
            "grad_L": s.Lt.grad}


# ------------------------------------------------------------------ in 64 bits


class Fock:
    """The kets of a space in its order, and its operators, in plain 64-bit torch."""

    def __init__(self, case):
        self.case = case
        M, (lo, hi) = case["M"], _range(case)
        self.M = M
        rem = torch.arange(lo, hi + 1, device=DEV)
        total = rem.clone()
        occ = []
        for m in range(M):
            if m == M - 1:
                occ.append(rem.to(torch.uint8))
                break
            k = rem + 1
            at = torch.repeat_interleave(torch.arange(rem.numel(), device=DEV), k)
            val = torch.arange(at.numel(), device=DEV) - (torch.cumsum(k, 0) - k)[at]
            occ = [o[at] for o in occ] + [val.to(torch.uint8)]
            total, rem = total[at], rem[at] - val
            del at, val
        lab = _labels(M)
        P = sum(lab[m] * occ[m].long() for m in range(M))
        if not case["exact"]:
            P %= M
        if case["p0"]:
            keep = P == 0
            occ, P, total = [o[keep] for o in occ], P[keep], total[keep]
        self.base = hi + 2
        span = 2 * (max(abs(v) for v in lab) * hi + 1) if case["exact"] else M
        key = (total * span + P + (span // 2 if case["exact"] else 0)) * self.base ** M
        self.unit = [self.base ** (M - 1 - m) for m in range(M)]
        for m in range(M):
            key += occ[m].long() * self.unit[m]
        del P, rem
        self.key, order = torch.sort(key)
        self.occ = [o[order] for o in occ]
        self.total = total[order]
        self.span = span
        self.n = self.key.numel()
        self.sqrt = torch.sqrt(torch.arange(hi + 4, device=DEV, dtype=torch.float64))
        self.lab = lab
        self.cache = {}
        del order, key

    def at(self, change):
        """(index, held) of the kets n + change, change = {mode: particles}."""
        key = self.key
        d = sum(v * self.unit[m] for m, v in change.items())
        dn, dp = sum(change.values()), sum(self.lab[m] * v for m, v in change.items())
        if not dn and (dp == 0 if self.case["exact"] else dp % self.M == 0):
            key = key + d
        else:
            sec = self.key // self.base ** self.M
            tot, P = sec // self.span + dn, sec % self.span
            if self.case["exact"]:
                P = P + dp
            else:
                P = (P + dp) % self.M
            key = (tot * self.span + P) * self.base ** self.M + self.key % self.base ** self.M + d
        ok = torch.ones(self.n, dtype=torch.bool, device=DEV)
        for m, v in change.items():
            if v < 0:
                ok &= self.occ[m] >= -v
        i = torch.searchsorted(self.key, key).clamp_(max=self.n - 1)
        ok &= self.key[i] == key
        return i.to(torch.int32), ok

    def pairs(self):
        """{(a, b, c, d): a <= b, c <= d} that conserve momentum: the operators a_a^+ a_b^+ a_c a_d."""
        cons = _conserving(self.case)
        M = self.M
        return [(a, b, c, d) for a in range(M) for b in range(a, M) for c in range(M) for d in range(c, M)
                if cons[a, b, c, d]]

    def two_body(self, op, psi):
        """a_a^+ a_b^+ a_c a_d psi: row n takes the ket n - a - b + c + d."""
        a, b, c, d = op
        if op not in self.cache:
            change = {}
            for m, v in ((a, -1), (b, -1), (c, 1), (d, 1)):
                change[m] = change.get(m, 0) + v
            na, nb = self.occ[a].int(), self.occ[b].int() - int(a == b)
            ok = (na >= 1) & (nb >= 1)
            i, held = self.at({m: v for m, v in change.items() if v})
            # the particles left after a and b are taken away, then c and d put back
            left = lambda m: self.occ[m].int() - int(m == a) - int(m == b)  # noqa: E731
            mc, md = left(c) + 1, left(d) + 1 + int(c == d)
            s = lambda k: self.sqrt[k.clamp(min=0).long()]  # noqa: E731
            coef = s(na) * s(nb) * s(mc) * s(md) * (ok & held)
            if self.n * len(self.pairs()) * 12 > 120e9:
                return coef * psi[i.long()]
            self.cache[op] = (i, coef)
        i, coef = self.cache[op]
        return coef * psi[i.long()]

    def hamiltonian(self, psi, w, couplings):
        """(sum w n + sum L a^+ a^+ a a) psi; couplings: {op: value}."""
        out = torch.zeros_like(psi)
        for m in range(self.M):
            out += float(w[m]) * self.occ[m].double() * psi
        for op, v in couplings.items():
            if v != 0:
                out += (v if v.imag else v.real) * self.two_body(op, psi)
        return out

    def couplings(self, L, scale=1.0):
        """Coefficient of each pair operator: the sum over its orderings."""
        got = {}
        for a, b, c, d in self.pairs():
            v = sum(L[p, q, r, s] for p, q in {(a, b), (b, a)} for r, s in {(c, d), (d, c)})
            got[(a, b, c, d)] = complex(v) * scale
        return got

    def coherent(self, z, only=None):
        """prod z_i^n_i / sqrt(n_i!), normalised over the kets held."""
        hi = int(self.total.max())
        fact = torch.sqrt(torch.exp(torch.lgamma(torch.arange(hi + 1, dtype=torch.float64) + 1))).to(DEV)
        psi = torch.ones(self.n, dtype=torch.complex128, device=DEV)
        zd = torch.as_tensor(z, dtype=torch.complex128, device=DEV) if not torch.is_tensor(z) else z.to(DEV)
        for m in range(self.M):
            row = [torch.ones((), dtype=torch.complex128, device=DEV)]
            for v in range(1, hi + 1):
                row.append(row[-1] * zd[m])
            psi = psi * (torch.stack(row) / fact)[self.occ[m].long()]
        return psi / torch.sqrt((psi.real ** 2 + psi.imag ** 2).sum())

    def rk4(self, psi, apply, dt, steps):
        for _ in range(steps):
            v = psi
            for d in (4, 3, 2, 1):
                v = psi - (1j * dt / d) * apply(v)
            psi = v
        return psi

    def moments(self, psi):
        """<a_i>, <a_i^+ a_j>, <a_i a_j>, normalised."""
        M = self.M
        nrm = (psi.real ** 2 + psi.imag ** 2).sum()
        bra = psi.conj() / nrm
        s = lambda k: self.sqrt[k.clamp(min=0).long()]  # noqa: E731

        def mean(change, coef):
            i, ok = self.at(change)
            return (bra * (coef * ok * psi[i.long()])).sum()

        n = [o.int() for o in self.occ]
        # row n: (a_i psi)_n = sqrt(n_i + 1) psi[n + e_i]
        a = torch.stack([mean({i: 1}, s(n[i] + 1)) for i in range(M)])
        Mij = torch.zeros((M, M), dtype=torch.complex128, device=DEV)
        aa = torch.zeros((M, M), dtype=torch.complex128, device=DEV)
        rows, cols = [], []
        for i in range(M):
            for j in range(M):
                if i == j:
                    rows.append((bra * n[i].double() * psi).sum())
                else:  # (a_i^+ a_j psi)_n = sqrt(n_i (n_j + 1)) psi[n - e_i + e_j]
                    rows.append(mean({i: -1, j: 1}, s(n[i]) * s(n[j] + 1)))
                if j >= i:
                    cols.append(mean({i: 2}, s(n[i] + 1) * s(n[i] + 2)) if i == j else
                                mean({i: 1, j: 1}, s(n[i] + 1) * s(n[j] + 1)))
                else:
                    cols.append(cols[j * M + i])
        return nrm, a, torch.stack(rows).reshape(M, M), torch.stack(cols).reshape(M, M)

    def observables(self, psi, w, couplings):
        nrm, a, Mij, aa = self.moments(psi)
        H = (psi.conj() * self.hamiltonian(psi, w, couplings)).sum().real / nrm
        N = ((psi.real ** 2 + psi.imag ** 2) * self.total.double()).sum() / nrm
        nrm, H, N = float(nrm), float(H), float(N)
        a, Mij, aa = (x.cpu().numpy() for x in (a, Mij, aa))
        n_tot = float(np.trace(Mij).real)
        cov = Mij - np.outer(a.conj(), a)
        var = aa - np.outer(a, a)
        eig, vec = np.linalg.eigh(Mij)
        xi = vec[:, -1]
        dd, vv = (xi.conj() @ cov @ xi).real, xi @ var @ xi
        return {"norm": nrm, "N": N, "H": H, "n_tot": n_tot, "Q": float(np.trace(cov).real) / n_tot, "lam_p": eig[-1],
                "PO": 1 - eig[-1] / n_tot, "gap": eig[-1] - eig[-2], "Vminus_p": 1 + 2 * dd - 2 * abs(vv), "a": a,
                "Mij": Mij, "aa": aa, "eigvals": eig, "xi": xi,
                "Vminus_modes": 1 + 2 * np.diag(cov).real - 2 * np.abs(np.diag(var))}


class _Apply(torch.autograd.Function):
    """H psi with its gradients: H is Hermitian, so the costate of psi is H times the result's."""

    @staticmethod
    def forward(ctx, psi, wt, vals, fock, ops, w, couplings):
        ctx.save_for_backward(psi)
        ctx.rest = fock, ops, w, couplings
        return fock.hamiltonian(psi, w, couplings)

    @staticmethod
    def backward(ctx, g):
        psi, = ctx.saved_tensors
        fock, ops, w, couplings = ctx.rest
        gw = torch.stack([(g.conj() * fock.occ[m].double() * psi).sum().real for m in range(fock.M)])
        gv = torch.stack([(fock.two_body(op, psi).conj() * g).sum() for op in ops])
        return fock.hamiltonian(g, w, couplings), gw.cpu(), gv.cpu(), None, None, None, None


def _gradients(case, seed):
    fock = Fock(case)
    M, w, L = case["M"], _dispersion(case["M"]), _coupling(case)
    z = torch.tensor(_amplitudes(case, seed), dtype=torch.complex128, requires_grad=True)
    wt = torch.tensor(w, dtype=torch.float64, requires_grad=True)
    ops, couplings = fock.pairs(), fock.couplings(L)
    vals = torch.tensor([couplings[op] for op in ops], dtype=torch.complex128, requires_grad=True)
    psi = fock.rk4(fock.coherent(z), lambda v: _Apply.apply(v, wt, vals, fock, ops, w, couplings), case["dt"],
                   case["steps"])
    nrm, a, Mij, aa = fock.moments(psi)
    if case["loss"] == "Q":
        n_tot = torch.diagonal(Mij).real.sum()
        loss = 1 - (a.real ** 2 + a.imag ** 2).sum() / n_tot
    else:
        loss = torch.linalg.eigvalsh(0.5 * (Mij + Mij.conj().T))[-1]
    loss.backward()
    # the orderings of a pair operator are one operator: each entry has its gradient
    grad_l = np.zeros((M, M, M, M), dtype=np.complex128)
    for (a_, b, c, d), g in zip(ops, vals.grad.numpy()):
        for p, q in {(a_, b), (b, a_)}:
            for r, s in {(c, d), (d, c)}:
                grad_l[p, q, r, s] = g
    cv = np.array([couplings[op] for op in ops])
    scale = float(np.sum((np.conj(vals.grad.numpy()) * cv).real))
    return float(loss.detach()), scale, wt.grad.numpy(), z.grad.numpy(), grad_l


def exact(case, seed):
    op, M = case["op"], case["M"]
    passes = {"hpsi": 1, "observables": 2}.get(op) or 4 * case["steps"] * case.get("batch", 1)
    cost = (_terms(case) + 2 * _kets(M, case["state"], case["n_tot"], case["p0"])) * 1.6e-9
    cost += 400e-6 * passes * len(_labels(M)) ** 2
    cost += passes * _terms(case) * {"adjoint": 3.0, "autograd": 3.0}.get(op, 1.0) * 3e-10
    if cost > 15:
        return None
    if op in ("adjoint", "autograd"):
        loss, gs, gw, gz, gl = _gradients(case, seed)
        if op == "adjoint":
            return {"loss": loss, "grad_scale": gs, "grad_w": gw, "grad_z": gz}
        return {"loss": torch.tensor(loss, dtype=torch.float64), "grad_scale": torch.tensor(gs, dtype=torch.float64),
                "grad_w": torch.tensor(gw), "grad_z": torch.tensor(gz), "grad_L": torch.tensor(gl)}
    fock = Fock(case)
    w, L = _dispersion(M), _coupling(case)
    if case["state"] == "number":
        occ = _number(case, seed)
        hit = torch.ones(fock.n, dtype=torch.bool, device=DEV)
        for m in range(M):
            hit &= fock.occ[m] == int(occ[m])
        psi = hit.to(torch.complex128)
    else:
        psi = fock.coherent(_amplitudes(case, seed))
    couplings = fock.couplings(L)
    if op in ("observables", "hpsi"):
        phase = sum(o.double() * (o.double() - 1) for o in fock.occ)
        psi = psi * torch.exp(-1j * _twist(seed) * phase)
    if op == "hpsi":
        return {"hpsi": fock.hamiltonian(psi, w, couplings)}
    if op == "observables":
        return _observed([fock.observables(psi, w, couplings)])
    if op == "sweep":
        rows = []
        for k in range(case["batch"]):
            c = {o: v * 0.25 * (k + 1) for o, v in couplings.items()}
            rows.append(fock.rk4(psi, lambda v: fock.hamiltonian(v, w, c), case["dt"], case["steps"]))
        return {"psi": torch.stack(rows)}
    if op == "series":
        rows = [fock.observables(psi, w, couplings)]
        for _ in range(case["steps"] // case["every"]):
            psi = fock.rk4(psi, lambda v: fock.hamiltonian(v, w, couplings), case["dt"], case["every"])
            rows.append(fock.observables(psi, w, couplings))
        return {**_observed(rows), "psi": psi}
    return {"psi": fock.rk4(psi, lambda v: fock.hamiltonian(v, w, couplings), case["dt"], case["steps"])}
