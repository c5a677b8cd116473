"""The work that a user of this library has it do, as cases that can be timed and compared.

A solve is what most programs do: an Exact-Cover-3 Hamiltonian, a path, an initial state, a
number of grid steps, then the state with its success probability, energy and norm.  Small states
(n <= 12) are solved alone and whole, the middle sizes (n = 14..20) are what batches, sweeps and
the serving loop are made of, and the large ones (n = 22..28) are bound by memory.  Beside the
solves: the stand-alone matvec, a batch of small states stepped together, and the Lanczos solve
that gives the gap above the ground state.  Every input is seeded: the instance (its clauses and
couplings) comes from the seed.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from instances import SplitMix64, generate_ec3, xx_pairs
from paper_1311_3938_gb300 import AQC_C64, AQC_C128
from paper_1311_3938_gb300 import hamiltonians as HB
from paper_1311_3938_gb300.engine import Batch, Context

# A state whose integrator vectors (y, the predictor, three derivatives) fit the second-level
# cache need not go through memory on every step.
_CACHE_BYTES = 126e6
_KAPPA = 0.1


def listed():
    return [
        # one small state alone, whole: the latency of a step is all there is
        {"name": "solve_c128_n10", "kind": "solve", "n": 10, "prec": "c128", "path": "linear", "s": 0, "T": 20.0,
         "steps": -1, "opt": ""},
        # the same in the precision of batches and sweeps, with couplings: smallest batch size
        {"name": "solve_c64_n12", "kind": "solve", "n": 12, "prec": "c64", "path": "nonlinear", "s": 1, "T": 10.0,
         "steps": -1, "opt": ""},
        # a middle size: several tiles, state far inside the cache
        {"name": "solve_c64_n16", "kind": "solve", "n": 16, "prec": "c64", "path": "nonlinear", "s": 0, "T": 50.0,
         "steps": 512, "opt": ""},
        # the 20-qubit sweep: nonlinear path, smoothstep schedule
        {"name": "solve_c64_n20", "kind": "solve", "n": 20, "prec": "c64", "path": "nonlinear", "s": 1, "T": 50.0,
         "steps": 256, "opt": ""},
        # the same sweep's reference runs in double precision
        {"name": "solve_c128_n20", "kind": "solve", "n": 20, "prec": "c128", "path": "linear", "s": 0, "T": 50.0,
         "steps": 64, "opt": ""},
        # a served request beyond the cache, a size with a ragged last layout
        {"name": "solve_c64_n23", "kind": "solve", "n": 23, "prec": "c64", "path": "linear", "s": 0, "T": 100.0,
         "steps": 64, "opt": ""},
        # the XY algorithm with its catalyst, from the Dicke state of the solution's sector
        {"name": "xy_c64_n24", "kind": "solve", "n": 24, "prec": "c64", "path": "xy", "s": 0, "T": 20.0,
         "steps": 32, "opt": ""},
        # the full-size instance: 2 GiB per vector
        {"name": "solve_c64_n28", "kind": "solve", "n": 28, "prec": "c64", "path": "linear", "s": 0, "T": 100.0,
         "steps": 24, "opt": ""},
        # a large double-precision solve
        {"name": "solve_c128_n26", "kind": "solve", "n": 26, "prec": "c128", "path": "linear", "s": 0, "T": 100.0,
         "steps": 12, "opt": ""},
        # the stand-alone matvec H(t) psi on a caller's vector
        {"name": "hpsi_c64_n26", "kind": "hpsi", "n": 26, "prec": "c64", "path": "linear", "s": 0, "T": 100.0,
         "steps": 0, "opt": ""},
        # a batch of uneven instances, each from its start through 256 grid steps
        {"name": "batch_c64_24", "kind": "batch", "n": 12, "prec": "c64", "path": "nonlinear", "s": 0, "T": 60.0,
         "steps": 256, "opt": "", "members": 24, "n_max": 18},
        # one point of a gap curve: the two lowest Ritz values after 64 Lanczos steps
        {"name": "lanczos_c128_n16", "kind": "lanczos", "n": 16, "prec": "c128", "path": "linear", "s": 0, "T": 1.0,
         "steps": 64, "opt": ""},
    ]


def draw(rng):
    kind = rng.choice(["solve"] * 7 + ["hpsi", "hpsi", "batch", "lanczos"])
    prec = rng.choice(["c64", "c64", "c128"])
    path = rng.choice(["linear", "nonlinear", "xy"])
    s = rng.choice([0, 1])
    if kind == "solve":
        n = rng.randint(5, 27 if prec == "c64" else 24)
        if path == "xy":
            n = min(n, 24 if prec == "c64" else 21)
        if path == "nonlinear" and prec == "c128":
            n = min(n, 22)
        # a few hundred steps, fewer as the state grows, so that a pass takes tens of milliseconds
        most = min(600.0, 2.0 ** ((30 if prec == "c64" else 27 if path == "linear" else 26) - n))
        steps = max(8, int(rng.uniform(0.5, 1.0) * most))
        # an option of the integrator now and then: the compensated corrector (complex64), or
        # step-size control at a tolerance every step meets (complex128)
        opt = rng.choice(["", "", "", "ycomp" if prec == "c64" else "adaptive"])
        return {"kind": kind, "n": n, "prec": prec, "path": path, "s": s, "T": round(rng.uniform(40.0, 200.0), 3),
                "steps": steps, "opt": opt}
    if kind == "hpsi":
        n = rng.randint(6, 27 if prec == "c64" else 25)
        return {"kind": kind, "n": n, "prec": prec, "path": "linear" if n > 24 else path, "s": s,
                "T": round(rng.uniform(40.0, 200.0), 3), "steps": 0, "opt": ""}
    if kind == "batch":
        lo = rng.randint(6, 13)
        return {"kind": kind, "n": lo, "prec": prec, "path": "nonlinear" if path == "xy" else path, "s": s,
                "T": round(rng.uniform(60.0, 200.0), 3), "steps": rng.choice([64, 128, 192, 256]), "opt": "",
                "members": rng.randint(4, 32), "n_max": lo + rng.randint(0, 4)}
    return {"kind": kind, "n": rng.randint(9, 18), "prec": prec, "path": "linear" if path == "xy" else path, "s": s,
            "T": 1.0, "steps": rng.choice([24, 40, 56, 64]), "opt": ""}


# ---- the instance of a case ---------------------------------------------------------------------

def _members(case, seed):
    """(n, instance seed) of each state a case holds."""
    if case["kind"] != "batch":
        return [(case["n"], 1 + seed % (1 << 30))]
    rng = SplitMix64(case["members"] * 7919 + 17)  # the mix of sizes belongs to the case
    return [(case["n"] + rng.below(case["n_max"] - case["n"] + 1), 1 + (seed + 131 * k) % (1 << 30))
            for k in range(case["members"])]


def _data(n, iseed, path):
    """Clauses, solution and the couplings of the nonlinear path (none for other paths)."""
    inst = generate_ec3(n, iseed)
    pairs = xx_pairs(n, iseed, min(2 * n, n * (n - 1) // 2)) if path == "nonlinear" else []
    return inst, pairs


def _removed(n, clauses):
    """The clause that the catalyst H_{m-1} of the XY algorithm lacks (None without a catalyst)."""
    rem = HB.removable_clauses(n, list(clauses))
    return rem[-1] if rem else len(clauses) - 1


_ALPHA = 8.0  # catalyst strength of the XY algorithm


def _context(case, n, iseed):
    prec = AQC_C64 if case["prec"] == "c64" else AQC_C128
    inst, pairs = _data(n, iseed, case["path"])
    ctx = Context(n, prec, extra_vector=case["opt"] != "")
    if case["path"] == "xy":
        sched, weight = HB.load_xy(ctx, inst, driver="xy", catalyst_alpha=_ALPHA,
                                   removed=_removed(n, inst.clauses))
        start = ("dicke", weight)
    else:
        HB.load_ec3(ctx, inst, pairs=pairs)
        sched = HB.nonlinear_schedule() if pairs else HB.linear_schedule()
        start = "uniform"
    ctx.set_schedule(case["T"], sched, case["s"])
    if case["opt"] == "adaptive":
        ctx.set_integrator(0, 0.0, adaptive=True, tol=1.0)
        ctx.set_step_growth(0)
    else:
        ctx.set_integrator(0, 0.0)
    if case["opt"] == "ycomp":
        ctx.set_y_compensation(True)
    return ctx, inst, start


def _vector(n, seed, prec):
    """A normalised random state on the GPU."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    v = torch.randn(1 << n, 2, generator=g, device="cuda", dtype=torch.float64)
    v = torch.view_as_complex(v / v.norm())
    return v.to(torch.complex64) if prec == "c64" else v


def prepare(case, seed):
    state = {"case": case, "members": [_context(case, n, iseed) for n, iseed in _members(case, seed)]}
    if case["kind"] in ("hpsi", "lanczos"):
        state["psi"] = _vector(case["n"], seed, case["prec"])
    if case["kind"] == "batch":
        ns = [n for n, _ in _members(case, seed)]
        items = 1024 + sum(1 << max(0, n - 5) for n in ns)
        state["batch"] = Batch(AQC_C64 if case["prec"] == "c64" else AQC_C128, max_members=len(ns), max_items=items)
    return state


def run(state):
    case = state["case"]
    ctx, inst, start = state["members"][0]
    if case["kind"] == "hpsi":
        return ctx.hpsi(0.4 * case["T"], state["psi"])
    if case["kind"] == "lanczos":
        eig, _, iters = ctx.lanczos(0.4 * case["T"], state["psi"], max_iter=case["steps"], n_eig=2, tol=0.0)
        return {"eig": np.array(eig, dtype=np.float32 if case["prec"] == "c64" else np.float64), "iters": int(iters)}
    if case["kind"] == "solve":
        ctx.set_initial_state(start)
        stats = ctx.propagate(case["steps"])
        return {"psi": ctx.state(device=True), "P1": ctx.fidelity(inst.solution), "E": ctx.energy(),
                "norm2": stats["norm2"], "steps": int(stats["steps_done"])}
    # a batch: every member from its initial state through 3 + steps grid steps
    b = state["batch"]
    slots = []
    for c, _, st in state["members"]:
        c.set_initial_state(st)
        slots.append(b.add(c))
    b.run(case["steps"] // b.steps_per_round)
    steps, _, _ = b.poll()
    out = []
    for slot in slots:
        c = b.remove(slot)
        out.append({"psi": c.state(device=True), "steps": int(steps[slot])})
    return out


# ---- what a pass cannot do without --------------------------------------------------------------

def _terms(n, m, path):
    """Off-diagonal products of one instance (a hop counts as one)."""
    return {"linear": n, "nonlinear": 3 * n, "xy": 2.5 * m}[path]


def work(case):
    amp = 8.0 if case["prec"] == "c64" else 16.0
    if case["kind"] == "batch":
        mid = range(case["n"], case["n_max"] + 1)
        parts = [(n, case["members"] / len(mid)) for n in mid]
    else:
        parts = [(case["n"], 1.0)]
    nbytes = flops = 0.0
    for n, count in parts:
        N = 2.0 ** n
        per_eval = 4.0 * _terms(n, 1.2 * n, case["path"]) + 4.0
        if case["kind"] == "hpsi":
            nbytes += count * 2.0 * N * amp
            flops += count * N * per_eval
            continue
        if case["kind"] == "lanczos":
            k = case["steps"]
            # the Krylov basis is read for each of two orthogonalisations, and written once
            nbytes += count * N * amp * (k * (k + 1) + 2.0 * k)
            flops += count * N * (k * per_eval + 16.0 * k * (k + 1))
            continue
        steps = case["steps"] if case["steps"] > 0 else case["T"] * n / _KAPPA
        steps += 3 if case["kind"] == "batch" else 0
        fits = 5.0 * N * amp <= _CACHE_BYTES
        # the state comes in and goes out; a state beyond the cache also reads y and the derivatives
        # and writes y and the new derivative on every step (18 vectors per Runge-Kutta step)
        nbytes += count * N * amp * (2.0 if fits else 2.0 + 3 * 18.0 + 8.0 + 7.0 * max(0, steps - 3))
        flops += count * N * ((13 + max(0, steps - 3)) * per_eval + 42.0 * steps)
    return {"bytes": nbytes, "flops": flops}


# ---- the same in 64 bits, with plain torch ------------------------------------------------------

class _Dense64:
    """H(s) of one instance as a diagonal per group and strided-view updates, complex128."""

    def __init__(self, case, n, iseed):
        inst, pairs = _data(n, iseed, case["path"])
        self.n, self.N, self.case = n, 1 << n, case
        z = torch.arange(self.N, device="cuda", dtype=torch.int32)

        def penalty(clauses):
            e = torch.zeros(self.N, device="cuda", dtype=torch.float64)
            for c in clauses:
                e += (sum(((z >> b) & 1) for b in c) != 1)
            return e

        cl = list(inst.clauses)
        self.solution = inst.solution
        self.ident = 0.0
        self.flips, self.hops = [], []  # (group, bits, coefficient)
        self.diag = [None, penalty(cl), None]
        self.bound = [0.0, float(len(cl)), 0.0]
        self.alpha = 0.0
        if case["path"] == "xy":
            nij = {}
            for c in cl:
                a, b, d = sorted(c)
                for key in ((a, b), (a, d), (b, d)):
                    nij[key] = nij.get(key, 0) + 1
            self.ident = 3.0 * len(cl)
            self.hops = [(i, j, -v / 2.0) for (i, j), v in sorted(nij.items())]
            self.bound[0] = 3.0 * len(cl) + sum(2 * (v / 2.0) for _, v in sorted(nij.items()))
            k = _removed(n, inst.clauses)
            self.diag[2] = penalty(cl[:k] + cl[k + 1:])
            self.bound[2] = float(len(cl) - 1)
            self.alpha = _ALPHA
            w = bin(int(inst.solution)).count("1")
            ones = sum(((z >> b) & 1) for b in range(n))
            self.y0 = (ones == w).to(torch.complex128) / math.sqrt(math.comb(n, w))
        else:
            self.ident = 0.5 * n
            self.flips = [(0, (q,), -0.5) for q in range(n)] + [(2, (i, j), J) for (i, j, J) in pairs]
            self.bound[0] = 0.5 * n + sum(0.5 for _ in range(n))
            self.bound[2] = sum(abs(J) for (_, _, J) in pairs)
            self.alpha = 1.0 if pairs else 0.0
            self.y0 = torch.full((self.N,), 1.0 / math.sqrt(self.N), device="cuda", dtype=torch.complex128)

    def weights(self, s):
        return (1.0 - s, s, self.alpha * s * (1.0 - s))

    def s_of(self, t):
        tau = t / self.case["T"]
        return tau * tau * (3.0 - 2.0 * tau) if self.case["s"] else tau

    def grid(self):
        lam = max(sum(abs(w) * b for w, b in zip(self.weights(i / 1024.0), self.bound)) for i in range(1025))
        return max(4, math.ceil(self.case["T"] * lam / _KAPPA))

    def apply(self, w, psi):
        d = w[0] * self.ident + (w[1] * self.diag[1] if w[1] else 0.0)
        if self.diag[2] is not None:
            d = d + w[2] * self.diag[2]
        out = d * psi
        for g, bits, c in self.flips:
            cw = c * w[g]
            if cw == 0.0:
                continue
            if len(bits) == 1:
                o, p = out.view(-1, 2, 1 << bits[0]), psi.view(-1, 2, 1 << bits[0])
                o[:, 0].add_(p[:, 1], alpha=cw)
                o[:, 1].add_(p[:, 0], alpha=cw)
            else:
                i, j = bits
                o, p = (v.view(-1, 2, 1 << (j - i - 1), 2, 1 << i) for v in (out, psi))
                for a in (0, 1):
                    for b in (0, 1):
                        o[:, a, :, b].add_(p[:, 1 - a, :, 1 - b], alpha=cw)
        for i, j, c in self.hops:
            cw = 2.0 * c * w[0]
            o, p = (v.view(-1, 2, 1 << (j - i - 1), 2, 1 << i) for v in (out, psi))
            o[:, 0, :, 1].add_(p[:, 1, :, 0], alpha=cw)
            o[:, 1, :, 0].add_(p[:, 0, :, 1], alpha=cw)
        return out

    def f(self, t, psi):
        return self.apply(self.weights(self.s_of(t)), psi).mul_(-1j)

    def solve(self, steps):
        """Three Runge-Kutta steps, then the predictor-corrector, on the step rule's grid."""
        N = self.grid()
        h = self.case["T"] / N
        steps = N if steps < 0 else min(steps, N)
        y, hist = self.y0.clone(), []
        for k in range(min(3, steps)):
            t = k * h
            k1 = self.f(t, y)
            k2 = self.f(t + h / 2, y + (h / 2) * k1)
            k3 = self.f(t + h / 2, y + (h / 2) * k2)
            k4 = self.f(t + h, y + h * k3)
            y = y + (h / 6) * (k1 + 2 * k2 + 2 * k3 + k4)
            hist.append(k1)
            del k2, k3, k4
        if steps > 3:
            hist.append(self.f(3 * h, y))
            for k in range(3, steps):
                f3, f2, f1, f0 = hist
                p = y + (h / 24) * (55 * f0 - 59 * f1 + 37 * f2 - 9 * f3)
                fn = self.f((k + 1) * h, p)
                y = y + (h / 24) * (9 * fn + 19 * f0 - 5 * f1 + f2)
                hist = [f2, f1, f0, fn]
        return y, steps


def exact(case, seed):
    (n, iseed), kind = _members(case, seed)[0], case["kind"]
    if kind == "batch":
        out = []
        for n, iseed in _members(case, seed):
            y, steps = _Dense64(case, n, iseed).solve(3 + case["steps"])
            out.append({"psi": y, "steps": steps})
        return out
    H = _Dense64(case, n, iseed)
    if kind == "hpsi":
        return H.apply(H.weights(H.s_of(0.4 * case["T"])), _vector(n, seed, case["prec"]).to(torch.complex128))
    if kind == "lanczos":
        w = H.weights(H.s_of(0.4 * case["T"]))
        V = torch.empty(case["steps"] + 1, H.N, device="cuda", dtype=torch.complex128)
        v = _vector(n, seed, case["prec"]).to(torch.complex128)
        V[0] = v / v.norm()
        a, b = [], []
        for j in range(case["steps"]):
            r = H.apply(w, V[j])
            alpha = 0.0
            for _ in range(2):
                c = V[:j + 1].conj() @ r
                alpha += float(c[j].real)
                r = r - V[:j + 1].T @ c
            a.append(alpha)
            b.append(float(r.norm()))
            V[j + 1] = r / b[-1]
        ritz = np.linalg.eigvalsh(np.diag(a) + np.diag(b[:-1], 1) + np.diag(b[:-1], -1))
        return {"eig": ritz[:2].copy(), "iters": None}
    y, steps = H.solve(case["steps"])
    p = y.abs().square()
    return {"psi": y, "P1": float(p[H.solution]), "E": float((p * H.diag[1]).sum()), "norm2": float(p.sum()),
            "steps": steps}
