"""The workloads this framework's speed is judged on, through its public calls.

Each case is one job a user's program has the simulator do, over the range of
sizes, sparsities, precisions and schedules the library takes: quantum walks
from |b~> to the register marginals, CKS linear solves, batches of independent
walks, the paper's literal and register-faithful schedules, and a checkpoint
that is resumed and saved again.  ``exact`` restates the mathematics (W = S (2
T~ Pi T~^dag - 1) on the pairs of a padded sparse matrix, and the Chebyshev sum
of the solver) in 64-bit numpy / torch without any of the library's code.

complex64 simulations return their read-outs in single precision, the
precision their amplitudes carry; complex128 ones in double precision.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2303_06890_gb300 import qwalk
from paper_2303_06890_gb300 import workloads as wl

C128, C64 = "complex128", "complex64"


def listed():
    return [
        # the plain N = 16 walk: the smallest call, all latency and launches
        dict(name="walk_n16_s4_c128", kind="walk", n=16, s=4, matrix="random", precision=C128, steps=10,
             complex_b=False),
        # an ordinary walk of a ragged size, plain FP64 path, 100 steps, complex right-hand side
        dict(name="walk_n1000_s8_c128", kind="walk", n=1000, s=8, matrix="random", precision=C128, steps=100,
             complex_b=True),
        # the headline walk: N = 16384, 16 entries a column, 20 steps, complex64 amplitudes
        dict(name="walk_n16384_s16_c64", kind="walk", n=16384, s=16, matrix="random", precision=C64, steps=20,
             complex_b=False),
        # the same walk on the plain FP64 path
        dict(name="walk_n16384_s16_c128", kind="walk", n=16384, s=16, matrix="random", precision=C128, steps=20,
             complex_b=False),
        # the widest band matrix of the paper's Table 1 (E: s = 64, 3.1 M branches), complex128
        dict(name="walk_n16384_s64_c128", kind="walk", n=16384, s=64, matrix="band", precision=C128, steps=20,
             complex_b=False),
        # the largest N, ragged, near the library's limit of 65536 rows
        dict(name="walk_n50001_s16_c64", kind="walk", n=50001, s=16, matrix="random", precision=C64, steps=20,
             complex_b=False),
        # the linear solver on a matrix of condition number 100 (13 878 walk steps), complex64
        dict(name="qls_n1024_s8_c64", kind="qls", n=1024, s=8, matrix="conditioned", precision=C64, kappa=403.9),
        # the linear solver on a small band matrix (Table 1 B's shape), complex128: many tiny steps
        dict(name="qls_n128_s16_c128", kind="qls", n=128, s=16, matrix="band", precision=C128, kappa=100.0),
        # independent walks of uneven size advanced together, 50 steps
        dict(name="batch_64_s8_c64", kind="batch", count=64, s=8, lo=64, hi=4096, precision=C64, steps=50),
        # the paper's literal schedule: one branch list, a global sort per interference operation
        dict(name="flat_n16384_s16_c128", kind="schedule", schedule="flat", n=16384, s=16, matrix="random", steps=2),
        # the register-faithful schedule on Table 1 D's shape: every working register held in 640-bit keys
        dict(name="faithful_n8192_s32_c128", kind="schedule", schedule="faithful", n=8192, s=32, matrix="band",
             steps=1),
        # resume a saved state, walk on, and save it: the whole state goes in and comes out
        dict(name="resume_n2047_s8_c128", kind="resume", n=2047, s=8, matrix="random", steps=10),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(2.0 ** rng.uniform(math.log2(lo), math.log2(hi))))))


def draw(rng):
    kind = rng.choice(["walk", "walk", "walk", "walk", "qls", "qls", "batch", "schedule", "resume"])
    if kind == "walk":
        s = rng.choice([4, 8, 16, 32, 64])
        n = _log_int(rng, 2 * s, min(50001, (1 << 20) // s))
        return dict(kind=kind, n=n, s=s, matrix="band" if s >= 32 else "random", precision=rng.choice([C128, C64]),
                    steps=rng.randint(1, 20) if n * s > 32768 else rng.randint(1, 100),
                    complex_b=rng.random() < 0.3)
    if kind == "qls":
        s = rng.choice([4, 8, 16])
        return dict(kind=kind, n=_log_int(rng, 4 * s, 1024), s=s, matrix="band" if s == 16 else "conditioned",
                    precision=rng.choice([C128, C64]), kappa=round(rng.uniform(20.0, 300.0), 1))
    if kind == "batch":
        return dict(kind=kind, count=_log_int(rng, 3, 64), s=8, lo=rng.choice([16, 64]), hi=rng.choice([1024, 4096]),
                    precision=rng.choice([C128, C64]), steps=rng.randint(5, 50))
    if kind == "schedule":
        schedule, s = rng.choice(["flat", "faithful"]), rng.choice([4, 8, 16, 32])
        n = _log_int(rng, 2 * s, 16384 * 16 // s if schedule == "flat" else min(16384, 8192 * 16 // s))
        return dict(kind=kind, schedule=schedule, n=min(n, 16384), s=s, matrix="band" if s >= 32 else "random",
                    steps=rng.randint(1, 2))
    s = rng.choice([4, 8, 16])
    return dict(kind=kind, n=_log_int(rng, 4 * s, 4096 * 4 // s), s=s, matrix="random", steps=rng.randint(1, 20))


# --- inputs --------------------------------------------------------------------

def _matrix(kind, n, s, seed):
    if kind == "random":  # diagonal and random symmetric pairs, at most s entries a column
        return wl.random_symmetric(n, s, 1 if s == 8 else 0, (3 * n * s) // 8, seed)
    if kind == "conditioned":  # the solver's matrices: condition number 100
        return wl.conditioned_symmetric(n, s, (3 * n) // 2, 100.0, seed)
    return wl.band_positive(n, s // 2 - 1, 15, seed)  # full positive band, Table 1's shape


def _b(case, n, seed):
    rng = np.random.default_rng(seed)
    b = rng.standard_normal(n)
    if case.get("complex_b"):
        b = b + 1j * rng.standard_normal(n)
    return b / np.linalg.norm(b)


def _inputs(case, seed):
    """The case's matrices and right-hand sides, from the seed alone."""
    if case["kind"] == "resume":  # one matrix, other states: the branch list's length is the matrix's
        return [_matrix(case["matrix"], case["n"], case["s"], case["n"])], [_b(case, case["n"], seed + 1)]
    if case["kind"] != "batch":
        return [_matrix(case["matrix"], case["n"], case["s"], seed)], [_b(case, case["n"], seed + 1)]
    rng = np.random.default_rng(case["count"])  # the batch's sizes are the case's own
    sizes = np.rint(2.0 ** rng.uniform(math.log2(case["lo"]), math.log2(case["hi"]), case["count"])).astype(int)
    return ([wl.random_symmetric(int(n), case["s"], 1, (3 * int(n)) // 2, seed + 2 + i) for i, n in enumerate(sizes)],
            [_b(case, int(n), seed + 1000 + i) for i, n in enumerate(sizes)])


def _precision(case):
    return case.get("precision", C128)


def _sim(case, mats, **kw):
    code = qwalk.QW_FP64 if _precision(case) == C128 else qwalk.QW_FP32_AMP
    return qwalk.Sim(mats if len(mats) > 1 else mats[0], s_pad=case["s"], precision=code, **kw)


def prepare(case, seed):
    mats, bs = _inputs(case, seed)
    state = dict(case=case, bs=bs, ns=[m.n for m in mats])
    if case["kind"] == "schedule":
        state["sim"] = _sim(case, mats, walk_variant=5 if case["schedule"] == "flat" else 6)
        return state
    sim = state["sim"] = _sim(case, mats)
    for i, b in enumerate(bs):
        sim.state_init(b, inst=i)
    sim.autotune()  # the step kernel is chosen once per simulator
    if case["kind"] == "qls":
        state["coeffs"] = qwalk.cks_coefficients(case["kappa"])[0]
    if case["kind"] == "resume":  # what an earlier run saved: the state after T~ and two steps
        sim.state_init(bs[0])
        sim.apply_walk_step(2)
        state["keys"], state["amps"] = sim.state_export()
    return state


# --- one pass ------------------------------------------------------------------

def _real(case, x):
    return x.astype(np.float32) if _precision(case) == C64 else x


def run(state):
    case, sim, bs, ns = state["case"], state["sim"], state["bs"], state["ns"]
    if case["kind"] in ("walk", "schedule"):
        sim.state_init(bs[0])
        sim.enqueue_walk_steps(case["steps"])
        return {"j": _real(case, sim.measure_register("j", ns[0])), "k": _real(case, sim.measure_register("k", ns[0]))}
    if case["kind"] == "qls":
        sim.state_init(bs[0])
        y, p = sim.apply_qls(state["coeffs"])
        return {"y": y.astype(np.complex64) if _precision(case) == C64 else y, "p": _real(case, p)}
    if case["kind"] == "batch":
        for i, b in enumerate(bs):
            sim.state_init(b, inst=i)
        sim.enqueue_walk_steps(case["steps"])
        return {"j": _real(case, np.concatenate([sim.measure_register("j", n, inst=i) for i, n in enumerate(ns)]))}
    sim.state_import(state["keys"], state["amps"])
    sim.apply_walk_step(case["steps"])
    keys, amps = sim.state_export()
    return {"keys": keys, "amps": amps}


# --- what a pass cannot do without ---------------------------------------------

def work(case):
    """Bytes: the right-hand side and the QRAM image read once, the read-out
    written once, and the state read and written once by every walk step (2
    branches of row (j, 0) and 1 of row (j, 1) per QRAM slot; the literal
    schedules read and write the list of keys and amplitudes once for each of
    a step's three interference operations).  Flops: per slot and step the
    rotation into and out of the reflected group and its sum."""
    n = case["n"] if "n" in case else case["count"] * (case["hi"] - case["lo"]) / math.log(case["hi"] / case["lo"])
    s, amp = case["s"], 16 if _precision(case) == C128 else 8
    steps = case.get("steps", 0)
    out = 16 * n
    if case["kind"] == "qls":
        terms = len(qwalk.cks_coefficients(case["kappa"])[0])
        steps, out = 2 * terms, 16 * n + 8 * terms
    branches = 3 * n * s
    per_branch = 2 * amp
    if case["kind"] == "schedule":
        per_branch = 3 * 2 * (16 + (16 if case["schedule"] == "flat" else 80))
    if case["kind"] == "resume":
        out = 2 * branches * 32
    return {"bytes": float(8 * n + 4 * n * s + out + steps * branches * per_branch),
            "flops": float(steps * n * s * 36)}


# --- the same results in 64 bits, from the mathematics alone --------------------

def _padded(m, s):
    """Columns and values [n, s] of the rows completed to s entries with zero
    elements at the first columns j + 1, j + 2, ... (cyclic) not in the row."""
    n = m.n
    count = np.diff(m.colptr).astype(np.int64)
    row = np.repeat(np.arange(n, dtype=np.int64), count)
    have = row * n + m.rowidx
    cand = (np.arange(n, dtype=np.int64)[:, None] + np.arange(1, s + 1)) % n
    free = ~np.isin(np.arange(n, dtype=np.int64)[:, None] * n + cand, have)
    take = free & (np.cumsum(free, axis=1) <= (s - count)[:, None])
    pad_row, at = np.nonzero(take)
    code = np.concatenate([have, pad_row * n + cand[pad_row, at]])
    val = np.concatenate([m.val_q15.astype(np.float64) / 32768.0, np.zeros(len(pad_row))])
    order = np.argsort(code)
    return (code[order] % n).reshape(n, s), val[order].reshape(n, s)


class _Walk:
    """W on amplitudes x[pair, b1, b2] of |j, b1, k, b2> over the ordered pairs
    (j, k) with k in j's padded row or j in k's."""

    def __init__(self, m, s):
        n, (col, val) = m.n, _padded(m, s)
        j = np.repeat(np.arange(n, dtype=np.int64)[:, None], s, axis=1)
        self.n, self.s = n, s
        self.code = np.unique(np.concatenate([(j * n + col).ravel(), (col * n + j).ravel()]))
        self.slot = np.searchsorted(self.code, j * n + col)  # [n, s]
        self.swap = np.searchsorted(self.code, (self.code % n) * n + self.code // n)
        root = np.sqrt(np.abs(val))
        self.f = np.where(val < 0, 1j * np.where(j <= col, 1.0, -1.0), 1.0) * root
        self.g = np.sqrt(1.0 - np.abs(val))

    def start(self, b):
        x = np.zeros((len(self.code), 2, 2), dtype=np.complex128)
        h = (b / math.sqrt(self.s))[:, None]
        x[self.slot, 0, 0] = self.f * h
        x[self.slot, 0, 1] = self.g * h
        return x

    def step(self, x):
        y = -x
        u = np.conj(self.f) * x[self.slot, 0, 0] + self.g * x[self.slot, 0, 1]
        r = (2.0 / self.s) * u.sum(axis=1, keepdims=True)
        y[self.slot, 0, 0] += self.f * r
        y[self.slot, 0, 1] += self.g * r
        return y[self.swap].transpose(0, 2, 1)

    def run(self, b, steps):
        x = self.start(b)
        for _ in range(steps):
            x = self.step(x)
        return x

    def marginal(self, x, reg):
        p = (x.real ** 2 + x.imag ** 2).sum(axis=(1, 2))
        return np.bincount(self.code // self.n if reg == "j" else self.code % self.n, weights=p, minlength=self.n)


def _solve(case, m, b):
    """Y = sum_j a_j T_{2j+1}(A/s) b and ||.||^2 of its partial sums, by the
    Chebyshev recurrence."""
    coeffs = qwalk.cks_coefficients(case["kappa"])[0]
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    a = torch.from_numpy(m.dense() / case["s"]).to(dev)
    t0 = torch.from_numpy(np.ascontiguousarray(b)).to(dev)
    t1 = a @ t0
    y, p = torch.zeros_like(t0), torch.zeros(len(coeffs), dtype=torch.float64, device=dev)
    for i, c in enumerate(coeffs):
        y = y + float(c) * t1
        p[i] = torch.dot(y, y)
        for _ in range(2):
            t0, t1 = t1, torch.addmv(t0, a, t1, beta=-1.0, alpha=2.0)
    return y.cpu().numpy().astype(np.complex128), p.cpu().numpy()


def exact(case, seed):
    mats, bs = _inputs(case, seed)
    if case["kind"] == "qls":
        y, p = _solve(case, mats[0], bs[0])
        return {"y": y, "p": p}
    walks = [_Walk(m, case["s"]) for m in mats]
    if case["kind"] == "resume":
        x = walks[0].run(bs[0], 2 + case["steps"])
        n, code = walks[0].n, walks[0].code
        b1, b2 = np.arange(2)[None, :, None], np.arange(2)[None, None, :]
        order = ((code // n)[:, None, None] * 2 + b1) * (2 * n) + (code % n)[:, None, None] * 2 + b2
        amps = x.ravel()[np.argsort(order.ravel(), kind="stable")]
        return {"keys": None, "amps": amps[np.abs(amps) > 1e-13]}
    xs = [w.run(b, case["steps"]) for w, b in zip(walks, bs)]
    out = {"j": np.concatenate([w.marginal(x, "j") for w, x in zip(walks, xs)])}
    if case["kind"] != "batch":
        out["k"] = walks[0].marginal(xs[0], "k")
    return out
