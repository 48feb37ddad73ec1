"""Timing cases of the solver: what a program that uses it calls, through its public entry
points (``deer_solve``, ``deer_solve_batched``, ``deer_grad``, ``DeerFunction``).

A case is a dict of plain values; its ``family`` says which workload it is (see ``listed``).
``draw`` gives other sizes of the same workloads. Inputs are made from the seed alone, on the
GPU where they are large. ``exact`` is the same answer in float64 by plain torch: a sequential
rollout (the fixed point a converged solve ends at), the reverse recursion of its gradient, and
the filter recursion of the damped steps.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

import paper_2603_16850_gb300 as deer

# largest row count (B * T) a drawn case may have, per family: no drawn case costs more than
# the family's listed one
_MAX_ROWS = {
    "brusselator": 16 * 8192,
    "kinetics": 4096 * 16384,
    "kinetics_fp64": 1 << 21,
    "kinetics_train": 512 * 2047 * 4,
    "kinetics_wide": 256 * 8192,
    "kinetics_grad": 128 * 16384,
    "kinetics_ragged": 64 * 50500,
    "gru": 64 * 65536,
    "gru_elk": 16 * 16384,
    "rnn": 100000,
    "dense_elk": 4 * 4096,
    "langevin": 8 * 10000,
}


def listed():
    return [
        # one short kinetics trajectory in float64 (the smallest call: an interactive or
        # inner-loop solve, latency only)
        {"name": "brusselator_short", "family": "brusselator", "B": 1, "T": 1024},
        # the benchmark's batch of independent reaction networks (parameter sweeps): the
        # largest call, float32 with the compensated state and the sliding window
        {"name": "kinetics_d8_batch", "family": "kinetics", "B": 4096, "T": 16384, "d": 8,
         "R": 12},
        # a small sweep of odd size in float64, to full accuracy
        {"name": "kinetics_d8_fp64_odd", "family": "kinetics_fp64", "B": 37, "T": 1501, "d": 8,
         "R": 12},
        # one step of fitting rate constants and initial states: differentiable solve,
        # loss cotangent, gradients (forward and backward)
        {"name": "kinetics_d8_train", "family": "kinetics_train", "B": 512, "T": 2047, "d": 8,
         "R": 12},
        # larger networks (d = 32): the forward solve of the differentiation workload
        {"name": "kinetics_d32_solve", "family": "kinetics_wide", "B": 256, "T": 8192, "d": 32,
         "R": 48},
        # the adjoint alone at a converged d = 32 trajectory
        {"name": "kinetics_d32_grad", "family": "kinetics_grad", "B": 128, "T": 16384, "d": 32,
         "R": 48},
        # ragged batch, lengths 1000 to 100000, mixed precision (bf16 Jacobian, float64 state)
        {"name": "kinetics_d16_ragged_mixed", "family": "kinetics_ragged", "B": 64, "lo": 1000,
         "hi": 100000, "d": 16, "R": 24},
        # gated recurrent units over long sequences, diagonal Jacobian (quasi-DEER)
        {"name": "gru_d64_quasi_deer", "family": "gru", "B": 64, "T": 65536, "d": 64},
        # the same cell with Kalman damping (quasi-ELK)
        {"name": "gru_d64_quasi_elk", "family": "gru_elk", "B": 16, "T": 16384, "d": 64,
         "lam": 1.0},
        # one long trajectory of a predictable mean-field network: the case parallel-in-time
        # evaluation is for
        {"name": "rnn_d32_long", "family": "rnn", "B": 1, "T": 100000, "d": 32, "g": 0.5},
        # full-Jacobian Newton with Kalman damping (ELK), float64: a fixed number of steps,
        # as the repository's benchmark runs it
        {"name": "kinetics_d8_dense_elk", "family": "dense_elk", "B": 4, "T": 4096, "d": 8,
         "R": 12, "lam": 0.5, "iters": 8},
        # Langevin sampling in a two-well potential, float64, random initial guess
        {"name": "langevin_d4_two_well", "family": "langevin", "B": 4, "T": 10000, "d": 4},
    ]


def _log_int(rng, lo, hi):
    return int(min(hi, max(lo, round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    """Another case: the workload at random, its sizes over the range it is used at."""
    f = rng.choice(sorted(_MAX_ROWS))
    most = _MAX_ROWS[f]

    def sizes(b_lo, b_hi, t_lo, t_hi):
        B, T = _log_int(rng, b_lo, b_hi), _log_int(rng, t_lo, t_hi)
        return B, max(t_lo, min(T, most // B))

    if f == "brusselator":
        B, T = sizes(1, 64, 64, 8192)
        return {"family": f, "B": B, "T": T}
    if f in ("kinetics", "kinetics_fp64", "kinetics_train"):
        b_hi, t_hi = {"kinetics": (4096, 16384), "kinetics_fp64": (512, 8192),
                      "kinetics_train": (1024, 8192)}[f]
        B, T = sizes(1, b_hi, 500, t_hi)
        d = rng.choice([4, 8, 8, 8])
        return {"family": f, "B": B, "T": T, "d": d, "R": rng.randint(d + 2, 2 * d)}
    if f in ("kinetics_wide", "kinetics_grad"):
        B, T = sizes(1, 256, 500, 32768)
        d = rng.choice([16, 32, 32])
        return {"family": f, "B": B, "T": T, "d": d, "R": rng.randint(d + d // 4, 2 * d)}
    if f == "kinetics_ragged":
        lo = _log_int(rng, 100, 2000)
        hi = _log_int(rng, 5000, 100000)
        B = max(1, min(_log_int(rng, 8, 256), 2 * most // (lo + hi)))
        return {"family": f, "B": B, "lo": lo, "hi": hi, "d": 16, "R": rng.randint(20, 32)}
    if f == "gru":
        B, T = sizes(1, 256, 500, 65536)
        return {"family": f, "B": B, "T": T, "d": rng.choice([16, 32, 64, 64, 64])}
    if f == "gru_elk":
        B, T = sizes(1, 64, 500, 16384)
        return {"family": f, "B": B, "T": T, "d": rng.choice([16, 32, 64, 64, 64]),
                "lam": rng.choice([0.01, 0.1, 1.0])}
    if f == "rnn":
        B, T = sizes(1, 8, 2000, 100000)
        return {"family": f, "B": B, "T": T, "d": rng.choice([16, 32, 32]),
                "g": rng.choice([0.4, 0.5, 0.6])}
    if f == "dense_elk":
        B, T = sizes(1, 16, 500, 8192)
        return {"family": f, "B": B, "T": T, "d": rng.choice([4, 8, 8]), "R": 12, "lam": 0.5,
                "iters": rng.randint(3, 8)}
    B, T = sizes(1, 32, 500, 20000)
    return {"family": "langevin", "B": B, "T": T, "d": rng.choice([2, 4, 4, 8])}


# --- inputs ------------------------------------------------------------------------------

_DT = 1e-3    # step of the reaction networks
_DT_B = 0.01  # step of the Brusselator
_EPS = 0.01   # step of the Langevin sampler
_PRECISION = {"kinetics": "fp32", "kinetics_train": "fp32", "kinetics_wide": "fp32",
              "kinetics_grad": "fp32", "gru": "fp32", "gru_elk": "fp32", "rnn": "fp32"}


def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _real(family):
    return torch.float32 if _PRECISION.get(family) == "fp32" else torch.float64


def _network(r, d, R):
    """One mass-conserving reaction network: species of mass 1 or 2, conversions between
    equals, associations of two light species into a heavy one and the reverse; every
    species takes part. Rows (i1, i2, p1, p2), -1 where absent."""
    while True:
        mass = [r.randint(1, 2) for _ in range(d)]
        light = [i for i in range(d) if mass[i] == 1]
        heavy = [i for i in range(d) if mass[i] == 2]
        if not light or not heavy:
            continue
        classes = [c for c in (light, heavy) if len(c) >= 2]
        rows = []
        for _ in range(R):
            kind = r.randint(0, 2) if classes else r.randint(1, 2)
            if kind == 0:
                x, y = r.sample(r.choice(classes), 2)
                rows.append((x, -1, y, -1))
            else:
                x, y, z = r.choice(light), r.choice(light), r.choice(heavy)
                rows.append((x, y, z, -1) if kind == 1 else (z, -1, x, y))
        if len({i for row in rows for i in row if i >= 0}) == d:
            return rows


def _kinetics_inputs(case, seed, dtype, B):
    """B systems: their own network each (of up to 64 drawn ones), log-uniform rate
    constants, s0 uniform on [0, 1]."""
    r = random.Random(seed)
    rng = np.random.default_rng(seed)
    d, R = case["d"], case["R"]
    pool = np.array([_network(r, d, R) for _ in range(min(B, 64))], dtype=np.int32)
    topo = pool[rng.integers(0, len(pool), B)] if B > len(pool) else pool
    k = np.exp(rng.uniform(math.log(1e-2), math.log(1e1), (B, R)))
    s0 = rng.uniform(0.0, 1.0, (B, d))
    dev = _device()
    return (torch.tensor(topo, device=dev).contiguous(), torch.tensor(k, dtype=dtype, device=dev),
            torch.tensor(s0, dtype=dtype, device=dev), rng)


def _lengths(case, seed):
    """Ragged lengths, stretched evenly over [lo, hi] and shuffled: every seed has the same
    number of rows."""
    B = case["B"]
    n = np.linspace(case["lo"], case["hi"], B).round().astype(np.int64)
    return np.random.default_rng(seed + 1).permutation(n)


def _gru_inputs(case, seed):
    d, dev = case["d"], _device()
    g = torch.Generator(device=dev).manual_seed(seed)

    def randn(*shape):
        return torch.randn(*shape, generator=g, device=dev, dtype=torch.float32)

    W, U = randn(3, d, d) * d ** -0.5, randn(3, d, d) * d ** -0.5
    x = randn(case["B"] * case["T"], d)
    return W, U, x, torch.zeros(case["B"], d, dtype=torch.float32, device=dev)


def _rnn_inputs(case, seed):
    B, T, d, dev = case["B"], case["T"], case["d"], _device()
    rng = np.random.default_rng(seed)
    W = rng.standard_normal((d, d)) * (case["g"] / math.sqrt(d))
    np.fill_diagonal(W, 0.0)
    phase = rng.uniform(0.0, 2.0 * np.pi, (B, 1, d))
    t = np.arange(1, T + 1, dtype=np.float64).reshape(1, T, 1)
    x = 0.1 * np.sin(2.0 * np.pi * t / 50.0 + phase)
    s0 = rng.standard_normal((B, d))

    def f(a):
        return torch.tensor(a, dtype=torch.float32, device=dev)

    return f(W), f(x.reshape(-1, d)), f(s0)


def _langevin_inputs(case, seed):
    """Two Gaussians at -1.4 and +1.6 on coordinate 1, variance 0.5 there and 1 elsewhere."""
    B, T, d, dev = case["B"], case["T"], case["d"], _device()
    m1, m2, v = np.zeros(d), np.zeros(d), np.ones(d)
    m1[1], m2[1], v[1] = -1.4, 1.6, 0.5
    p = torch.tensor(np.concatenate([m1, m2, v, v, [0.5, 0.5]]), device=dev)
    g = torch.Generator(device=dev).manual_seed(seed)
    x = torch.randn(B * T, d, generator=g, device=dev, dtype=torch.float64)
    s0 = torch.randn(B, d, generator=g, device=dev, dtype=torch.float64)
    return p, x, s0


def _brusselator_inputs(case, seed):
    rng = np.random.default_rng(seed)
    B = case["B"]
    ab = np.stack([rng.uniform(0.9, 1.1, B), rng.uniform(2.8, 3.2, B)], axis=1)
    s0 = rng.uniform(0.9, 1.1, (B, 2))
    return torch.tensor(ab, device=_device()), torch.tensor(s0, device=_device())


# Convergence as the repository's benchmark and tests ask for it, per workload; the cap on
# iterations is far above what converging inputs need.
_OPTIONS = {
    "brusselator": dict(jac="full", tol=1e-12, prec="fp64", init="s0", reset=True),
    "kinetics": dict(jac="full", tol=5e-8, confirm=2, prec="fp32", init="s0", reset=True,
                     window=True),
    "kinetics_fp64": dict(jac="full", tol=1e-12, confirm=2, prec="fp64", init="s0", reset=True,
                          window=True),
    "kinetics_train": dict(jac="full", tol=5e-8, confirm=2, prec="fp32", init="s0", reset=True),
    "kinetics_wide": dict(jac="full", tol=5e-8, confirm=2, prec="fp32", init="zeros",
                          reset=True),
    "kinetics_ragged": dict(jac="full", tol=1e-12, prec="mixed_bf16", init="zeros", reset=True,
                            window=True),
    "gru": dict(jac="diag", tol=1e-5, confirm=2, prec="fp32", init="zeros"),
    "gru_elk": dict(jac="diag", damp="elk", tol=1e-5, confirm=2, prec="fp32", init="zeros"),
    "rnn": dict(jac="full", tol=1e-5, prec="fp32", init="zeros", reset=True, window=True),
    "dense_elk": dict(jac="full", damp="elk", tol=0.0, prec="fp64", init="s0", reset=True),
    "langevin": dict(jac="full", tol=1e-11, prec="fp64", init="randn", reset=True),
}
_MAX_ITERS = 600


def prepare(case, seed):
    f = case["family"]
    st = {"case": case, "opts": dict(_OPTIONS.get(f, {}), max_iters=_MAX_ITERS)}
    if f == "brusselator":
        ab, s0 = _brusselator_inputs(case, seed)
        return dict(st, dyn=deer.Dynamics.brusselator(ab, _DT_B), s0=s0, x=None)
    if f in ("gru", "gru_elk"):
        W, U, x, s0 = _gru_inputs(case, seed)
        if f == "gru_elk":
            st["opts"]["damp_param"] = case["lam"]
        return dict(st, dyn=deer.Dynamics.gru(W, U), s0=s0, x=x)
    if f == "rnn":
        W, x, s0 = _rnn_inputs(case, seed)
        return dict(st, dyn=deer.Dynamics.rnn_tanh(W), s0=s0, x=x)
    if f == "langevin":
        p, x, s0 = _langevin_inputs(case, seed)
        st["opts"]["seed"] = seed
        return dict(st, dyn=deer.Dynamics.langevin_2well(p, _EPS), s0=s0, x=x)
    B = case["B"]
    topo, k, s0, rng = _kinetics_inputs(case, seed, _real(f), B)
    dyn = deer.Dynamics.massaction(topo, k, case["d"], _DT)
    st = dict(st, dyn=dyn, s0=s0, x=None)
    if f == "dense_elk":
        st["opts"].update(damp_param=case["lam"], max_iters=case["iters"])
    elif f == "kinetics_ragged":
        st["offsets"] = np.concatenate([[0], np.cumsum(_lengths(case, seed))])
    elif f == "kinetics_train":
        st["target"] = _targets(case, s0, seed)
    elif f == "kinetics_grad":
        # the converged trajectory, and the cotangent of a squared distance to targets
        wide = deer.Dynamics.massaction(topo, k.double(), case["d"], _DT)
        st["s"] = deer.deer_rollout(wide, s0.double(), case["T"]).float()
        st["g"] = 2.0 * (st["s"] - _targets(case, s0, seed))
    return st


def _targets(case, s0, seed):
    """Observations to fit: the initial state with 10 % noise at every step."""
    g = torch.Generator(device=s0.device).manual_seed(seed + 7)
    B, T, d = case["B"], case["T"], case["d"]
    y = torch.randn(B, T, d, generator=g, device=s0.device, dtype=s0.dtype)
    return (s0[:, None, :] * (1.0 + 0.1 * y)).reshape(-1, d)


def run(state):
    case, dyn, s0 = state["case"], state["dyn"], state["s0"]
    f = case["family"]
    if f == "kinetics_grad":
        dk, ds0 = deer.deer_grad(dyn, s0, case["T"], state["s"], state["g"], prec="fp32")
        return {"dk": dk, "ds0": ds0}
    if f == "kinetics_train":
        k = dyn.params.detach().requires_grad_(True)
        s0 = s0.detach().requires_grad_(True)
        s = deer.DeerFunction.apply(k, s0, dyn, case["T"], None, state["opts"])
        dk, ds0 = torch.autograd.grad(s, (k, s0), 2.0 * (s.detach() - state["target"]))
        return {"s": s.detach(), "dk": dk, "ds0": ds0}
    if f == "kinetics_ragged":
        s, _ = deer.deer_solve_batched(dyn, s0, state["offsets"], **state["opts"])
        return s
    s, _ = deer.deer_solve(dyn, s0, case["T"], state["x"], **state["opts"])
    return s


def _rows(case):
    if case["family"] == "kinetics_ragged":
        return int(_lengths(case, 0).sum())
    return case["B"] * case["T"]


def work(case):
    """The state written once, the inputs read once, and one linearisation and one affine
    composition per row: a solve iterates more often than once, how often depends on the
    inputs."""
    f, rows = case["family"], _rows(case)
    d = case.get("d", 2)
    size = 4 if _PRECISION.get(f) == "fp32" else 8
    per_row, values = {
        # value and Jacobian of the step, and (P, v) <- (A P, A v + b)
        "brusselator": (30 + 2 * 8 + 8, d),
        "gru": (6 * d * d + 2 * d * d + 2 * d, 2 * d),
        "gru_elk": (6 * d * d + 2 * d * d + 20 * d, 2 * d),
        "rnn": (2 * d * d + d * d + 2 * d ** 3 + 2 * d * d, 2 * d),
        "langevin": (20 * d + 3 * d * d + 2 * d ** 3 + 2 * d * d, 2 * d),
    }.get(f, (3 * 2 * d ** 3 + 2 * d ** 3 + 2 * d * d + 4 * 6 * case.get("R", 1), d))
    if f == "kinetics_grad":
        # states and cotangents read; the adjoint is a vector: stage products, one
        # matrix-vector product and the rate-constant gradient
        per_row, values = 4 * 12 * case["R"] + 2 * d * d, 2 * d
    if f == "kinetics_train":
        per_row, values = per_row + 4 * 12 * case["R"] + 2 * d * d, 2 * d
    if f == "dense_elk":
        per_row = (per_row + 7 * d ** 3) * case["iters"]
    return {"bytes": float(rows * values * size), "flops": float(rows * per_row)}


# --- the same in float64, by plain torch -------------------------------------------------

def _rollout64(step, s0, T, xs=None, block=64):
    """s_t = step(s_{t-1}, xs[t]) for t = 1..T in order: [T][B][d]. On a GPU the steps run as
    replays of one CUDA graph of `block` steps."""
    out = torch.empty((T,) + tuple(s0.shape), dtype=s0.dtype, device=s0.device)
    if not s0.is_cuda or T < 4 * block:
        s = s0
        for t in range(T):
            s = step(s, None if xs is None else xs[t])
            out[t] = s
        return out
    cur, got = s0.clone(), torch.empty_like(out[:block])
    part = None if xs is None else torch.empty_like(xs[:block])

    def body():
        s = cur
        for i in range(block):
            s = step(s, None if xs is None else part[i])
            got[i].copy_(s)
        cur.copy_(s)

    if xs is not None:
        part.copy_(xs[:block])
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        step(cur, None if xs is None else part[0])
    torch.cuda.current_stream().wait_stream(side)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        body()
    done = T // block * block
    for t in range(0, done, block):
        if xs is not None:
            part.copy_(xs[t:t + block])
        graph.replay()
        out[t:t + block].copy_(got)
    s = cur
    for t in range(done, T):
        s = step(s, None if xs is None else xs[t])
        out[t] = s
    return out


class _Kinetics64:
    """RK4 steps of mass-action networks: dc/dt = S (k * phi(c))."""

    def __init__(self, topo, k, d):
        t = topo.long()
        B, R, _ = t.shape
        S = torch.zeros(B, R, d + 1, dtype=torch.float64, device=t.device)
        one = torch.ones(B, R, dtype=torch.float64, device=t.device)
        for col, sign in ((0, -1.0), (1, -1.0), (2, 1.0), (3, 1.0)):
            i = torch.where(t[:, :, col] >= 0, t[:, :, col], d)
            S.scatter_add_(2, i[:, :, None], sign * one[:, :, None])
        self.S = S[:, :, :d].transpose(1, 2).contiguous()  # [B][d][R]
        self.i1 = t[:, :, 0]
        self.i2 = torch.where(t[:, :, 1] >= 0, t[:, :, 1], d)
        self.k, self.d = k.double(), d

    def _both(self, c):
        c1 = torch.nn.functional.pad(c, (0, 1), value=1.0)
        return c1.gather(1, self.i1), c1.gather(1, self.i2)

    def rhs(self, c):
        a, b = self._both(c)
        return (self.S * (self.k * a * b)[:, None, :]).sum(2)

    def step(self, c, _=None):
        h = _DT
        k1 = self.rhs(c)
        k2 = self.rhs(c + 0.5 * h * k1)
        k3 = self.rhs(c + 0.5 * h * k2)
        k4 = self.rhs(c + h * k3)
        return c + (h / 6.0) * (k1 + 2.0 * k2 + 2.0 * k3 + k4)

    def many(self, n):
        """The same systems, each for n rows in a row ([B * n] rows)."""
        m = object.__new__(_Kinetics64)
        m.S, m.i1, m.i2, m.k = (v.repeat_interleave(n, 0)
                                for v in (self.S, self.i1, self.i2, self.k))
        m.d = self.d
        return m

    def linearise(self, c):
        """The step of every row and its Jacobian (d vector-Jacobian products over all rows
        at once); the step keeps its graph."""
        c = c.detach().requires_grad_(True)
        eye = torch.eye(self.d, dtype=torch.float64, device=c.device)
        with torch.enable_grad():
            y = self.step(c)
        A = [torch.autograd.grad(y, c, e.expand_as(c), retain_graph=True)[0] for e in eye]
        return y, torch.stack(A, 1)

    def elk(self, s0, T, lam, iters):
        """`iters` Newton steps from the constant guess s0, each the mean of a Kalman filter:
        process noise I, the previous iterate observed with variance 1 / lam, s0 known."""
        B, d = s0.shape
        eye = torch.eye(d, dtype=torch.float64, device=s0.device)
        many, s = self.many(T), s0[:, None].repeat(1, T, 1)
        for _ in range(iters):
            prev = torch.cat([s0[:, None], s[:, :-1]], 1)
            y, A = many.linearise(prev.reshape(B * T, d))
            y, A = y.detach().reshape(B, T, d), A.reshape(B, T, d, d)
            P, dx, new = torch.zeros(B, d, d, dtype=s.dtype, device=s.device), None, s.clone()
            for t in range(T):
                Pm = A[:, t] @ P @ A[:, t].transpose(1, 2) + eye
                G = torch.linalg.inv_ex(eye + lam * Pm)[0]
                P = G @ Pm
                # the mean's difference from the previous iterate
                v = y[:, t] - s[:, t]
                if dx is not None:
                    v = v + (A[:, t] @ dx[:, :, None])[:, :, 0]
                dx = (G @ v[:, :, None])[:, :, 0]
                new[:, t] += dx
            s = new
        return s.reshape(B * T, d)

    def grad(self, s0, s, g):
        """dl/dk [B][R] and dl/ds0 [B][d] of a loss with cotangents g [T][B][d] along the
        trajectory s [T][B][d]: lambda_t = g_t + A_{t+1}^T lambda_{t+1}, from the end, one
        vector-Jacobian product of the step per row."""
        T, B, d = s.shape
        prev = torch.cat([s0[None], s[:-1]])
        lam = torch.zeros(B, d, dtype=torch.float64, device=s.device)
        dk = torch.zeros_like(self.k)
        n = max(1, min(T, (1 << 24) // (B * d * d)))
        many, at = None, 0
        for hi in range(T, 0, -n):
            lo = max(0, hi - n)
            m = hi - lo
            if at != m:
                many, at = self.many(m), m
            many.k = many.k.detach().requires_grad_(True)
            y, A = many.linearise(prev[lo:hi].transpose(0, 1).reshape(B * m, d))
            A = A.reshape(B, m, d, d)
            lams = torch.empty(B, m, d, dtype=torch.float64, device=s.device)
            for j in range(m - 1, -1, -1):
                lam = lam + g[lo + j]
                lams[:, j] = lam
                lam = torch.bmm(lam[:, None, :], A[:, j])[:, 0]
            gk, = torch.autograd.grad(y, many.k, lams.reshape(B * m, d))
            dk += gk.reshape(B, m, -1).sum(1)
        return dk, lam


def _flat(s):
    """[T][B][d] -> packed rows [B * T][d]."""
    return s.transpose(0, 1).reshape(-1, s.shape[2])


def exact(case, seed):
    f = case["family"]
    B, T = case["B"], case.get("T", 0)
    if f == "brusselator":
        ab, s0 = _brusselator_inputs(case, seed)
        a, b = ab[:, 0], ab[:, 1]

        def step(s, _):
            x, y = s[:, 0], s[:, 1]
            xxy = x * x * y
            return s + _DT_B * torch.stack([a - (b + 1.0) * x + xxy, b * x - xxy], 1)

        return _flat(_rollout64(step, s0, T))
    if f in ("gru", "gru_elk"):
        d = case["d"]
        W, U, x, s0 = (v.double() for v in _gru_inputs(case, seed))
        xs = (x @ W.reshape(3 * d, d).T).reshape(B, T, 3 * d).transpose(0, 1).contiguous()
        Uzr, Uh = U[:2].reshape(2 * d, d).T.contiguous(), U[2].T.contiguous()

        def step(h, p):
            zr = torch.sigmoid(p[:, :2 * d] + h @ Uzr)
            n = torch.tanh(p[:, 2 * d:] + (zr[:, d:] * h) @ Uh)
            return torch.lerp(h, n, zr[:, :d])

        return _flat(_rollout64(step, s0, T, xs))
    if f == "rnn":
        W, x, s0 = (v.double() for v in _rnn_inputs(case, seed))
        xs, Wt = x.reshape(B, T, -1).transpose(0, 1).contiguous(), W.T.contiguous()
        return _flat(_rollout64(lambda s, u: torch.tanh(s) @ Wt + u, s0, T, xs))
    if f == "langevin":
        p, x, s0 = _langevin_inputs(case, seed)
        d = case["d"]
        m1, m2, v1, v2 = (p[i * d:(i + 1) * d] for i in range(4))
        xs = (math.sqrt(2.0 * _EPS) * x).reshape(B, T, d).transpose(0, 1).contiguous()
        base = 0.5 * (torch.log(v2) - torch.log(v1)).sum() + torch.log(p[4 * d] / p[4 * d + 1])

        def step(s, u):
            q1, q2 = (s - m1) / v1, (s - m2) / v2
            odds = base + 0.5 * ((s - m2) * q2 - (s - m1) * q1).sum(1, keepdim=True)
            r1, r2 = torch.sigmoid(odds), torch.sigmoid(-odds)
            return s - _EPS * (r1 * q1 + r2 * q2) + u

        return _flat(_rollout64(step, s0, T, xs))
    topo, k, s0, _ = _kinetics_inputs(case, seed, _real(f), B)
    sys64 = _Kinetics64(topo, k, case["d"])
    c0 = s0.double()
    if f == "dense_elk":
        return sys64.elk(c0, T, case["lam"], case["iters"])
    if f == "kinetics_ragged":
        n = _lengths(case, seed)
        s = _rollout64(sys64.step, c0, int(n.max()))
        return torch.cat([s[:int(n[b]), b] for b in range(B)])
    s = _rollout64(sys64.step, c0, T)
    if f not in ("kinetics_grad", "kinetics_train"):
        return _flat(s)
    if f == "kinetics_grad":
        s = s.float().double()
    d = case["d"]
    y = _targets(case, s0, seed).reshape(B, T, d).transpose(0, 1).double()
    if f == "kinetics_grad":
        # the cotangent is formed in float32 there
        g = (2.0 * (s.float() - y.float())).double()
    else:
        g = 2.0 * (s - y)
    dk, ds0 = sys64.grad(c0, s, g)
    if f == "kinetics_grad":
        return {"dk": dk, "ds0": ds0}
    return {"s": _flat(s), "dk": dk, "ds0": ds0}
