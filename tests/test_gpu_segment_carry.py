"""The two-level carry of the dense scans (few sequences of 128 or more chunks: chunks folded
into segments, segments walked, then the chunks of each segment): ragged batches whose
sequences end inside, at and just past a segment, beside short and empty ones. One Newton
step in float64 equals the oracle's forward substitution to 1e-10 for every state size;
windowed solves (the first chunk moves) and the mixed-precision path reach the rollout within
the tolerances of their precision (1e-5, 1e-9).
"""
import numpy as np
import pytest
import torch

import synth
from oracle import dynamics as odyn
from oracle import newton as onewton

pytestmark = pytest.mark.gpu


def _t(a, dt=torch.float64):
    return torch.tensor(np.ascontiguousarray(a), dtype=dt, device="cuda")


def _relerr(a, b):
    return np.max(np.abs(a - b)) / max(np.max(np.abs(b)), 1e-300)


@pytest.mark.parametrize("d", [2, 4, 5, 8, 16, 32])
def test_segment_carry_newton_step(d):
    import paper_2603_16850_gb300 as deer
    lengths = [1024, 7, 0, 1025, 1088, 1500]  # chunks of 8: 128, 1, 0, 129, 136, 188
    B, T = len(lengths), max(lengths)
    off = np.concatenate([[0], np.cumsum(lengths)])
    if d == 5:
        p = synth.word_problem(B, T, seed=4, d=d)
        dyn = deer.Dynamics.permute(d, torch.float64, "cuda")
    else:
        p = synth.mean_field_rnn(B, T, d, 0.9, seed=4)
        dyn = deer.Dynamics.rnn_tanh(_t(p["W"]))
    x = _t(np.concatenate([p["x"][b, :lengths[b]] for b in range(B)]))
    s, _ = deer.deer_solve_batched(dyn, _t(p["s0"]), off, x, jac="full", tol=0.0, max_iters=1,
                                   init="s0", chunk=8, block_solve=False)
    s = s.cpu().numpy()
    for b in range(B):
        if lengths[b] == 0:
            continue
        xb, s0 = p["x"][b:b + 1], p["s0"][b:b + 1]
        od = odyn.Permute(xb) if d == 5 else odyn.MeanFieldRNN(p["W"], xb)
        ref = onewton.initial_guess(od, s0, lengths[b], init="s0")
        ref = onewton.quasi_newton_step(od, s0, ref, "full")
        assert _relerr(s[off[b]:off[b + 1]], ref[0]) <= 1e-10, b


@pytest.mark.parametrize("d", [16, 32])
def test_segment_carry_windowed_fp32(d):
    import paper_2603_16850_gb300 as deer
    B, T = 3, 3000
    p = synth.mean_field_rnn(B, T, d, 0.6, seed=5)
    f = torch.float32
    dyn = deer.Dynamics.rnn_tanh(_t(p["W"], f))
    s, info = deer.deer_solve(dyn, _t(p["s0"], f), T, _t(p["x"].reshape(-1, d), f), jac="full",
                              tol=5e-7, confirm=2, prec="fp32", init="zeros", reset=True,
                              window=True, chunk=8)
    ref = onewton.rollout(odyn.MeanFieldRNN(p["W"], p["x"]), p["s0"], T)
    assert bool(info.converged.all())
    assert _relerr(s.cpu().double().numpy().reshape(B, T, d), ref) <= 1e-5


@pytest.mark.parametrize("rc", [False, True])
def test_segment_carry_mixed(rc):
    import paper_2603_16850_gb300 as deer
    lengths = [2100, 40, 1100]
    B, d = len(lengths), 16
    off = np.concatenate([[0], np.cumsum(lengths)])
    p = synth.massaction(B, d, 24, 1, seed=6)
    dyn = deer.Dynamics.massaction(_t(p["topology"], torch.int32), _t(p["params"]), d, p["dt"])
    s, info = deer.deer_solve_batched(dyn, _t(p["s0"]), off, jac="full", tol=1e-12,
                                      prec="mixed_bf16", init="zeros", reset=True, window=True,
                                      chunk=16, max_iters=400,
                                      jac_bytes_max=1024 if rc else 0)
    assert bool(info.converged.all())
    s = s.cpu().numpy()
    for b in range(B):
        od = odyn.MassAction(p["topology"][b:b + 1], p["params"][b:b + 1], p["dt"], "rk4", d=d)
        ref = onewton.rollout(od, p["s0"][b:b + 1], lengths[b])[0]
        assert _relerr(s[off[b]:off[b + 1]], ref) <= 1e-9
