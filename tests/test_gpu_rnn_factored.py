"""The mean-field RNN's scan from the column factors of its Jacobians (d = 32, float32) at the
edges of its chunks and staged rows, with a weight matrix per sequence, scale damping and the
sliding window: two Newton iterations against the dense path (tensor cores off) to 1e-5, a
hundred float32 roundings of values of order one, and the converged trajectory against the
float64 rollout to 1e-5.
"""
import numpy as np
import pytest
import torch

import synth
from oracle import dynamics as odyn
from oracle import newton as onewton

pytestmark = pytest.mark.gpu


def _t(a, dt=torch.float32):
    return torch.tensor(np.ascontiguousarray(a), dtype=dt, device="cuda")


def _relerr(a, b):
    return np.max(np.abs(a - b)) / max(np.max(np.abs(b)), 1e-300)


@pytest.mark.parametrize("damp", [{}, {"damp": "scale", "damp_param": 0.3}])
@pytest.mark.parametrize("lengths", [[1], [7, 8, 9, 0, 31, 32, 33, 1], [300, 299]])
def test_factored_iterates(lengths, damp):
    import paper_2603_16850_gb300 as deer
    d, B, T = 32, len(lengths), max(lengths)
    p = synth.mean_field_rnn(B, T, d, 0.7, seed=1)
    W = np.stack([synth.mean_field_rnn(1, 1, d, 0.7, seed=10 + b)["W"] for b in range(B)])
    x = _t(np.concatenate([p["x"][b, :lengths[b]] for b in range(B)]))
    off = np.concatenate([[0], np.cumsum(lengths)])
    dyn = deer.Dynamics.rnn_tanh(_t(W if B > 1 else W[0]))
    o = dict(jac="full", tol=0.0, max_iters=2, init="s0", prec="fp32", chunk=8, **damp)
    try:
        a, _ = deer.deer_solve_batched(dyn, _t(p["s0"]), off, x, **o)
        deer.set_tensor_cores(False)
        b, _ = deer.deer_solve_batched(dyn, _t(p["s0"]), off, x, **o)
    finally:
        deer.set_tensor_cores(True)
    assert _relerr(a.double().cpu().numpy(), b.double().cpu().numpy()) <= 1e-5


@pytest.mark.parametrize("window", [False, True])
def test_factored_fixed_point(window):
    import paper_2603_16850_gb300 as deer
    B, T, d = 2, 1500, 32
    p = synth.mean_field_rnn(B, T, d, 0.6, seed=2)
    dyn = deer.Dynamics.rnn_tanh(_t(p["W"]))
    s, info = deer.deer_solve(dyn, _t(p["s0"]), T, _t(p["x"].reshape(-1, d)), jac="full",
                              tol=5e-7, confirm=2, prec="fp32", init="zeros", reset=True,
                              window=window)
    ref = onewton.rollout(odyn.MeanFieldRNN(p["W"], p["x"]), p["s0"], T)
    assert bool(info.converged.all())
    assert _relerr(s.double().cpu().numpy().reshape(B, T, d), ref) <= 1e-5
