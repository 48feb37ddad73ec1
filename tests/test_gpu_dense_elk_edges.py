"""Dense ELK's covariance kernels (a group of lanes per chunk, every d x d product spread over
it) at their edges, float64 against the oracle's sequential filter (1e-10, two damped steps):
every state size, sequences of one row, one chunk, one row past a chunk and many chunks, with
one chain per sequence (few chunks) and in parallel over time (8 or more chunks each), for weak
and strong damping. Float32 against float64 on the same inputs: 1e-4.
"""
import numpy as np
import pytest
import torch

import synth
from oracle import dynamics as odyn
from oracle import elk as oelk
from oracle import newton as onewton

pytestmark = pytest.mark.gpu


def _t(a, dt=torch.float64):
    return torch.tensor(np.ascontiguousarray(a), dtype=dt, device="cuda")


def _relerr(a, b):
    return np.max(np.abs(a - b)) / max(np.max(np.abs(b)), 1e-300)


def _solve(p, d, T, lam, dt, prec):
    import paper_2603_16850_gb300 as deer
    dyn = deer.Dynamics.rnn_tanh(_t(p["W"], dt))
    s, _ = deer.deer_solve(dyn, _t(p["s0"], dt), T, _t(p["x"].reshape(-1, d), dt), jac="full",
                           damp="elk", damp_param=lam, tol=0.0, max_iters=2, init="s0",
                           chunk=8, prec=prec)
    return s.double().cpu().numpy()


@pytest.mark.parametrize("d", [1, 2, 4, 8, 16])
@pytest.mark.parametrize("T,lam", [(1, 0.5), (8, 20.0), (9, 0.05), (64, 0.5), (65, 20.0),
                                   (203, 0.05)])
def test_dense_elk_edges(d, T, lam):
    B = 3
    p = synth.mean_field_rnn(B, T, d, 0.9, seed=d)
    od = odyn.MeanFieldRNN(p["W"], p["x"])
    s = _solve(p, d, T, lam, torch.float64, "fp64")
    ref = onewton.initial_guess(od, p["s0"], T, "s0")
    for _ in range(2):
        ref = oelk.elk_filter_step(od, p["s0"], ref, "full", lam)
    assert _relerr(s, ref.reshape(-1, d)) <= 1e-10
    s32 = _solve(p, d, T, lam, torch.float32, "fp32")
    assert _relerr(s32, s) <= 1e-4
