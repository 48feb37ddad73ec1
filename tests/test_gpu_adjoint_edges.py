"""The adjoint's scan kernels at the edges of their chunks and rings (float64 against the
oracle's reverse recursion, 1e-10): sequences of one row, one short of, equal to and one past
the staged rows and the chunk, every state size the kernels are built for, and networks dense
enough that a species takes part in more reactions than the packed lists of the
rate-constant gradient hold. The float32 d = 32 chunk pass (register tiles) against the
float64 gradient of the same inputs: 2e-4 normwise, about 64 rows x 48 terms of float32
rounding, ten times what the sizes here leave.
"""
import numpy as np
import pytest
import torch

import synth
from oracle import adjoint as oadj
from oracle import dynamics as odyn
from oracle import newton as onewton

pytestmark = pytest.mark.gpu


def _t(a, dt=torch.float64):
    return torch.tensor(np.ascontiguousarray(a), dtype=dt, device="cuda")


def _relerr(a, b):
    return np.max(np.abs(a - b)) / max(np.max(np.abs(b)), 1e-300)


def _kinetics(B, d, R, T, seed):
    p = synth.massaction(B, d, R, T, seed, dt=1e-2)
    od = odyn.MassAction(p["topology"], p["params"], p["dt"], "rk4", d=d)
    s = onewton.rollout(od, p["s0"], T)
    g = synth.targets_noise(s.shape, seed=seed + 1)
    dk, ds0, _ = oadj.adjoint_grad(od, p["s0"], s, g)
    return p, s, g, dk, ds0


@pytest.mark.parametrize("d,R", [(2, 3), (4, 16), (8, 40), (16, 20), (16, 64), (32, 100)])
@pytest.mark.parametrize("T", [1, 4, 9, 65])
def test_kinetics_gradient_edges_fp64(d, R, T):
    import paper_2603_16850_gb300 as deer
    B = 3
    p, s, g, dk, ds0 = _kinetics(B, d, R, T, seed=d + T)
    dyn = deer.Dynamics.massaction(_t(p["topology"], torch.int32), _t(p["params"]), d, p["dt"])
    gk, gs0 = deer.deer_grad(dyn, _t(p["s0"]), T, _t(s.reshape(-1, d)), _t(g.reshape(-1, d)),
                             chunk=16)
    assert _relerr(gk.cpu().numpy(), dk) <= 1e-10
    assert _relerr(gs0.cpu().numpy(), ds0) <= 1e-10


@pytest.mark.parametrize("d", [1, 2, 4, 5, 8, 16, 32])
@pytest.mark.parametrize("T", [1, 15, 16, 17, 50])
def test_state_gradient_edges_fp64(d, T):
    import paper_2603_16850_gb300 as deer
    B = 5
    if d == 5:
        p = synth.word_problem(B, T, seed=2, d=d)
        od, dyn = odyn.Permute(p["x"]), deer.Dynamics.permute(d, torch.float64, "cuda")
    else:
        p = synth.mean_field_rnn(B, T, d, 0.8, seed=2)
        od, dyn = odyn.MeanFieldRNN(p["W"], p["x"]), deer.Dynamics.rnn_tanh(_t(p["W"]))
    s = onewton.rollout(od, p["s0"], T)
    g = synth.targets_noise(s.shape, seed=3)
    _, ds0, _ = oadj.adjoint_grad(od, p["s0"], s, g)
    _, gs0 = deer.deer_grad(dyn, _t(p["s0"]), T, _t(s.reshape(-1, d)), _t(g.reshape(-1, d)),
                            x=_t(p["x"].reshape(-1, d)), chunk=16)
    assert _relerr(gs0.cpu().numpy(), ds0) <= 1e-10


@pytest.mark.parametrize("T", [1, 3, 4, 5, 31, 32, 33, 97])
def test_d32_float32_chunk_tiles(T):
    import paper_2603_16850_gb300 as deer
    B, d, R = 2, 32, 48
    p, s, g, dk, ds0 = _kinetics(B, d, R, T, seed=T)
    f = torch.float32
    dyn = deer.Dynamics.massaction(_t(p["topology"], torch.int32), _t(p["params"], f), d, p["dt"])
    gk, gs0 = deer.deer_grad(dyn, _t(p["s0"], f), T, _t(s.reshape(-1, d), f),
                             _t(g.reshape(-1, d), f), prec="fp32")
    assert _relerr(gk.cpu().double().numpy(), dk) <= 2e-4
    assert _relerr(gs0.cpu().double().numpy(), ds0) <= 2e-4
