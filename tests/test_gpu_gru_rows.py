"""Row handling of the GRU kernels (d = 64, float32) and of the quasi-ELK passes at their edges:
ragged batches whose sequences end inside, at and past a 128-row tile, with a non-zero initial
state, on the tcgen05 linearisation against the SIMT one (two iterates, 2e-6: the float32
rounding of the two forms, as for the uniform batches); inputs that start off a 16-byte
boundary (bit for bit); and, in float64, the batches of rows and chunks the quasi-ELK passes
load ahead, for strong and weak damping, against the oracle's filter (1e-10).
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


def _gru64(lengths, seed):
    import paper_2603_16850_gb300 as deer
    f = torch.float32
    g = synth.gru(1, int(sum(lengths)), 64, 64, seed=seed)
    dyn = deer.Dynamics.gru(_t(g["W"], f), _t(g["U"], f))
    s0 = _t(np.random.default_rng(seed).uniform(-0.9, 0.9, (len(lengths), 64)), f)
    return dyn, s0, _t(g["x"][0], f), np.concatenate([[0], np.cumsum(lengths)])


@pytest.mark.parametrize("jac", ["diag", "identity"])
@pytest.mark.parametrize("lengths", [[1], [1, 127, 0, 128, 129, 300, 2], [128] * 3])
def test_gru_tiles_of_ragged_rows(lengths, jac):
    import paper_2603_16850_gb300 as deer
    dyn, s0, x, off = _gru64(lengths, seed=8)
    o = dict(jac=jac, tol=0.0, max_iters=2, init="s0", prec="fp32")
    try:
        tc, _ = deer.deer_solve_batched(dyn, s0, off, x, **o)
        deer.set_tensor_cores(False)
        simt, _ = deer.deer_solve_batched(dyn, s0, off, x, **o)
    finally:
        deer.set_tensor_cores(True)
    assert _relerr(tc.double().cpu().numpy(), simt.double().cpu().numpy()) <= 2e-6


def test_gru_inputs_off_a_16_byte_boundary():
    import paper_2603_16850_gb300 as deer
    dyn, s0, x, off = _gru64([200, 57], seed=9)
    buf = torch.empty(x.numel() + 1, dtype=x.dtype, device="cuda")
    shifted = buf[1:].view_as(x)
    shifted.copy_(x)
    assert shifted.data_ptr() % 16 == 4
    o = dict(jac="diag", tol=0.0, max_iters=3, init="zeros", prec="fp32")
    a, _ = deer.deer_solve_batched(dyn, s0, off, x, **o)
    b, _ = deer.deer_solve_batched(dyn, s0, off, shifted, **o)
    assert torch.equal(a, b)


@pytest.mark.parametrize("lam", [0.01, 1000.0])
@pytest.mark.parametrize("T", [1, 7, 8, 9, 127, 129, 17 * 128 + 3])
def test_quasi_elk_rows_and_chunks(lam, T):
    import paper_2603_16850_gb300 as deer
    B, d = 2, 8
    g = synth.gru(B, T, d, d, seed=3)
    od = odyn.GRU(g["W"], g["U"], g["x"])
    dyn = deer.Dynamics.gru(_t(g["W"]), _t(g["U"]))
    s, _ = deer.deer_solve(dyn, _t(g["s0"]), T, _t(g["x"].reshape(-1, d)), jac="diag",
                           damp="elk", damp_param=lam, tol=0.0, max_iters=2, init="zeros")
    ref = onewton.initial_guess(od, g["s0"], T, "zeros")
    for _ in range(2):
        ref = oelk.elk_filter_step(od, g["s0"], ref, "diag", lam)
    assert _relerr(s.cpu().numpy(), ref.reshape(-1, d)) <= 1e-10
