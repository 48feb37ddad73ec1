"""The dense scan for d <= 8 (a group of lanes per chunk, rows staged eight ahead in a
shared-memory ring) at the sizes where it can go wrong: sequences shorter than, equal to and
just past the ring and the chunk, empty and one-row sequences in a ragged batch, state sizes
that are not a power of two, fewer and more sequences than a warp holds groups. Two Newton
iterations equal the oracle's forward substitution to 1e-10 in float64 (the Langevin step
evaluates exp and log; the association order of the scan is the only other difference), and
the default chunk length (which shrinks for small batches) gives the iterates of the 64-row
chunks it replaces to 1e-11.
"""
import numpy as np
import pytest
import torch

import synth
from oracle import dynamics as odyn
from oracle import newton as onewton

pytestmark = pytest.mark.gpu

DEV = "cuda"


def _t(a, dt=torch.float64):
    return torch.tensor(np.ascontiguousarray(a), dtype=dt, device=DEV)


def _relerr(got, ref):
    return np.max(np.abs(got - ref)) / max(np.max(np.abs(ref)), 1e-300)


@pytest.mark.parametrize("d", [1, 2, 4, 5, 8])
@pytest.mark.parametrize("lengths", [[1, 0, 7, 8, 9, 15, 16, 17, 33, 0], [3],
                                     [16 * 9 + 1] * 37])
def test_small_dense_scan_edges(d, lengths):
    import paper_2603_16850_gb300 as deer
    B, T = len(lengths), max(lengths)
    off = np.concatenate([[0], np.cumsum(lengths)])
    if d == 5:
        p = synth.word_problem(B, T, seed=3, d=d)
        x = _t(np.concatenate([p["x"][b, :lengths[b]] for b in range(B)]))
        dyn = deer.Dynamics.permute(d, torch.float64, DEV)

        def od(b):
            return odyn.Permute(p["x"][b:b + 1])
    else:
        p = synth.two_well(B, T, d, seed=3)
        x = _t(np.concatenate([p["x"][b, :lengths[b]] for b in range(B)]))
        dyn = deer.Dynamics.langevin_2well(_t(p["params"]), p["dt"])

        def od(b):
            return odyn.TwoWellLangevin(p["params"], p["dt"], p["x"][b:b + 1], d=d)
    s, _ = deer.deer_solve_batched(dyn, _t(p["s0"]), off, x, jac="full", tol=0.0, max_iters=2,
                                   init="s0", chunk=16, block_solve=False)
    s = s.cpu().numpy()
    for b in range(B):
        if lengths[b] == 0:
            continue
        ref = onewton.initial_guess(od(b), p["s0"][b:b + 1], lengths[b], init="s0")
        for _ in range(2):
            ref = onewton.quasi_newton_step(od(b), p["s0"][b:b + 1], ref, "full")
        assert _relerr(s[off[b]:off[b + 1]], ref[0]) <= 1e-10, b


@pytest.mark.parametrize("B,T,d", [(37, 1501, 8), (3, 200, 4), (1, 4097, 8)])
def test_default_chunk_of_small_batches(B, T, d):
    import paper_2603_16850_gb300 as deer
    p = synth.massaction(B, d, d + 4, T, seed=11)
    dyn = deer.Dynamics.massaction(_t(p["topology"], torch.int32), _t(p["params"]), d, p["dt"])
    o = dict(jac="full", tol=0.0, max_iters=3, init="s0", block_solve=False)
    s, _ = deer.deer_solve(dyn, _t(p["s0"]), T, **o)
    s64, _ = deer.deer_solve(dyn, _t(p["s0"]), T, chunk=64, **o)
    assert _relerr(s.cpu().numpy(), s64.cpu().numpy()) <= 1e-11


@pytest.mark.parametrize("d", [4, 5, 8])
def test_entry_and_group_forms_agree(d):
    """Float64: 5000 chunks take a group of lanes per chunk, an eighth of them a warp per
    chunk with its entries spread over the lanes; every sum runs in the same order, so one
    Newton step is the same bit for bit."""
    import paper_2603_16850_gb300 as deer
    B, T = 40, 1000
    if d == 5:
        p = synth.word_problem(B, T, seed=7, d=d)
        dyn = deer.Dynamics.permute(d, torch.float64, DEV)
    else:
        p = synth.mean_field_rnn(B, T, d, 0.9, seed=7)
        dyn = deer.Dynamics.rnn_tanh(_t(p["W"]))
    x, s0 = _t(p["x"]), _t(p["s0"])
    o = dict(jac="full", tol=0.0, max_iters=1, init="s0", chunk=8, block_solve=False)
    whole, _ = deer.deer_solve(dyn, s0, T, x.reshape(-1, d), **o)
    for b in range(0, B, 5):
        part, _ = deer.deer_solve(dyn, s0[b:b + 5].contiguous(), T,
                                  x[b:b + 5].reshape(-1, d).contiguous(), **o)
        assert torch.equal(part, whole[b * T:(b + 5) * T]), b
