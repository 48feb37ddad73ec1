"""The convergence test of the one-kernel solve against the multi-kernel loop's: a tolerance that
no residual meets (negative, NaN) runs to the iteration cap on both, also with an empty sequence
in the batch, and a sequence counts as converged exactly when its reported largest residual is at
or below the tolerance, at the last bit.
"""
import math

import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu


def _brusselator(prec):
    import paper_2603_16850_gb300 as deer
    dt = torch.float64 if prec == "fp64" else torch.float32
    p = synth.brusselator(T=64)
    dyn = deer.Dynamics.brusselator(torch.tensor(p["params"], dtype=dt, device="cuda"), p["dt"])
    return deer, dyn, torch.tensor(p["s0"], dtype=dt, device="cuda")


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("tol", [-1.0, -1e-300, math.nan])
@pytest.mark.parametrize("init", ["s0", "zeros"])
def test_tolerance_that_nothing_meets(prec, tol, init):
    deer, dyn, s0 = _brusselator(prec)
    got = {}
    for block in (True, False):
        s, info = deer.deer_solve(dyn, s0, 64, jac="full", tol=tol, max_iters=7, prec=prec,
                                  init=init, reset=True, block_solve=block)
        assert info.iters.tolist() == [7] and not bool(info.converged.any()), (block, info)
        got[block] = s
    scale = got[False].abs().max()
    assert (got[True] - got[False]).abs().max() <= (1e-10 if prec == "fp64" else 1e-4) * scale


@pytest.mark.parametrize("tol", [-1.0, math.nan])
def test_empty_sequence_under_such_a_tolerance(tol):
    deer, dyn, s0 = _brusselator("fp64")
    for block in (True, False):
        _, info = deer.deer_solve_batched(dyn, s0.repeat(3, 1), [0, 20, 20, 50], jac="full",
                                          tol=tol, max_iters=3, prec="fp64", init="s0",
                                          block_solve=block)
        assert info.iters.tolist() == [3, 3, 3] and not bool(info.converged.any()), (block, info)


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_converged_exactly_when_the_reported_residual_meets_the_tolerance(prec):
    import paper_2603_16850_gb300 as deer
    dt = torch.float64 if prec == "fp64" else torch.float32
    real = np.float64 if prec == "fp64" else np.float32
    rng = np.random.default_rng(3)
    B, T = 96, 64
    ab = np.stack([rng.uniform(0.9, 1.1, B), rng.uniform(2.8, 3.2, B)], axis=1)
    s0 = torch.tensor(rng.uniform(0.9, 1.6, (B, 2)), dtype=dt, device="cuda")
    dyn = deer.Dynamics.brusselator(torch.tensor(ab, dtype=dt, device="cuda"), 0.01)

    def solve(tol, k):
        return deer.deer_solve(dyn, s0, T, jac="full", tol=tol, max_iters=k, prec=prec,
                               init="s0")[1]

    for k in (1, 2):
        res = solve(-1.0, k).max_resid.numpy()  # every sequence after k steps
        assert np.all(res > 0)
        for r in res[:24]:
            for tol in (float(r), float(np.nextafter(real(r), real(0)))):
                info = solve(tol, k)
                ended = info.iters.numpy() == k
                assert np.array_equal(info.converged.numpy()[ended],
                                      info.max_resid.numpy()[ended] <= tol)
                assert np.array_equal(ended & info.converged.numpy(), ended & (res <= tol))
