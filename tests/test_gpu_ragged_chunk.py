"""The default chunk length of a ragged batch follows its longest sequence, whose carry is the
longest chain of an iteration: one long sequence among short ones takes the chunks that it would
take alone, not those of the mean length (same bits after two iterations as with that length given;
another length rounds its products differently).
"""
import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lengths,chunk", [([500] * 60 + [40000], 64),
                                           ([300] * 40 + [20000], 32),
                                           ([100] * 7 + [2049], 16),
                                           ([100] * 7 + [2048], 8)])
def test_default_chunk_of_ragged_batch(lengths, chunk):
    import paper_2603_16850_gb300 as deer
    B, off = len(lengths), np.concatenate([[0], np.cumsum(lengths)])
    p = synth.massaction(B, 8, 12, 1, seed=31)
    dyn = deer.Dynamics.massaction(
        torch.tensor(p["topology"], dtype=torch.int32, device="cuda"),
        torch.tensor(p["params"], device="cuda"), 8, p["dt"])
    s0 = torch.tensor(p["s0"], device="cuda")

    def solve(c):
        return deer.deer_solve_batched(dyn, s0, off, jac="full", tol=0.0, max_iters=2, prec="fp64",
                                       init="s0", reset=True, chunk=c)[0]

    got, shorter = solve(0), solve(8 if chunk > 8 else 16)
    assert torch.equal(got, solve(chunk))
    assert not torch.equal(got, shorter)  # the length does show in the bits
