"""Mixed precision at d = 32 over long sequences: the carry over segments of chunks costs no
iterations against the carry over the chunks themselves (longer chunks, fewer than the 128 from
which they are folded). Newton's last factors converge linearly at the rounding of the composed
products, so a fold at lower precision than the chunk products shows as more iterations.
"""
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu


def test_folded_carry_takes_no_more_iterations():
    import paper_2603_16850_gb300 as deer
    lengths = [60000] * 2
    off = synth.offsets_from_lengths(lengths)
    p = synth.massaction(2, 32, 48, 1, seed=5)
    dyn = deer.Dynamics.massaction(
        torch.tensor(p["topology"], dtype=torch.int32, device="cuda"),
        torch.tensor(p["params"], device="cuda"), 32, p["dt"])
    s0 = torch.tensor(p["s0"], device="cuda")

    def iters(chunk):
        info = deer.deer_solve_batched(dyn, s0, off, jac="full", tol=1e-12, prec="mixed_bf16",
                                       init="zeros", reset=True, window=True, max_iters=600,
                                       chunk=chunk)[1]
        assert bool(info.converged.all())
        return info.iters

    folded, plain = iters(0), iters(1024)
    assert bool((folded <= plain + 2).all()), (folded, plain)
