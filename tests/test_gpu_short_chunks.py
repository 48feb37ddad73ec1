"""Float64 kinetics on a few warps, whose default chunk goes down to eight rows: sequences of less
than a chunk, a whole number of chunks, one row more, and both sides of the rule's longest
sequence (2048 rows). The fixed point is the float64 rollout, to 1e-10.
"""
import numpy as np
import pytest
import torch

import synth
from oracle import cma

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,T", [(1, 1), (5, 7), (5, 8), (37, 65), (3, 2048), (3, 2049)])
@pytest.mark.parametrize("window", [False, True])
def test_default_chunk(B, T, window):
    import paper_2603_16850_gb300 as deer
    p = synth.massaction(B, 8, 12, 1, seed=17)
    dyn = deer.Dynamics.massaction(
        torch.tensor(p["topology"], dtype=torch.int32, device="cuda"),
        torch.tensor(p["params"], device="cuda"), 8, p["dt"])
    s, _ = deer.deer_solve(dyn, torch.tensor(p["s0"], device="cuda"), T, jac="full",
                           prec="fp64", tol=1e-12, confirm=2, init="s0", reset=True,
                           window=window)
    off = np.arange(B + 1) * T
    ref = cma.Batch(p["topology"], p["params"], p["dt"], "rk4", d=8).rollout(p["s0"], off)
    got = s.cpu().numpy().reshape(B * T, 8)
    assert np.max(np.abs(got - ref.reshape(B * T, 8))) / np.max(np.abs(ref)) <= 1e-10
