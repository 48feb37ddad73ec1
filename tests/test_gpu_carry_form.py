"""The carry of a dense scan takes one form for a whole call, also where the active set falls
below the batch size at which the chunks would be folded into segments: the device-resident loop
(sized for the whole batch) and the host loop (sized for the active set) return the same bits, and
so does a sequence in a batch whose other members converge at once.
"""
import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu


def test_same_form_while_the_active_set_shrinks():
    import paper_2603_16850_gb300 as deer
    # 128 chunks of 8 rows; more sequences than the folds are taken for, most of which start at
    # their solution
    B, T, d, live = 2440, 1024, 8, 40
    p = synth.mean_field_rnn(live, T, d, 0.9, seed=9)
    f = torch.float32
    W = torch.tensor(p["W"], dtype=f, device="cuda")
    x = torch.zeros(B, T, d, dtype=f, device="cuda")
    s0 = torch.zeros(B, d, dtype=f, device="cuda")
    x[-live:] = torch.tensor(p["x"], dtype=f, device="cuda")
    s0[-live:] = torch.tensor(p["s0"], dtype=f, device="cuda")

    def solve(**extra):
        return deer.deer_solve(deer.Dynamics.rnn_tanh(W), s0, T, x.reshape(-1, d), jac="full",
                               tol=5e-7, prec="fp32", init="zeros", chunk=8, block_solve=False,
                               **extra)

    s_h, i_h = solve(device_loop=False)
    s_d, i_d = solve(device_loop=True)
    iters = i_h.iters.numpy()
    assert bool(i_h.converged.all()) and np.all(iters[:-live] == 0) and np.all(iters[-live:] > 1)
    assert torch.equal(s_h, s_d)
    assert i_h.iters.tolist() == i_d.iters.tolist()
    assert torch.equal(i_h.max_resid, i_d.max_resid)
