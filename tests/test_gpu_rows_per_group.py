"""Kinetics at d = 16 and 32: how many rows a group of lanes linearises, and at d = 16 in mixed
precision which form does, goes by the number of rows. A sequence alone (a row per group) ends at
the same bits as in a batch that fills the GPU (eight rows per group; two columns per lane).
"""
import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,R", [(16, 24), (16, 64), (32, 48)])
@pytest.mark.parametrize("prec", ["fp32", "fp64", "mixed_bf16"])
@pytest.mark.parametrize("integrator", ["rk4", "euler"])
@pytest.mark.parametrize("iters", [1, 4, 12])
def test_alone_as_in_a_batch(d, R, prec, integrator, iters):
    import paper_2603_16850_gb300 as deer
    lengths = [1, 9, 700] + [2003] * 72  # 144926 rows
    B, off = len(lengths), synth.offsets_from_lengths([1, 9, 700] + [2003] * 72)
    p = synth.massaction(B, d, R, 1, seed=51, integrator=integrator)
    dt = torch.float32 if prec == "fp32" else torch.float64
    topo = torch.tensor(p["topology"], dtype=torch.int32, device="cuda")
    k = torch.tensor(p["params"], dtype=dt, device="cuda")
    s0 = torch.tensor(p["s0"], dtype=dt, device="cuda")

    def solve(first, last, offsets):
        dyn = deer.Dynamics.massaction(topo[first:last].contiguous(), k[first:last].contiguous(), d,
                                       p["dt"], integrator)
        s, info = deer.deer_solve_batched(dyn, s0[first:last].contiguous(), offsets, jac="full",
                                          prec=prec, init="s0", reset=True, tol=0.0,
                                          max_iters=iters)
        return s, info.max_resid

    whole, resid = solve(0, B, off)
    for b in (0, 1, 2, 3, B - 1):
        one, r = solve(b, b + 1, np.array([0, lengths[b]]))
        assert torch.equal(one, whole[off[b]:off[b + 1]]), b
        assert torch.equal(r[0].isnan(), resid[b].isnan()), b
        assert bool(r[0].isnan()) or float(r[0]) == float(resid[b]), b
