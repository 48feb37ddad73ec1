"""Kinetics whose species take part in more reactions than the linearisations keep in shared
memory (16), with a network per sequence and sequences shorter than, equal to and longer than
the eight rows that a group of lanes walks: the fixed point is the float64 rollout, to 1e-9 in
float64 and mixed precision and to 2e-5 in float32 (130 steps of one rounding each).
"""
import numpy as np
import pytest
import torch

import synth
from oracle import cma

pytestmark = pytest.mark.gpu

LENGTHS = [1, 7, 9, 0, 130, 3, 8, 64]


@pytest.mark.parametrize("d,R,prec,jac_bytes", [
    (16, 24, "mixed_bf16", 0), (16, 64, "mixed_bf16", 0), (16, 64, "mixed_bf16", 1),
    (32, 64, "mixed_bf16", 0), (16, 64, "fp32", 0), (32, 33, "fp32", 0), (32, 128, "fp32", 0),
    (16, 64, "fp64", 0), (32, 128, "fp64", 0)])
@pytest.mark.parametrize("integrator", ["rk4", "euler"])
def test_long_species_lists(d, R, prec, jac_bytes, integrator):
    import paper_2603_16850_gb300 as deer
    B = len(LENGTHS)
    off = synth.offsets_from_lengths(LENGTHS)
    p = synth.massaction(B, d, R, 1, seed=41, integrator=integrator)
    dt = torch.float32 if prec == "fp32" else torch.float64
    dyn = deer.Dynamics.massaction(
        torch.tensor(p["topology"], dtype=torch.int32, device="cuda"),
        torch.tensor(p["params"], dtype=dt, device="cuda"), d, p["dt"], integrator)
    s, _ = deer.deer_solve_batched(dyn, torch.tensor(p["s0"], dtype=dt, device="cuda"), off,
                                   jac="full", prec=prec, init="s0", reset=True, tol=0.0,
                                   max_iters=12, jac_bytes_max=jac_bytes)
    ref = cma.Batch(p["topology"], p["params"], p["dt"], integrator, d=d).rollout(p["s0"], off)
    got = s.double().cpu().numpy()
    err = np.max(np.abs(got - ref)) / np.max(np.abs(ref))
    assert err <= (2e-5 if prec == "fp32" else 1e-9)
