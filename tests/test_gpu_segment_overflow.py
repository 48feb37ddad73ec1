"""The two-level carry of the dense scans where the product over a segment of chunks overflows and
the products over single chunks do not: systems whose growing coordinates stay at zero while the
others are driven (linear, and the mean-field RNN, whose Jacobian at zero is W). The growing
coordinates end exactly zero, the driven ones at the sequential recurrence (float64 1e-13,
float32 1e-5: 1 / (1 - 0.5) times the rounding of a row), and the call converges.
"""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

# longest sequence: 256 chunks of 32 rows, folded by 16 (512 rows: 1.5^512 and 4^512 overflow);
# the others end inside a chunk, inside a segment, just past one, and before the first
LENGTHS = [8192, 8191, 7 * 512 + 33, 512, 513, 0, 5]


@pytest.mark.parametrize("kind,d", [("linear", 16), ("linear", 32), ("rnn", 2), ("rnn", 4),
                                    ("rnn", 8), ("rnn", 16), ("rnn", 32)])
@pytest.mark.parametrize("prec,growth", [("fp32", 1.5), ("fp64", 4.0)])
@pytest.mark.parametrize("reset", [False, True])
@pytest.mark.parametrize("window", [False, True])
def test_overflowing_segment_products(kind, d, prec, growth, reset, window):
    import paper_2603_16850_gb300 as deer
    dt = torch.float32 if prec == "fp32" else torch.float64
    B, off = len(LENGTHS), np.concatenate([[0], np.cumsum(LENGTHS)])
    a = np.where(np.arange(d) % 2 == 0, growth, 0.5)
    rng = np.random.default_rng(d)
    x = rng.uniform(-1.0, 1.0, (off[-1], d)) * (a < 1.0)
    s0 = rng.uniform(-1.0, 1.0, (B, d)) * (a < 1.0)

    def dev(v):
        return torch.tensor(v, dtype=dt, device="cuda")

    W = dev(np.diag(a))
    dyn = deer.Dynamics.linear(W) if kind == "linear" else deer.Dynamics.rnn_tanh(W)
    s, info = deer.deer_solve_batched(dyn, dev(s0), off, dev(x), jac="full", confirm=2,
                                      tol=1e-5 if prec == "fp32" else 1e-13, prec=prec,
                                      init="zeros", chunk=32, reset=reset, window=window,
                                      max_iters=20, block_solve=False)
    assert bool(info.converged.all()), info
    act = (lambda v: v) if kind == "linear" else np.tanh
    xr, sr = dev(x).double().cpu().numpy(), dev(s0).double().cpu().numpy()  # as rounded
    ref = np.zeros_like(x)
    for b in range(B):
        s_t = sr[b]
        for t in range(off[b], off[b + 1]):
            s_t = a * act(s_t) + xr[t]
            ref[t] = s_t
    got = s.double().cpu().numpy()
    assert np.all(got[:, a > 1.0] == 0.0)
    assert np.max(np.abs(got - ref)) <= (1e-5 if prec == "fp32" else 1e-13)


@pytest.mark.parametrize("d,prec,growth", [(16, "fp32", 1.5), (32, "fp32", 1.5),
                                           (16, "fp64", 4.0), (32, "fp64", 4.0)])
@pytest.mark.parametrize("reset", [False, True])
def test_solution_as_guess(d, prec, growth, reset):
    """s = 0 solves s_t = g s_{t-1} from s_0 = 0; the one scan between the two confirming passes
    must leave it there (default chunk length)."""
    import paper_2603_16850_gb300 as deer
    dt = torch.float32 if prec == "fp32" else torch.float64
    dyn = deer.Dynamics.linear(growth * torch.eye(d, dtype=dt, device="cuda"))
    s0 = torch.zeros(1, d, dtype=dt, device="cuda")
    s, info = deer.deer_solve(dyn, s0, 8192, jac="full", tol=1e-6, confirm=2, prec=prec,
                              init="zeros", reset=reset)
    assert info.iters.tolist() == [1] and bool(info.converged.all()), info
    assert not bool(s.any())


@pytest.mark.parametrize("d", [16, 32])
@pytest.mark.parametrize("prec,limit", [("fp32", 1e18), ("fp64", 1e30)])
def test_correction_that_overflows_itself(d, prec, limit):
    """s_t = 2 s_{t-1} from the zero guess: the one step's correction is 2^t, exact until it
    overflows; entries above the reset threshold, and all from the overflow on, end at zero. A
    sequence beside it is solved as ever."""
    import paper_2603_16850_gb300 as deer
    dt = torch.float32 if prec == "fp32" else torch.float64
    T = 8192
    A = torch.diag(torch.tensor([2.0] + [0.5] * (d - 1), dtype=dt, device="cuda"))
    s0 = torch.zeros(2, d, dtype=dt, device="cuda")
    s0[0, 0] = s0[0, 1] = s0[1, 1] = 1.0
    s, _ = deer.deer_solve(deer.Dynamics.linear(A), s0, T, jac="full", tol=0.0, max_iters=1,
                           prec=prec, init="zeros", reset=True, chunk=32)
    got = s.double().cpu().numpy().reshape(2, T, d)
    t = np.arange(1, T + 1, dtype=np.float64)
    over = 128 if prec == "fp32" else 1024  # 2^t is not a number of the type from here on
    with np.errstate(over="ignore", under="ignore"):
        up, down = np.exp2(t), np.exp2(-t)
    assert np.array_equal(got[0, :, 0], np.where(up <= limit, up, 0.0))
    assert np.all(got[:, :, 2:] == 0.0) and np.all(got[1, :, 0] == 0.0)
    # float32 subnormals and below: not more than the smallest normal number away
    tiny = 1.2e-38 if prec == "fp32" else 2.3e-308
    assert np.all(np.abs(got[1, :, 1] - down) <= tiny)
    # the coordinate beside the growing one: solved before the overflow, zero after it
    assert np.all(np.abs(got[0, :over - 1, 1] - down[:over - 1]) <= tiny)
    assert np.all(got[0, over:, 1] == 0.0)
