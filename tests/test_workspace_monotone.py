"""A workspace that holds a problem holds every smaller one of the same system and options:
deer_workspace_bytes and deer_grad_workspace_bytes never fall as sequences or rows are added,
across the sizes at which the default chunk length changes (host arithmetic only).
"""
import ctypes as C

import pytest


def _sizes(lo, hi):
    out, n = set(), lo
    while n <= hi:
        out.update((n - 1, n, n + 1))
        n = n * 5 // 4 + 1
    # both sides of the default chunk's limits on T
    out.update(t + e for t in (512, 2048, 2051, 4096, 8192, 32768) for e in (-1, 0, 1))
    return sorted(t for t in out if lo <= t <= hi)


@pytest.mark.parametrize("kind,d", [("massaction_rk4", 4), ("massaction_rk4", 8),
                                    ("massaction_rk4", 16), ("langevin_2well", 4),
                                    ("brusselator_euler", 2), ("rnn_tanh", 8)])
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("damp", ["none", "elk"])
def test_workspace_never_falls(kind, d, prec, damp):
    from paper_2603_16850_gb300 import _native as N
    lib = N.load()
    o = N.deer_options()
    lib.deer_default_options(C.byref(o))
    o.prec, o.jac, o.damp = N.PREC[prec], N.JAC["full"], N.DAMP[damp]
    o.damp_param = 0.5
    R = 12 if kind.startswith("mass") else 0
    stride = {"massaction_rk4": 12, "langevin_2well": 4 * d + 2, "brusselator_euler": 2,
              "rnn_tanh": d * d}[kind]
    dyn = N.deer_dynamics(N.KIND[kind], d, d, R, 0.01, 8, stride, 8 if R else 0, 4 * R)
    batches = [1, 2, 3, 7, 37, 101, 300, 301, 512, 4000]
    times = _sizes(1, 40000)
    before = [0] * len(times)
    for B in batches:
        last = 0
        for j, T in enumerate(times):
            need = lib.deer_workspace_bytes(C.byref(dyn), B, B * T, C.byref(o))
            assert need >= last and need >= before[j], (B, T)
            last = before[j] = need
    last = 0
    for N_rows in times:  # ragged: any row count with a batch size
        need = lib.deer_workspace_bytes(C.byref(dyn), 37, N_rows, C.byref(o))
        assert need >= last, N_rows
        last = need
    if damp == "none":
        for B in (1, 37):
            last = 0
            for T in times:
                need = lib.deer_grad_workspace_bytes(C.byref(dyn), B, T, C.byref(o))
                assert need >= last, (B, T)
                last = need
