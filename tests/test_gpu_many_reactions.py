"""Networks of more reactions than 16 bits number (d = 16 and 32): the solve and the adjoint
against the recurrence written out in float64, whose gradient is torch's. Only the last reactions
and a few early ones run at rates that matter, so that a list naming reaction r - 65536 in
place of r is far off. Tolerance 1e-10 (float64).
"""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d", [16, 32])
@pytest.mark.parametrize("R", [65535, 65536, 65552])
def test_many_reactions(d, R):
    import paper_2603_16850_gb300 as deer
    T, dt = 24, 1e-2
    rng = np.random.default_rng(R + d)
    topo = np.full((R, 4), -1, dtype=np.int32)
    topo[:, 0] = rng.integers(0, d, R)
    topo[:, 2] = (topo[:, 0] + rng.integers(1, d, R)) % d
    two = rng.random(R) < 0.5
    topo[two, 1] = rng.integers(0, d, int(two.sum()))
    k = np.full(R, 1e-9)
    k[-20:] = rng.uniform(0.5, 2.0, 20)
    k[rng.integers(0, 1000, 20)] = rng.uniform(0.5, 2.0, 20)
    s0 = rng.uniform(0.2, 1.0, (1, d))

    def dev(a, t=torch.float64):
        return torch.tensor(a, dtype=t, device="cuda")

    dyn = deer.Dynamics.massaction(dev(topo[None], torch.int32), dev(k[None]), d, dt, "euler")
    s, info = deer.deer_solve(dyn, dev(s0), T, jac="full", tol=1e-13, init="s0", max_iters=30)
    assert bool(info.converged.all())
    # the same recurrence: ds_i/dt = sum_r nu_ri k_r c_i1 c_i2
    i1, i2, p1 = (torch.tensor(topo[:, j].astype(np.int64)) for j in (0, 1, 2))
    start = torch.tensor(s0[0], requires_grad=True)
    kt = torch.tensor(k)
    c, out = start, []
    for _ in range(T):
        rate = kt * c[i1] * torch.where(i2 < 0, torch.ones_like(kt), c[i2.clamp(min=0)])
        rate2 = torch.where(i2 < 0, torch.zeros_like(rate), rate)
        dc = torch.zeros(d, dtype=torch.float64).index_add(0, p1, rate).index_add(0, i1, -rate)
        c = c + dt * dc.index_add(0, i2.clamp(min=0), -rate2)
        out.append(c)
    ref = torch.stack(out)
    assert (s.cpu() - ref.detach()).abs().max() <= 1e-10
    g = torch.tensor(rng.standard_normal((T, d)))
    (ref * g).sum().backward()
    _, ds0 = deer.deer_grad(dyn, dev(s0), T, s, g.cuda())
    assert (ds0.cpu()[0] - start.grad).abs().max() <= 1e-10 * start.grad.abs().max()
