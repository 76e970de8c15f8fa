"""The deposit of few particles by global atomics against the binned one (which set shapes select):
the same exact sums and conversions, so densities, forces, VJPs and whole gradients are equal
bit for bit, at the edges of the rule, from an even lattice to all particles in one cell."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,n,npc,batch", [(0, 8, 4, 1), (1, 8, 8, 2), (0, 32, 16, 3), (1, 32, 8, 2),
                                                   (0, 64, 64, 1), (0, 64, 32, 2), (0, 64, 32, 8), (0, 128, 64, 1),
                                                   (1, 128, 16, 1)])
@pytest.mark.parametrize("spread", [0.0, 2.0, None])
def test_equal_to_the_binned_deposit(precision, n, npc, batch, spread):
    import torch
    from paper_2211_09815_gb300 import inputs, pm
    dt = torch.float64 if precision else torch.float32
    N = npc ** 3
    g = torch.Generator(device="cuda").manual_seed(n + npc)
    if spread is None:   # every particle into the cell of the first
        j = torch.arange(npc, device="cuda", dtype=dt) * (n // npc)
        q = torch.stack(torch.meshgrid(j, j, j, indexing="ij")).reshape(1, 3, N)
        d = (-q + 0.25 * torch.rand((batch, 3, N), generator=g, device="cuda", dtype=dt)).contiguous()
    else:
        d = spread * torch.randn((batch, 3, N), generator=g, device="cuda", dtype=dt)
    p = torch.randn((batch, 3, N), generator=g, device="cuda", dtype=dt)
    om = torch.randn((batch, npc, npc, npc), generator=g, device="cuda", dtype=dt)
    tgt = torch.randn((batch, n ** 3), generator=g, device="cuda", dtype=dt)
    res = []
    for binned in (False, True):
        ctx = pm.PMContext(float(n), n, npc, 3, [inputs.THETA_FIDUCIAL] * batch, om, precision=precision, batch=batch)
        if binned:
            t = ctx.get_tuning()
            t["fused_x"] = 0
            ctx.set_tuning(t)
        dens = torch.empty(batch, n ** 3, device="cuda", dtype=dt)
        a1, a2, al = (torch.empty(batch, 3, N, device="cuda", dtype=dt) for _ in range(3))
        gw = torch.empty(batch, N, device="cuda", dtype=dt)
        for _ in range(2):   # the sums are left zero
            ctx.op_density(d, dens)
            ctx.op_force(d, a1)
            ctx.op_force_vjp(d, p, a2, al)
            ctx.gradient(tgt, grad_omega=gw)
        ctx.close()
        res.append([x.cpu().numpy() for x in (dens, a1, a2, al, gw)])
    for a, b in zip(*res):
        assert np.array_equal(a, b)
