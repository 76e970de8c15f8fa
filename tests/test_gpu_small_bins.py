"""The binned deposit on meshes shorter than its tiles (8^3 and 16^3), which batches take by
default and set shapes always: equal to single instances bit for bit, since the sums are exact."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def evaluate(torch, n, npc, sel, om, disp, pi, tgt, tuning=None):
    from paper_2211_09815_gb300 import inputs, pm
    b, N, dt = len(sel), npc ** 3, om.dtype
    ctx = pm.PMContext(float(n), n, npc, 2, [inputs.THETA_FIDUCIAL] * b, om[sel].contiguous(),
                       precision=int(dt == torch.float64), batch=b)
    if tuning:
        ctx.set_tuning(tuning)
    dens = torch.empty(b, n ** 3, device="cuda", dtype=dt)
    acc, acc2, alpha = (torch.empty(b, 3, N, device="cuda", dtype=dt) for _ in range(3))
    gw = torch.empty(b, N, device="cuda", dtype=dt)
    ctx.op_density(disp[sel].contiguous(), dens)
    ctx.op_force(disp[sel].contiguous(), acc)
    ctx.op_force_vjp(disp[sel].contiguous(), pi[sel].contiguous(), acc2, alpha)
    ctx.gradient(tgt[sel].contiguous(), grad_omega=gw)
    ctx.close()
    return [v.cpu().numpy() for v in (dens, acc, acc2, alpha, gw)]


def arrays(torch, n, npc, batch, precision):
    dt = torch.float64 if precision else torch.float32
    g = torch.Generator(device="cuda").manual_seed(n * npc)
    def rand(*shape):
        return torch.randn(shape, generator=g, device="cuda", dtype=dt)
    return rand(batch, npc, npc, npc), 2.0 * rand(batch, 3, npc ** 3), rand(batch, 3, npc ** 3), rand(batch, n ** 3)


# (16, 16): VJP binned from 17 instances on, density from 65; (16, 8) and (16, 4): VJP from 129;
# (8, 8): VJP from 129; from 304 instances of 16^3 on the larger default tiles
@pytest.mark.parametrize("precision,n,npc,batch", [(0, 16, 16, 20), (1, 16, 16, 20), (0, 16, 16, 80), (0, 16, 4, 160),
                                                   (0, 8, 8, 130), (1, 8, 8, 600), (0, 16, 16, 310)])
def test_batches_equal_single_instances(precision, n, npc, batch):
    import torch
    data = arrays(torch, n, npc, batch, precision)
    whole = evaluate(torch, n, npc, list(range(batch)), *data)
    for i in (0, batch // 2, batch - 1):
        for a, b in zip(whole, evaluate(torch, n, npc, [i], *data)):
            assert np.array_equal(a[i], b[0])


# shapes cut to fewer than 2^9 cells: a row of the mesh per tile the smallest
@pytest.mark.parametrize("n,npc,batch", [(8, 8, 1), (16, 16, 1), (16, 16, 9), (64, 16, 2), (128, 16, 1), (256, 16, 1)])
def test_set_shapes_equal_the_default(n, npc, batch):
    import torch
    data = arrays(torch, n, npc, batch, 0)
    sel = list(range(batch))
    default = evaluate(torch, n, npc, sel, *data)
    for tile in ([0, 0, 9], [2, 0, 9], [9, 0, 2], [2, 2, 7], [3, 3, 3]):
        other = evaluate(torch, n, npc, sel, *data,
                         tuning={"tile_log2_density": tile, "tile_log2_adjoint": tile, "fused_x": 0})
        for a, b in zip(default, other):
            assert np.array_equal(a, b)
