"""Operators whose inputs start at any byte: a particle array of the C interface need not be aligned
to its elements, and gives the results of an aligned copy."""
import ctypes

import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,shift", [(0, 1), (0, 2), (1, 1), (1, 4)])
@pytest.mark.parametrize("n,npc", [(32, 16), (64, 64)])   # deposits by atomics and by bins (VJP)
def test_inputs_off_their_alignment(precision, shift, n, npc):
    import torch
    from paper_2211_09815_gb300 import inputs, pm
    dt = torch.float64 if precision else torch.float32
    v, size = 3 * npc ** 3, 8 if precision else 4
    g = torch.Generator(device="cuda").manual_seed(5)
    d = 2.0 * torch.randn(v, generator=g, device="cuda", dtype=dt)
    p = torch.randn(v, generator=g, device="cuda", dtype=dt)
    ctx = pm.PMContext(50.0, n, npc, 1, [inputs.THETA_FIDUCIAL], torch.zeros(npc, npc, npc, device="cuda", dtype=dt),
                       precision=precision)
    dens, dens2 = (torch.empty(n ** 3, device="cuda", dtype=dt) for _ in range(2))
    acc, acc2, alpha, alpha2 = (torch.empty(v, device="cuda", dtype=dt) for _ in range(4))
    ctx.op_density(d, dens)
    ctx.op_force_vjp(d, p, acc, alpha)

    def shifted(t):
        raw = torch.empty(size * v + 16, device="cuda", dtype=torch.uint8)
        raw[shift:shift + size * v] = t.view(torch.uint8)
        return raw, ctypes.c_void_p(raw.data_ptr() + shift)

    (raw_d, pd), (raw_p, pp) = shifted(d), shifted(p)
    out = [ctypes.c_void_p(t.data_ptr()) for t in (dens2, acc2, alpha2)]
    lib = pm.load_library()
    assert lib.pm_op_density(ctx._h, pd, out[0]) == 0
    assert lib.pm_op_force_vjp(ctx._h, pd, pp, out[1], out[2]) == 0
    ctx.check()
    assert torch.equal(dens, dens2) and torch.equal(acc, acc2) and torch.equal(alpha, alpha2)
    acc2.zero_()
    assert lib.pm_op_force(ctx._h, pd, out[1]) == 0
    ctx.check()
    assert torch.equal(acc, acc2)
    ctx.close()
