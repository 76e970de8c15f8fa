"""Small FFT tiles (meshes and side planes of few sequences) against the full ones: a batch
large enough for full tiles and single instances, which take the small ones, run the same
radix stages on every sequence, so the results are equal bit for bit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,n,npc,batch", [(0, 8, 4, 3), (0, 16, 8, 64), (0, 32, 16, 96), (1, 32, 16, 48),
                                                   (0, 64, 32, 40), (1, 64, 16, 20), (0, 128, 64, 9)])
def test_batch_equals_single_instances(precision, n, npc, batch):
    import torch
    from paper_2211_09815_gb300 import inputs, pm
    dt = torch.float32 if precision == 0 else torch.float64
    g = torch.Generator(device="cuda").manual_seed(n)
    om = torch.randn((batch, npc, npc, npc), generator=g, device="cuda", dtype=dt)
    disp = 3.0 * torch.randn((batch, 3, npc ** 3), generator=g, device="cuda", dtype=dt)
    pi = torch.randn((batch, 3, npc ** 3), generator=g, device="cuda", dtype=dt)
    mesh = torch.randn((batch, n, n, n), generator=g, device="cuda", dtype=dt)

    def evaluate(b, sel):
        ctx = pm.PMContext(float(2 * n), n, npc, 1, [inputs.THETA_FIDUCIAL] * b, om[sel].contiguous(),
                           precision=precision, batch=b, lpt_order=2)
        acc, alpha, s0 = (torch.empty(b, 3, npc ** 3, device="cuda", dtype=dt) for _ in range(3))
        spec = torch.empty(b, n, n, n // 2 + 1, 2, device="cuda", dtype=dt)
        back = torch.empty(b, n, n, n, device="cuda", dtype=dt)
        ctx.op_force_vjp(disp[sel].contiguous(), pi[sel].contiguous(), acc, alpha)
        ctx.op_fft(-1, mesh[sel].contiguous(), spec)
        ctx.op_fft(+1, spec, back)
        ctx.op_ic(s0=s0)
        ctx.close()
        return [v.cpu().numpy() for v in (acc, alpha, spec, back, s0)]

    whole = evaluate(batch, slice(0, batch))
    for i in sorted({0, 1, batch - 1}):
        for a, b in zip(whole, evaluate(1, slice(i, i + 1))):
            assert np.array_equal(a[i], b[0])
    # the round trip returns the mesh times n^3
    m = mesh.cpu().numpy()
    tol = (1e-5 if precision == 0 else 1e-13) * np.abs(m).max()
    assert np.max(np.abs(whole[3] / n ** 3 - m)) < tol
