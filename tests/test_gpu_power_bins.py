"""The shell sums of the power spectrum at the edges of their runs and bins: the smallest
meshes (runs of 4 kx), runs of 8, batches, and the z-blocked rows of 1024^3, against FP64 sums
over the numpy layout; rows of very different magnitude in one bin."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def reference(torch, d, box):
    """(P, modes) of one FP64 mesh on the device."""
    n = d.shape[0]
    f = torch.fft.fftfreq(n, 1.0 / n, dtype=torch.float64, device="cuda")
    n2 = f.view(n, 1, 1) ** 2 + f.view(1, n, 1) ** 2 + torch.arange(n // 2 + 1, device="cuda").view(1, 1, -1) ** 2
    b = torch.floor(torch.sqrt(n2)).to(torch.int64).reshape(-1)
    del n2
    w = torch.full((n // 2 + 1,), 2.0, dtype=torch.float64, device="cuda")
    w[0] = w[-1] = 1.0
    p = torch.fft.rfftn(d).abs().square_().mul_(w).reshape(-1)
    size = int(b.max()) + 1
    s = torch.zeros(size, dtype=torch.float64, device="cuda").index_add_(0, b, p)[: n // 2]
    c = torch.zeros(size, dtype=torch.float64, device="cuda").index_add_(
        0, b, w.expand(n, n, -1).reshape(-1))[: n // 2]
    return (box ** 3 / n ** 6 * s / c).cpu().numpy(), c.cpu().numpy()


@pytest.mark.parametrize("precision,n,batch", [(0, 8, 3), (1, 8, 1), (0, 16, 2), (1, 16, 2), (0, 128, 2), (1, 64, 1),
                                               (0, 1024, 1)])
def test_shell_sums(precision, n, batch):
    import torch
    from paper_2211_09815_gb300 import inputs, pm
    dt = torch.float32 if precision == 0 else torch.float64
    npc, box = max(4, n // 4), 50.0
    ctx = pm.PMContext(box, n, npc, 1, [inputs.THETA_FIDUCIAL] * batch, torch.zeros(batch, npc, npc, npc,
                                                                                   device="cuda", dtype=dt),
                       precision=precision, batch=batch)
    g = torch.Generator(device="cuda").manual_seed(n)
    d = torch.randn((batch, n, n, n), generator=g, device="cuda", dtype=dt)
    # one plane wave 2^10 above the rest: the modes of its bin differ by 2^20 in power
    x = torch.arange(n, device="cuda", dtype=dt) * (2 * np.pi / n)
    d += 1024.0 * n ** -1.5 * torch.cos(2 * x).view(1, n, 1, 1)
    km, pk, modes = ctx.power_spectrum(d)
    # the FP32 transform is good to about 1e-6 of the largest mode; the sums add nothing to that
    tol = 1e-12 if precision else 1e-5
    for b in range(batch):
        p, c = reference(torch, d[b].double(), box)
        assert np.array_equal(modes, c)
        assert np.max(np.abs(pk[b][1:] / p[1:] - 1)) < tol
    ctx.close()
