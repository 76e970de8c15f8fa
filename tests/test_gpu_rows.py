"""The x passes that keep a row in the lanes of a warp (rows of 128 to 1024 reals, FP32), at every
row length: both directions of the 3-D transform against FP64, and the force through the
three- and four-component C2R in FP32 and in the FP16 form."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,batch", [(128, 3), (256, 1), (512, 1), (1024, 1)])
def test_transforms_match_fp64(n, batch):
    import torch
    from paper_2211_09815_gb300 import inputs, pm
    g = torch.Generator(device="cuda").manual_seed(n)
    x = torch.randn((batch, n, n, n), generator=g, device="cuda")
    ctx = pm.PMContext(100.0, n, 16, 1, [inputs.THETA_FIDUCIAL] * batch, torch.zeros(batch, 16, 16, 16, device="cuda"),
                       batch=batch)
    spec = torch.empty((batch, n, n, n // 2 + 1, 2), device="cuda")
    ctx.op_fft(-1, x, spec)
    back = torch.empty_like(x)
    ctx.op_fft(+1, spec, back)
    ctx.close()
    # FP32 rounding through 3 log2(n) stages: well below 3 log2(n) eps = 2e-6 in the 2-norm
    for b in range(batch):
        ref = torch.view_as_real(torch.fft.rfftn(x[b].double()))
        assert float((spec[b] - ref).norm() / ref.norm()) < 1e-6
        del ref
        assert float((back[b].double() / n ** 3 - x[b]).norm() / x[b].double().norm()) < 1e-6


@pytest.mark.parametrize("n,npc", [(128, 32), (256, 32), (512, 64)])
def test_force_forms_agree(n, npc):
    import torch
    from paper_2211_09815_gb300 import inputs, pm
    g = torch.Generator(device="cuda").manual_seed(npc)
    d = 4.0 * torch.randn((3, npc ** 3), generator=g, device="cuda")
    q = torch.randn((3, npc ** 3), generator=g, device="cuda")
    out = {}
    for name, prec, half in (("f32", 0, False), ("f64", 1, False), ("half", 0, True)):
        dt = torch.float64 if prec else torch.float32
        ctx = pm.PMContext(float(n), n, npc, 1, [inputs.THETA_FIDUCIAL], torch.zeros(npc, npc, npc, device="cuda", dtype=dt),
                           precision=prec, half_force=half)
        a1, a2, al = (torch.empty((3, npc ** 3), device="cuda", dtype=dt) for _ in range(3))
        ctx.op_force(d.to(dt), a1)            # three components
        ctx.op_force_vjp(d.to(dt), q.to(dt), a2, al)   # four
        ctx.close()
        out[name] = (a1.double(), a2.double(), al.double())
    def rel(u, v):
        return float((u - v).norm() / v.norm())
    # positions of order 4 cells rounded to FP32 move a weight by 2e-7: a force error of that order,
    # and one at a cell face flips the VJP's weight gradient with a chance of 1e-6 per particle
    for k in (0, 1):
        assert rel(out["f32"][k], out["f64"][k]) < 5e-6
        assert rel(out["half"][k], out["f32"][k]) < 1e-3       # 11 bits per value: 2e-4 in the 2-norm
    assert rel(out["half"][2], out["f32"][2]) < 1e-2
