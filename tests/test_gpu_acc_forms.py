"""The accelerations of the forward and of the adjoint force chain (C2R of three and of four
components) are equal bit for bit, which the exact reversal of the fixed-point state rests on: at
every row length with a form of its own, and in a reverse pass on 256^3."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,half", [(64, False), (128, False), (256, False), (512, False), (1024, False), (128, True),
                                    (256, True), (512, True)])
def test_force_and_vjp_give_the_same_accelerations(n, half):
    import torch
    from paper_2211_09815_gb300 import inputs, pm
    npc = 32
    g = torch.Generator(device="cuda").manual_seed(n)
    d = 4.0 * torch.randn((3, npc ** 3), generator=g, device="cuda")
    q = torch.randn((3, npc ** 3), generator=g, device="cuda")
    ctx = pm.PMContext(float(n), n, npc, 1, [inputs.THETA_FIDUCIAL], torch.zeros(npc, npc, npc, device="cuda"),
                       half_force=half)
    if n >= 128:
        ctx.set_tuning({"fused_x": 0})   # the fixed-point state's x pass in both chains
    a1, a2, al = (torch.empty_like(d) for _ in range(3))
    ctx.op_force(d, a1)
    ctx.op_force_vjp(d, q, a2, al)
    ctx.close()
    assert torch.equal(a1, a2)


@pytest.mark.parametrize("half", [False, True])
def test_reverse_pass_recovers_the_initial_state_at_256(half):
    import torch
    from paper_2211_09815_gb300 import inputs, pm
    n, npc = 256, 64
    om = torch.from_numpy(inputs.white_noise(npc, 1)).cuda()
    ctx = pm.PMContext(400.0, n, npc, 8, [inputs.THETA_FIDUCIAL], om, fixed_state=True, half_force=half)
    u0, w0, u1, w1 = (torch.empty(3 * npc ** 3, device="cuda", dtype=torch.int64) for _ in range(4))
    ctx.op_ic()
    ctx.get_fixed_state(u0, w0)
    ctx.gradient(torch.zeros(n ** 3, device="cuda"))
    ctx.get_fixed_state(u1, w1)
    ctx.close()
    assert torch.equal(u0, u1) and torch.equal(w0, w1)
