"""Which deposit runs with which launch shapes: the shapes that pm_get_tuning and pm_autotune
report are those that run, and setting a context's own shapes changes nothing.  Seen by the
launches of a density and of a VJP: two for a deposit by atomics, five for one by bins."""
import pytest

pytestmark = pytest.mark.gpu

ATOMICS, BINS = 2, 5


def context(torch, npc, nm, batch=1, precision=0):
    from paper_2211_09815_gb300 import inputs, pm
    dt = torch.float64 if precision else torch.float32
    return pm.PMContext(float(nm), nm, npc, 2, [inputs.THETA_FIDUCIAL] * batch,
                        torch.zeros(batch, npc, npc, npc, device="cuda", dtype=dt), precision=precision, batch=batch)


def deposits(torch, ctx):
    """Launches and results of the density and the pi deposit."""
    v = (ctx.batch, 3, ctx.N)
    g = torch.Generator(device="cuda").manual_seed(2)
    d = 2.0 * torch.randn(v, generator=g, device="cuda", dtype=ctx.dtype)
    p = torch.randn(v, generator=g, device="cuda", dtype=ctx.dtype)
    dens = torch.empty(ctx.batch, ctx.M, device="cuda", dtype=ctx.dtype)
    acc, alpha = torch.empty_like(d), torch.empty_like(d)
    ctx.profile()
    ctx.op_density(d, dens)
    n1 = ctx.profile_read()["scatter"][1]
    ctx.op_force_vjp(d, p, acc, alpha)
    n4 = ctx.profile_read()["scatter"][1]
    ctx.profile(False)
    return (n1, n4), (dens, acc, alpha)


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("npc,nm,batch,default", [(16, 32, 1, (ATOMICS, ATOMICS)), (16, 16, 20, (ATOMICS, BINS)),
                                                  (64, 64, 1, (ATOMICS, BINS)), (64, 128, 1, (ATOMICS, BINS)),
                                                  (64, 64, 2, (BINS, BINS))])
def test_own_shapes_keep_the_path_and_others_take_the_bins(precision, npc, nm, batch, default):
    import torch
    ctx = context(torch, npc, nm, batch, precision)
    t = ctx.get_tuning()
    n, first = deposits(torch, ctx)
    assert n == default
    ctx.set_tuning(t)
    assert ctx.get_tuning() == t
    n, again = deposits(torch, ctx)
    assert n == default and all(torch.equal(a, b) for a, b in zip(first, again))
    # one deposit's shape leaves the other's path
    ctx.set_tuning({"threads_density": 768 - t["threads_density"]})
    n, other = deposits(torch, ctx)
    assert n == (BINS, default[1]) and all(torch.equal(a, b) for a, b in zip(first, other))
    ctx.set_tuning({**t, "threads_adjoint": 768 - t["threads_adjoint"]})
    n, other = deposits(torch, ctx)
    assert n == (default[0], BINS) and all(torch.equal(a, b) for a, b in zip(first, other))
    ctx.set_tuning(t)
    assert deposits(torch, ctx)[0] == default
    ctx.close()


@pytest.mark.parametrize("npc,nm,batch", [(8, 8, 1), (16, 16, 20), (32, 32, 1), (16, 128, 1)])
def test_the_tuners_choice_is_what_runs(npc, nm, batch):
    import torch
    ctx = context(torch, npc, nm, batch)
    default = ctx.get_tuning()
    want, first = deposits(torch, ctx)
    chosen, _ = ctx.autotune(reps=5)
    assert ctx.get_tuning() == chosen
    n, out = deposits(torch, ctx)
    for k, (part, bit) in enumerate((("density", 1), ("adjoint", 2))):
        same = all(chosen[f"{f}_{part}"] == default[f"{f}_{part}"] for f in ("tile_log2", "threads"))
        atomics = same and not chosen["fused_x"] & bit and want[k] == ATOMICS
        assert n[k] == (ATOMICS if atomics else BINS)
    # 8 us against 21: the tuner finds the deposit by atomics
    if npc <= 16 and nm <= 16 and batch == 1:
        assert n[0] == ATOMICS
    assert torch.equal(first[0], out[0])
    ctx.close()


@pytest.mark.parametrize("precision,n,npc,batch", [(0, 8, 4, 1), (1, 8, 8, 2), (0, 32, 16, 3), (1, 32, 8, 2),
                                                   (0, 64, 32, 2), (0, 64, 32, 8), (0, 128, 64, 1), (1, 128, 16, 1)])
@pytest.mark.parametrize("spread", [0.0, 2.0, None])
def test_atomics_equal_the_bins(precision, n, npc, batch, spread):
    """From an even lattice to all particles in one cell: densities, accelerations, VJPs and
    gradients, bit for bit."""
    import torch
    from paper_2211_09815_gb300 import inputs, pm
    dt = torch.float64 if precision else torch.float32
    N = npc ** 3
    g = torch.Generator(device="cuda").manual_seed(n + npc)
    if spread is None:
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
            ctx.set_tuning({"threads_density": 512, "threads_adjoint": 256, "fused_x": 0})
        dens, gw = (torch.empty(batch, k, device="cuda", dtype=dt) for k in (n ** 3, N))
        a1, a2, al = (torch.empty(batch, 3, N, device="cuda", dtype=dt) for _ in range(3))
        for _ in range(2):   # the sums are left zero
            ctx.op_density(d, dens)
            ctx.op_force(d, a1)
            ctx.op_force_vjp(d, p, a2, al)
            ctx.gradient(tgt, grad_omega=gw)
        ctx.close()
        res.append((dens, a1, a2, al, gw))
    assert all(torch.equal(a, b) for a, b in zip(*res))
