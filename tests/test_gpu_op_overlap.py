"""Operators whose outputs overlap their inputs, wholly or in part: the results are those of
separate buffers."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1])
def test_outputs_over_inputs(precision):
    import ctypes
    import torch
    from paper_2211_09815_gb300 import inputs, pm
    dt = torch.float64 if precision else torch.float32
    n, npc = 32, 16
    v = 3 * npc ** 3
    g = torch.Generator(device="cuda").manual_seed(3)
    d = 2.0 * torch.randn(v, generator=g, device="cuda", dtype=dt)
    p = torch.randn(v, generator=g, device="cuda", dtype=dt)
    ctx = pm.PMContext(50.0, n, npc, 1, [inputs.THETA_FIDUCIAL], torch.zeros(npc, npc, npc, device="cuda", dtype=dt),
                       precision=precision)
    acc, acc2, alpha = (torch.empty(v, device="cuda", dtype=dt) for _ in range(3))
    ctx.op_force(d, acc)
    ctx.op_force_vjp(d, p, acc2, alpha)
    assert torch.equal(acc, acc2)
    # in place
    x = d.clone()
    ctx.op_force(x, x)
    assert torch.equal(x, acc)
    x, q = d.clone(), p.clone()
    ctx.op_force_vjp(x, q, q, x)
    assert torch.equal(q, acc) and torch.equal(x, alpha)
    # in part: inputs and outputs of one buffer, shifted by less than their length
    buf = torch.empty(2 * v, device="cuda", dtype=dt)
    for shift in (1, 1000, v - 1):
        buf[:v] = d
        ctx.op_force(buf[:v], buf[shift:shift + v])
        assert torch.equal(buf[shift:shift + v], acc)
    wide = torch.empty(n ** 3, device="cuda", dtype=dt)
    dens = torch.empty(n ** 3, device="cuda", dtype=dt)
    ctx.op_density(d, dens)
    wide[100:100 + v] = d
    ctx.op_density(wide[100:100 + v], wide)
    assert torch.equal(wide, dens)
    ctx.close()
