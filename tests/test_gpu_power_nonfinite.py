"""A shell that holds a non-finite mode has power NaN, also where finite modes follow that one in
its run of kx."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_shells_with_a_nonfinite_mode_are_nan():
    import torch
    from paper_2211_09815_gb300 import inputs, pm
    n = 8
    ctx = pm.PMContext(50.0, n, 4, 1, [inputs.THETA_FIDUCIAL], torch.zeros(4, 4, 4, device="cuda"))
    # rows of a constant c: the x pass adds four of them at a time (finite) and gives 8 c = inf at
    # kx = 0, zeros elsewhere; the y and z passes turn those into inf at the origin and NaN (inf - inf)
    # in the rest of the plane kx = 0, and leave the others zero
    c = 6e37
    assert 4 * c < float(np.finfo(np.float32).max) < 8 * c
    mesh = torch.full((n, n, n), c, device="cuda")
    spec = torch.empty(1, n, n, n // 2 + 1, 2, device="cuda")
    ctx.op_fft(-1, mesh, spec)
    bad = ~torch.isfinite(spec[0]).all(-1)
    assert bool(bad[:, :, 0].all()) and not bool(bad[:, :, 1:].any())
    # every shell 0..3 holds modes of that plane: (0, 0), (0, 1), (0, 2), (0, 3)
    _, pk, _ = ctx.power_spectrum(mesh)
    assert np.isnan(pk).all(), pk
    # a finite mesh afterwards
    _, pk, _ = ctx.power_spectrum(torch.zeros_like(mesh))
    assert (pk == 0).all()
    ctx.close()
