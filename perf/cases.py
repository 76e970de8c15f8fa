"""What the speed of this framework is measured on: the work that its users have it do,
through its public entry points (paper_2211_09815_gb300.pm), from the smallest calls to the
largest mesh, as plain dicts that prepare() turns into a context and its inputs.

The kinds of call:
  density    PMContext.op_density: CIC overdensity of displaced particles
  force      PMContext.op_force: the PM force of one leapfrog step
  vjp        PMContext.op_force_vjp: force and its vector-Jacobian product, one adjoint step
  fft        PMContext.op_fft: real mesh -> half spectrum and half spectrum -> real mesh
  power      PMContext.loss_power: power-spectrum objective and its density cotangent
  ic         PMContext.op_ic: Zel'dovich or 2LPT initial state from white noise
  forward    PMContext.forward: initial conditions and the whole leapfrog run
  gradient   PMContext.gradient: forward, field MSE and adjoint
  graph      PMContext.gradient_graph: the same for a batch, replayed from a CUDA graph

Contexts are made with their defaults, as a user's program makes them.
"""
import math

import numpy as np
import torch

from paper_2211_09815_gb300 import pm

THETA = (2.1e-9, 0.965, 0.31, 0.049, 0.68)     # A_s, n_s, Omega_m, Omega_b, h
A0 = 1.0 / 64
L2_BYTES = 126e6
PARTICLE_KINDS = ("density", "force", "vjp")
RUN_KINDS = ("forward", "gradient", "graph")


def _case(kind, n_mesh, n_ptcl, box, **more):
    c = {"kind": kind, "n_mesh": n_mesh, "n_ptcl": n_ptcl, "box": box, "precision": "f32", "batch": 1,
         "deconv": False, "n_steps": 1, "lpt": 1, "a1": 1.0}
    c.update(more)
    return c


def listed():
    return [
        # one density for a plot or a test statistic: a latency-bound call
        _case("density", 64, 32, 100.0, name="density 32/64"),
        # a whole FP64 reference run, 10 steps to a = 1 (the smallest configuration of the benchmark)
        _case("forward", 64, 32, 100.0, precision="f64", n_steps=10, name="forward f64 32/64"),
        # the force inside someone's own integrator, at the size of quick experiments
        _case("force", 128, 64, 100.0, name="force 64/128"),
        # an ensemble of small boxes for inference: batched gradients replayed from a graph
        _case("graph", 128, 64, 400.0, batch=8, n_steps=4, a1=0.05, name="graph gradient 8x64/128"),
        # one gradient of a large-volume reconstruction over the first steps of the run
        _case("gradient", 256, 128, 800.0, n_steps=4, a1=0.05, name="gradient 128/256"),
        # the adjoint step of the batched ensemble: 16 boxes of 128^3 on 256^3 meshes
        _case("vjp", 256, 128, 200.0, batch=16, name="vjp 16x128/256"),
        # a forward and an adjoint step of the medium run, clustered as at a = 1
        _case("force", 512, 256, 400.0, name="force 256/512"),
        _case("vjp", 512, 256, 400.0, name="vjp 256/512"),
        # an adjoint step of the largest run
        _case("vjp", 1024, 512, 1000.0, name="vjp 512/1024"),
        # the transforms alone, both ways, for a user's own Fourier-space operator
        _case("fft", 512, 256, 400.0, name="fft 512"),
        # the power-spectrum objective of a fit
        _case("power", 256, 128, 200.0, name="power 256"),
        # second-order initial conditions from white noise
        _case("ic", 256, 128, 200.0, lpt=2, name="ic 2lpt 128"),
    ]


def draw(rng):
    kind = rng.choice(["density", "force", "force", "vjp", "vjp", "vjp", "fft", "power", "ic", "forward", "gradient",
                       "graph"])
    prec = "f64" if rng.random() < 0.15 else "f32"
    top = {"gradient": 8, "graph": 7, "forward": 8, "power": 9, "ic": 9}.get(kind, 10)
    if prec == "f64":
        top = min(top, 7 if kind in RUN_KINDS else 8)
    lg = rng.randint(5, top)
    if lg == 10 and rng.random() < 0.5:
        lg = 9
    n_mesh = 1 << lg
    ratio = rng.choice([1, 2, 2, 2, 4])
    if lg == 10:
        ratio = 2 if kind != "density" else rng.choice([2, 4])
    n_ptcl = n_mesh // ratio
    # no more cells than 16 meshes of 256^3, in FP64 than 4; odd batch sizes among them
    most = max(1, min(16, ((4 if prec == "f64" else 16) << 24) >> (3 * lg)) if lg < 9 else 1)
    batch = 1 if rng.random() < 0.5 else rng.randint(1, most)
    if kind in ("gradient", "graph"):
        n_ptcl = n_mesh // 2
        batch = min(batch, max(1, (8 << 24) >> (3 * lg)))
    cell = math.exp(rng.uniform(math.log(0.6), math.log(2.5)))
    c = _case(kind, n_mesh, n_ptcl, 1.0, precision=prec, batch=batch)
    if kind in ("force", "vjp"):
        c["deconv"] = rng.random() < 0.25
    if kind == "ic":
        c["lpt"] = rng.choice([1, 2])
    if kind == "forward":
        c.update(n_steps=rng.randint(2, 7), lpt=rng.choice([1, 1, 2]))
    if kind in ("gradient", "graph"):
        # early steps of a coarse box: no particle comes near a cell face, where the gradient of
        # the CIC weights jumps, so that the FP32 gradient is a continuous function of its inputs
        cell = rng.uniform(3.0, 4.0)
        c.update(n_steps=rng.randint(2, 5), a1=rng.uniform(0.03, 0.05))
    c["box"] = round(cell * n_mesh, 3)
    return c


# ------------------------------------------------------------------------- cosmology (FP64)

def _plin(k, th):
    """Linear power spectrum, Eisenstein & Hu (1998) no-wiggle; k in h/Mpc, torch FP64."""
    As, ns, Om, Ob, h = th
    omh2, fb = Om * h * h, Ob / Om
    s = 44.5 * torch.log(9.83 / omh2) / torch.sqrt(1 + 10 * (Ob * h * h) ** 0.75)
    alpha = 1 - 0.328 * torch.log(431 * omh2) * fb + 0.38 * torch.log(22.3 * omh2) * fb * fb
    gam = Om * h * (alpha + (1 - alpha) / (1 + (0.43 * k * h * s) ** 4))
    q = k * (2.7255 / 2.7) ** 2 / gam
    l0 = torch.log(2 * math.e + 1.8 * q)
    t = l0 / (l0 + (14.2 + 731 / (1 + 62.5 * q)) * q * q)
    return 2 * math.pi ** 2 / k ** 3 * 0.16 * As * (k * h / 0.05) ** (ns - 1) * t * t * (2997.92458 * k) ** 4 / Om ** 2


def _growth(a, Om):
    """D1, G_D = a^2 H dD1/dlna and G_K = 3/2 Om D1 of flat LCDM (the integral form), torch FP64."""
    x, w = np.polynomial.legendre.leggauss(64)
    x = torch.tensor(0.5 * (x + 1), dtype=torch.float64, device=Om.device)
    w = torch.tensor(0.5 * w, dtype=torch.float64, device=Om.device)
    E2 = Om * a ** -3 + 1 - Om
    y = a * x * x                                   # a' = a x^2
    f = 2 * a * x * y ** 1.5 / (Om + (1 - Om) * y ** 3) ** 1.5
    d1 = 2.5 * Om * torch.sqrt(E2) * (f * w).sum()
    dd1 = -1.5 * Om * a ** -3 / E2 * d1 + 2.5 * Om / (a * a * E2)
    return d1, a * a * torch.sqrt(E2) * dd1, 1.5 * Om * d1


def _growth2(a, Om):
    """D2 and G_D2 = a^2 H dD2/dlna of second-order LPT: RK4 in ln a from a = 1e-4, floats."""
    def rhs(x, y):
        h2 = Om * math.exp(-3 * x) + 1 - Om
        om = Om * math.exp(-3 * x) / h2
        e = -1.5 * om
        return np.array([y[1], -(4 + e) * y[1] - (3 + e - 1.5 * om) * y[0],
                         y[3], -(6 + e) * y[3] - (8 + 2 * e - 1.5 * om) * y[2] + 1.5 * om * y[0] ** 2])
    y, x, n = np.array([1.0, 0.0, 3 / 7, 0.0]), math.log(1e-4), 4000
    h = (math.log(a) - x) / n
    for _ in range(n):
        k1 = rhs(x, y)
        k2 = rhs(x + h / 2, y + h / 2 * k1)
        k3 = rhs(x + h / 2, y + h / 2 * k2)
        k4 = rhs(x + h, y + h * k3)
        y, x = y + h / 6 * (k1 + 2 * k2 + 2 * k3 + k4), x + h
    return a * a * y[2], a * a * math.sqrt(Om * a ** -3 + 1 - Om) * a * a * (2 * y[2] + y[3])


def _modes(n, dtype=torch.float64):
    f = torch.fft.fftfreq(n, 1.0 / n, dtype=dtype, device="cuda")
    return f.view(n, 1, 1), f.view(1, n, 1), torch.arange(n // 2 + 1, dtype=dtype, device="cuda").view(1, 1, -1)


def _derivs(n, box, dtype=torch.float64):
    """k_c with its Nyquist plane zeroed, for c = 0..2, and k^2 with 1 at k = 0."""
    kf, m = 2 * math.pi / box, _modes(n, dtype)
    k2 = (m[0] ** 2 + m[1] ** 2 + m[2] ** 2) * kf ** 2
    k2[0, 0, 0] = 1
    return [torch.where(v.abs() == n // 2, torch.zeros_like(v), v) * kf for v in m], k2


def _amplitude(n, box, th, k2):
    a = torch.sqrt(_plin(torch.sqrt(k2.double()), th) / (box / n) ** 3)
    zero = torch.zeros_like(a)
    zero[0, 0, 0] = 1
    return a * (1 - zero)


def _theta(values):
    return [torch.tensor(float(v), dtype=torch.float64, device="cuda") for v in values]


def _irfftn(x, n):
    return torch.fft.irfftn(x, s=(n, n, n))


# ------------------------------------------------------------------------- inputs

def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _gaussian_displacement(n, box, gen, dtype):
    """First-order displacement at a = 1 (growth 0.78) of a random field, [3][n^3]."""
    ks, k2 = _derivs(n, box, torch.float32)
    amp = (0.78 * _amplitude(n, box, _theta(THETA), k2) / k2).float()
    wk = torch.fft.rfftn(torch.randn((n, n, n), generator=gen, device="cuda")) * amp
    out = torch.empty((3, n ** 3), dtype=dtype, device="cuda")
    for c in range(3):
        out[c] = _irfftn(wk * (1j * ks[c]), n).reshape(-1)
    return out


def _displacement(case, gen, dtype):
    """Displacements as a run holds them at a = 1: a linear flow in which the matter of one
    in eight regions of 4 Mpc/h has fallen into its middle (haloes)."""
    n, box, nm = case["n_ptcl"], case["box"], case["n_mesh"]
    cell = box / nm
    out = []
    for _ in range(case["batch"]):
        s = _gaussian_displacement(n, box, gen, torch.float32)
        x = torch.arange(n, device="cuda", dtype=torch.float32) * (box / n) + 0.5 * cell
        q = (x.view(n, 1, 1), x.view(1, n, 1), x.view(1, 1, n))
        nr = max(1, round(box / 4.0))
        r = box / nr
        idx, mid = None, []
        for c in range(3):
            p = q[c] + s[c].view(n, n, n)
            i = torch.floor(p / r)
            mid.append((i + 0.5) * r - p)
            j = torch.remainder(i, nr).to(torch.int64)
            idx = j if idx is None else idx * nr + j
        fallen = (torch.rand(nr ** 3, generator=gen, device="cuda") < 0.125).float()[idx] * 0.85
        for c in range(3):
            s[c] += (fallen * mid[c]).view(-1)
        # no particle on a cell face: the gradient of the CIC weights jumps there
        v = s / cell + 0.5
        f = torch.floor(v)
        s = (f + (v - f).clamp(2.0 ** -12, 1 - 2.0 ** -12) - 0.5) * cell
        out.append(s)
    return torch.stack(out).to(dtype)


def _thetas(case, gen):
    rows = [list(THETA)]
    for _ in range(case["batch"] - 1):
        u = torch.rand(3, generator=gen, device="cuda").tolist()
        rows.append([(1.8 + 0.6 * u[0]) * 1e-9, 0.94 + 0.05 * u[1], 0.25 + 0.10 * u[2], 0.049, 0.68])
    return rows


def _inputs(case, seed):
    """The tensors and numbers of a case, from the seed alone."""
    gen, B, nm, n = _generator(seed), case["batch"], case["n_mesh"], case["n_ptcl"]
    dtype = torch.float32 if case["precision"] == "f32" else torch.float64
    d = {"theta": _thetas(case, gen)}
    kind = case["kind"]
    if kind in PARTICLE_KINDS:
        d["disp"] = _displacement(case, gen, dtype)
        if kind == "vjp":
            # the adjoint momentum: a large-scale flow and small-scale noise
            d["pi"] = torch.stack([1e-4 * _gaussian_displacement(n, case["box"], gen, dtype)
                                   for _ in range(B)])
            d["pi"] += 1e-4 * torch.randn(d["pi"].shape, generator=gen, device="cuda", dtype=torch.float32)
    elif kind == "fft":
        d["real"] = torch.randn((B, nm, nm, nm), generator=gen, device="cuda", dtype=dtype)
        d["spec"] = torch.fft.rfftn(torch.randn((B, nm, nm, nm), generator=gen, device="cuda", dtype=dtype),
                                    dim=(1, 2, 3)).contiguous() * nm ** -1.5
    elif kind == "power":
        # a log-normal-like density, as a run's final one
        x = []
        k2 = _derivs(nm, case["box"], torch.float32)[1]
        amp = (0.78 * _amplitude(nm, case["box"], _theta(THETA), k2)).float() * torch.exp(-0.5 * k2)
        for _ in range(B):
            g = _irfftn(torch.fft.rfftn(torch.randn((nm,) * 3, generator=gen, device="cuda")) * amp, nm)
            x.append(torch.exp(g - 0.5 * g.var()) - 1)
        d["dens"] = torch.stack(x).to(dtype)
        u = torch.rand((2, B, nm // 2), generator=gen, device="cuda", dtype=torch.float64).cpu().numpy()
        d["target"], d["weights"] = 500.0 + 1000.0 * u[0], 1e-6 * (0.5 + u[1])
    if kind in RUN_KINDS or kind == "ic":
        d["omega"] = torch.randn((B, n, n, n), generator=gen, device="cuda", dtype=dtype)
    if kind in ("gradient", "graph"):
        d["target"] = 0.1 * torch.randn((B, nm ** 3), generator=gen, device="cuda", dtype=dtype)
    return d


def prepare(case, seed):
    B, nm, n = case["batch"], case["n_mesh"], case["n_ptcl"]
    dtype = torch.float32 if case["precision"] == "f32" else torch.float64
    d = _inputs(case, seed)
    stream = torch.cuda.Stream() if case["kind"] == "graph" else None    # a graph wants a stream of its own
    if stream is not None:
        stream.wait_stream(torch.cuda.current_stream())
    omega = d["omega"] if "omega" in d else torch.zeros((B, n, n, n), device="cuda", dtype=dtype)
    if stream is not None:
        torch.cuda.current_stream().synchronize()
    ctx = pm.PMContext(case["box"], nm, n, case["n_steps"], d["theta"], omega, a0=A0, a1=case["a1"],
                       precision=pm.PM_F32 if case["precision"] == "f32" else pm.PM_F64, deconv=case["deconv"],
                       batch=B, lpt_order=case["lpt"], stream=stream)

    def new(*shape, dtype=dtype):
        return torch.empty(shape, device="cuda", dtype=dtype)

    st = {"kind": case["kind"], "ctx": ctx, "f32": case["precision"] == "f32", **d}
    kind = case["kind"]
    if kind == "density":
        st["out"] = [new(B, nm ** 3)]
    elif kind == "force":
        st["out"] = [new(B, 3, n ** 3)]
    elif kind == "vjp":
        st["out"] = [new(B, 3, n ** 3), new(B, 3, n ** 3)]
    elif kind == "fft":
        st["out"] = [new(*d["spec"].shape, dtype=d["spec"].dtype), new(*d["real"].shape)]
        st["flat"] = [torch.view_as_real(v) for v in (d["spec"], st["out"][0])]
    elif kind == "power":
        st["out"] = [new(B, nm ** 3)]
    elif kind == "ic":
        st["out"] = [new(B, 3, n ** 3), new(B, 3, n ** 3)]
    elif kind == "forward":
        st["out"] = [new(B, 3, n ** 3), new(B, 3, n ** 3), new(B, nm ** 3)]
    else:
        st["out"] = [new(B, dtype=torch.float64), new(B, n ** 3), new(B, 5, dtype=torch.float64)]
    return st


def run(state):
    ctx, out, kind = state["ctx"], state["out"], state["kind"]
    if kind == "density":
        ctx.op_density(state["disp"], out[0])
    elif kind == "force":
        ctx.op_force(state["disp"], out[0])
    elif kind == "vjp":
        ctx.op_force_vjp(state["disp"], state["pi"], out[0], out[1])
    elif kind == "fft":
        ctx.op_fft(-1, state["real"], state["flat"][1])
        ctx.op_fft(+1, state["flat"][0], out[1])
    elif kind == "power":
        loss = ctx.loss_power(state["target"], state["weights"], out[0], dens=state["dens"])
        return [loss.astype(np.float32) if state["f32"] else loss, out[0]]
    elif kind == "ic":
        ctx.op_ic(out[0], out[1])
    elif kind == "forward":
        ctx.forward(disp=out[0], mom=out[1], dens=out[2])
    elif kind == "gradient":
        ctx.gradient(state["target"], omega=state["omega"], loss=out[0], grad_omega=out[1], grad_theta=out[2])
    else:
        ctx.gradient_graph(state["target"], loss=out[0], grad_omega=out[1], grad_theta=out[2])
        torch.cuda.current_stream().wait_stream(ctx.stream)
    if kind in ("gradient", "graph") and state["f32"]:
        # the FP64 sums of an FP32 run are as accurate as the FP32 fields they are summed from
        return [out[0].float(), out[1], out[2].float()]
    return out


def work(case):
    B, nm, n = case["batch"], case["n_mesh"], case["n_ptcl"]
    e = 4 if case["precision"] == "f32" else 8
    N, M = B * n ** 3, B * nm ** 3

    def transforms(count, cells):
        # a transform of a mesh that no cache holds reads it once and writes it once
        side = round((cells / B) ** (1 / 3))
        return {"bytes": 2.0 * e * cells * count if e * cells > L2_BYTES else 0.0,
                "flops": 2.5 * count * cells * 3 * math.log2(side)}
    kind = case["kind"]
    if kind == "density":
        return {"bytes": e * (3 * N + M), "flops": 40 * N}
    if kind == "fft":
        return {"bytes": 4 * e * M, "flops": transforms(2, M)["flops"]}
    if kind == "power":
        t = transforms(2, M)
        return {"bytes": max(2 * e * M, t["bytes"]), "flops": t["flops"] + 12 * M}
    if kind == "ic":
        t = transforms(4 if case["lpt"] == 1 else 14, N)
        return {"bytes": t["bytes"] + e * 7 * N, "flops": t["flops"] + 30 * N}
    f, v = transforms(4, M), transforms(8, M)
    force = {"bytes": f["bytes"] + e * 6 * N, "flops": f["flops"] + 110 * N}
    vjp = {"bytes": v["bytes"] + e * 12 * N, "flops": v["flops"] + 330 * N}
    if kind == "force":
        return force
    if kind == "vjp":
        return vjp
    steps = case["n_steps"] + 1
    if kind == "forward":
        return {"bytes": f["bytes"] * steps + e * (7 * N + M), "flops": force["flops"] * steps}
    return {"bytes": (f["bytes"] + v["bytes"]) * steps + e * (2 * N + M),
            "flops": (force["flops"] + vjp["flops"]) * steps}


# ------------------------------------------------------------------------- exact results (torch, FP64)

def _corners(s, n, nm, box):
    """(flat node index, weight, weight gradient of each axis) of the 8 CIC corners of the
    particles q + s, s [3][n^3]."""
    l = box / nm
    j = torch.arange(n, device="cuda", dtype=torch.int64) * (nm // n)
    grid = (j.view(n, 1, 1), j.view(1, n, 1), j.view(1, 1, n))
    t, cell = [], []
    for c in range(3):
        v = s[c] / l + 0.5
        f = torch.floor(v.detach())
        t.append(v - f)
        cell.append((grid[c].expand(n, n, n).reshape(-1) + f.to(torch.int64)) % nm)
    for d in range(8):
        b = ((d >> 2) & 1, (d >> 1) & 1, d & 1)
        w = [t[c] if b[c] else 1 - t[c] for c in range(3)]
        sg = [(1.0 if b[c] else -1.0) / l for c in range(3)]
        i = [(cell[c] + b[c]) % nm for c in range(3)]
        yield (i[0] * nm + i[1]) * nm + i[2], w, sg


def _scatter(s, values, n, nm, box):
    m = torch.zeros(nm ** 3, dtype=torch.float64, device="cuda")
    for idx, w, _ in _corners(s, n, nm, box):
        m = m.index_add(0, idx, w[0] * w[1] * w[2] if values is None else w[0] * w[1] * w[2] * values) \
            if torch.is_grad_enabled() else m.index_add_(0, idx, w[0] * w[1] * w[2] if values is None else
                                                         w[0] * w[1] * w[2] * values)
    return m.view(nm, nm, nm)


def _green(nm, box, Om, deconv):
    ks, k2 = _derivs(nm, box)
    g = -1.5 * Om / k2
    if deconv:
        for v in _modes(nm):
            g = g / torch.sinc(v / nm) ** 4
    first = torch.ones_like(k2)
    first[0, 0, 0] = 0
    return ks, g * first


def _delta(s, n, nm, box):
    return (nm / n) ** 3 * _scatter(s, None, n, nm, box) - 1


def _force(s, n, nm, box, Om, deconv=False):
    """Accelerations at the particles q + s."""
    ks, g = _green(nm, box, Om, deconv)
    dk = torch.fft.rfftn(_delta(s, n, nm, box)) * g
    f = [_irfftn(dk * (-1j * ks[c]), nm).reshape(-1) for c in range(3)]
    a = [0, 0, 0]
    for idx, w, _ in _corners(s, n, nm, box):
        ww = w[0] * w[1] * w[2]
        for c in range(3):
            a[c] = a[c] + ww * f[c][idx]
    return torch.stack(a)


def _force_vjp(s, pi, n, nm, box, Om, deconv):
    ks, g = _green(nm, box, Om, deconv)
    acc = None
    for c in range(3):
        t = torch.fft.rfftn(_scatter(s, pi[c], n, nm, box)).mul_(1j * ks[c])
        acc = t if acc is None else acc.add_(t)
        del t
    psi = (_irfftn(acc.mul_(g), nm) * (nm / n) ** 3).reshape(-1)
    del acc
    dk = torch.fft.rfftn(_delta(s, n, nm, box)).mul_(g)
    del g
    f = [_irfftn(dk * (-1j * ks[c]), nm).reshape(-1) for c in range(3)]
    del dk
    a, al = torch.zeros_like(s), torch.zeros_like(s)
    for idx, w, sg in _corners(s, n, nm, box):
        h = psi[idx]
        for c in range(3):
            fc = f[c][idx]
            a[c] += w[0] * w[1] * w[2] * fc
            h += pi[c] * fc
        al[0] += sg[0] * w[1] * w[2] * h
        al[1] += w[0] * sg[1] * w[2] * h
        al[2] += w[0] * w[1] * sg[2] * h
    return a, al


def _initial(omega, th, n, box, lpt):
    ks, k2 = _derivs(n, box)
    dk = torch.fft.rfftn(omega) * _amplitude(n, box, th, k2)
    s1 = torch.stack([_irfftn(1j * ks[c] / k2 * dk, n).reshape(-1) for c in range(3)])
    d1, gd, _ = _growth(A0, th[2])
    s, p = d1 * s1, gd * s1
    if lpt == 2:
        h = {(i, j): _irfftn(ks[i] * ks[j] / k2 * dk, n) for i in range(3) for j in range(i, 3)}
        src = sum(h[i, i] * h[j, j] - h[i, j] ** 2 for i, j in ((0, 1), (0, 2), (1, 2)))
        sk = torch.fft.rfftn(src)
        s2 = torch.stack([_irfftn(1j * ks[c] / k2 * sk, n).reshape(-1) for c in range(3)])
        d2, gd2 = _growth2(A0, float(th[2]))
        s, p = s + d2 * s2, p + gd2 * s2
    return s, p


def _simulate(case, omega, th):
    """Final displacement, momentum and overdensity of one instance."""
    n, nm, box, steps = case["n_ptcl"], case["n_mesh"], case["box"], case["n_steps"]
    s, p = _initial(omega, th, n, box, case["lpt"])
    a = [A0 + (case["a1"] - A0) * i / steps for i in range(steps + 1)]
    g = [_growth(v, th[2]) for v in a]
    acc = _force(s, n, nm, box, th[2], case["deconv"])
    for i in range(steps):
        _, gdh, _ = _growth(0.5 * (a[i] + a[i + 1]), th[2])
        p = p + acc * (gdh - g[i][1]) / g[i][2]
        s = s + p * (g[i + 1][0] - g[i][0]) / gdh
        acc = _force(s, n, nm, box, th[2], case["deconv"])
        p = p + acc * (g[i + 1][1] - gdh) / g[i + 1][2]
    return s, p, _delta(s, n, nm, box).reshape(-1)


def _power_loss(d, tgt, w, nm, box):
    m = _modes(nm)
    b = torch.floor(torch.sqrt(m[0] ** 2 + m[1] ** 2 + m[2] ** 2)).to(torch.int64)
    mult = torch.full((1, 1, nm // 2 + 1), 2.0, dtype=torch.float64, device="cuda")
    mult[..., 0] = mult[..., -1] = 1.0
    nb, dk = nm // 2, torch.fft.rfftn(d)
    size = int(b.max()) + 1
    flat, mult = b.reshape(-1), mult.expand(nm, nm, -1).reshape(-1)
    cnt = torch.zeros(size, dtype=torch.float64, device="cuda").index_add_(0, flat, mult)
    pw = torch.zeros(size, dtype=torch.float64, device="cuda").index_add_(0, flat, mult * dk.abs().square().reshape(-1))
    vol = box ** 3 / float(nm) ** 6
    diff = vol * pw[:nb] / cnt[:nb] - tgt
    g = torch.zeros(size, dtype=torch.float64, device="cuda")
    g[:nb] = 4 * w * diff * vol / cnt[:nb]
    return (w * diff ** 2).sum(), _irfftn(dk * g[b], nm) * nm ** 3


def exact(case, seed):
    d = _inputs(case, seed)
    B, nm, n, box, kind = case["batch"], case["n_mesh"], case["n_ptcl"], case["box"], case["kind"]
    if kind == "fft":
        return [torch.fft.rfftn(d["real"].double(), dim=(1, 2, 3)),
                torch.fft.irfftn(d["spec"].to(torch.complex128), s=(nm,) * 3, dim=(1, 2, 3)) * float(nm) ** 3]
    rows = []
    for b in range(B):
        th = _theta(d["theta"][b])
        if kind == "density":
            rows.append([_delta(d["disp"][b].double(), n, nm, box).reshape(-1)])
        elif kind == "force":
            with torch.no_grad():
                rows.append([_force(d["disp"][b].double(), n, nm, box, th[2], case["deconv"])])
        elif kind == "vjp":
            with torch.no_grad():
                rows.append(_force_vjp(d["disp"][b].double(), d["pi"][b].double(), n, nm, box, th[2],
                                       case["deconv"]))
        elif kind == "power":
            t, w = (torch.from_numpy(d[k][b]).cuda() for k in ("target", "weights"))
            loss, g = _power_loss(d["dens"][b].double(), t, w, nm, box)
            rows.append([loss, g.reshape(-1)])
        elif kind == "ic":
            rows.append(_initial(d["omega"][b].double(), th, n, box, case["lpt"]))
        elif kind == "forward":
            with torch.no_grad():
                rows.append(_simulate(case, d["omega"][b].double(), th))
        else:
            om = d["omega"][b].double().requires_grad_(True)
            th = [v.requires_grad_(True) for v in th]
            delta = _simulate(case, om, th)[2]
            loss = (delta - d["target"][b].double()).square().mean()
            loss.backward()
            rows.append([loss.detach(), om.grad.reshape(-1), torch.stack([v.grad for v in th])])
    return [torch.stack([r[i] for r in rows]) for i in range(len(rows[0]))]
