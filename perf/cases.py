"""Performance cases: the work that users of the library have it do.

A case is a dict of plain values.  `listed()` names the standing ones, `draw()`
gives more of the same ranges, `prepare()` makes what a program has in hand
before the call (the context, f, the field, a network), `run()` is one pass
through the public calls, `work()` what the pass cannot do without, and
`exact()` the same result from plain torch in 64 bits.

Initial states are the library's own analytic ones (Landau, two-stream,
self-gravitating slab, Plummer, uniform sphere, the sine of the advection
test), made here in torch with seeded amplitudes and phases.  A pass advances
the state, so repeated passes are the following steps of the run.
"""
import math

import numpy as np
import torch

KINDS = ("step1d", "sweeps1d", "step2d", "step3d", "sweeps3d", "rk", "ensemble", "learned", "train", "samples",
         "unsplit")


def listed():
    return [
        # the smallest call: one step of linear Landau damping in FP64, where latency is all there is
        dict(name="landau_64x128_f64", kind="step", profile="landau", nx="64", nv="128", precision="f64", order=5,
             scheme="sl", steps=1, dt=0.1, diag=False),
        # a nonlinear 1D1V run with the diagnostics of every step, as growth and damping rates are measured
        dict(name="two_stream_256x1024", kind="step", profile="two_stream", nx="256", nv="1024", precision="f32",
             order=7, scheme="sl", steps=10, dt=0.05, diag=True),
        # a run whose time step changes from step to step (here the convergence study in FP64): sweep by sweep
        dict(name="slab_512_f64_sweeps", kind="sweeps", profile="slab", nx="512", nv="512", precision="f64", order=7,
             dt=0.2 / 512, diag=False),
        # the fine 2D2V grid that training data and reference runs come from
        dict(name="landau2d_64x128", kind="step", profile="landau", nx="64x64", nv="128x128", precision="f32",
             order=7, scheme="sl", steps=1, dt=0.1, diag=False),
        # the largest: the self-gravitating 3D3V sphere of the benchmark
        dict(name="plummer_32x64", kind="step", profile="plummer", nx="32x32x32", nv="64x64x64", precision="f32",
             order=7, scheme="sl", steps=1, dt=0.05, diag=False),
        # the collapse of a uniform sphere with changing time step, odd sizes, energies monitored every step
        dict(name="sphere_ragged_sweeps", kind="sweeps", profile="sphere", nx="22x20x23", nv="31x33x30",
             precision="f32", order=7, dt=0.015, diag=True),
        # the Runge-Kutta scheme that the semi-Lagrangian one is compared with
        dict(name="rk_plummer_16x32", kind="step", profile="plummer", nx="16x16x16", nv="32x32x32", precision="f32",
             order=5, scheme="rk", steps=1, dt=0.025, diag=False),
        # a parameter study: 512 uneven 1D1V runs and 8 2D2V runs advanced together
        dict(name="ensemble_512_8", kind="ensemble", n1d=512, n2d=8, steps=1, dt=0.05),
        # a run on the coarse velocity grid with the learned correction
        dict(name="learned_64x32", kind="learned", nx="64x64", nv="32x32", steps=1, dt=0.1),
        # one training step of the correction network on a minibatch of cell pairs
        dict(name="train_32768", kind="train", pairs=16384),
        # training pairs of one spatial sweep: fine fluxes, restriction, features and targets
        dict(name="samples_64x128", kind="samples", nx="64x64", nv="128x128", dim=0, dt=0.1),
        # unsplit advection in two dimensions at the small CFL number it is used with
        dict(name="unsplit_4096", kind="unsplit", n1=4096, n2=4096, nv=1, steps=2, cfl=0.02),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _sizes(rng, dims, lo, hi):
    return "x".join(str(_log(rng, lo, hi)) for _ in range(dims))


def _shrink(nx, nv, most):
    """Halve the longest axis until the grid has at most `most` cells."""
    n = [int(k) for k in nx.split("x")] + [int(k) for k in nv.split("x")]
    d = len(n) // 2
    while np.prod(np.array(n, dtype=float)) > most:
        k = n.index(max(n))
        n[k] = (n[k] + 1) // 2
    return "x".join(map(str, n[:d])), "x".join(map(str, n[d:]))


def draw(rng):
    kind = rng.choice(KINDS)
    if kind == "step1d":
        profile, f64 = rng.choice(["landau", "two_stream"]), rng.random() < 0.4
        nx, nv = _shrink(str(_log(rng, 32, 1024)), str(_log(rng, 64, 2048)), 3e5 if f64 else 2e6)
        return dict(kind="step", profile=profile, nx=nx, nv=nv, precision="f64" if f64 else "f32",
                    order=rng.choice([5, 7]), scheme="sl", steps=rng.randint(1, 20), dt=round(rng.uniform(0.03, 0.12), 4),
                    diag=rng.random() < 0.5)
    if kind == "sweeps1d":
        n = _log(rng, 64, 1024)
        return dict(kind="sweeps", profile="slab", nx=str(n), nv=str(n), precision=rng.choice(["f32", "f64"]), order=7,
                    dt=0.2 / n, diag=False)
    if kind == "step2d":
        nx, nv = _shrink(_sizes(rng, 2, 16, 96), _sizes(rng, 2, 16, 128), 6e7)
        return dict(kind="step", profile="landau", nx=nx, nv=nv, precision="f32", order=rng.choice([5, 7]), scheme="sl",
                    steps=rng.randint(1, 3), dt=round(rng.uniform(0.05, 0.15), 4), diag=False)
    if kind == "step3d":
        nx, nv = _shrink(_sizes(rng, 3, 8, 40), _sizes(rng, 3, 12, 72), 2e8)
        return dict(kind="step", profile=rng.choice(["plummer", "sphere"]), nx=nx, nv=nv, precision="f32", order=7,
                    scheme="sl", steps=1, dt=round(rng.uniform(0.02, 0.06), 4), diag=False)
    if kind == "sweeps3d":
        nx, nv = _shrink(_sizes(rng, 3, 8, 48), _sizes(rng, 3, 12, 48), 2e8)
        return dict(kind="sweeps", profile=rng.choice(["plummer", "sphere"]), nx=nx, nv=nv, precision="f32", order=7,
                    dt=round(rng.uniform(0.01, 0.03), 4), diag=rng.random() < 0.5)
    if kind == "rk":
        nx, nv = _shrink(_sizes(rng, 3, 8, 24), _sizes(rng, 3, 12, 48), 1e8)
        return dict(kind="step", profile="plummer", nx=nx, nv=nv, precision="f32", order=5, scheme="rk", steps=1,
                    dt=round(rng.uniform(0.01, 0.025), 4), diag=False)
    if kind == "ensemble":
        return dict(kind="ensemble", n1d=_log(rng, 12, 512), n2d=rng.randint(0, 8), steps=rng.randint(1, 4),
                    dt=round(rng.uniform(0.03, 0.1), 4))
    if kind == "learned":
        nx, nv = _shrink(_sizes(rng, 2, 16, 80), _sizes(rng, 2, 8, 40), 8e6)
        return dict(kind="learned", nx=nx, nv=nv, steps=rng.randint(1, 3), dt=round(rng.uniform(0.05, 0.12), 4))
    if kind == "train":
        return dict(kind="train", pairs=_log(rng, 512, 1 << 20))
    if kind == "samples":
        nx = _sizes(rng, 2, 16, 64)
        nv = "x".join(str(4 * _log(rng, 6, 32)) for _ in range(2))
        return dict(kind="samples", nx=nx, nv=nv, dim=rng.randint(0, 1), dt=round(rng.uniform(0.05, 0.12), 4))
    return dict(kind="unsplit", n1=_log(rng, 128, 4096), n2=_log(rng, 128, 4096), nv=rng.choice([1, 1, 2]),
                steps=rng.randint(1, 4), cfl=0.02)


# ---- grids and states ---------------------------------------------------------------

def _ints(s):
    return [int(k) for k in s.split("x")]


def _grid(case):
    """Grid of a step or sweep case, as the keyword arguments of Simulation."""
    nx, nv = _ints(case["nx"]), _ints(case["nv"])
    D = len(nx)
    g = dict(dims=D, nx=nx, nv=nv, order=case.get("order", 7), mp=1, pp=1, alpha=4.0, xbc=0, poisson=0, pois_order=6,
             coupling=-1.0, rho_bg=1.0, scheme=1 if case.get("scheme") == "rk" else 0)
    p = case.get("profile", "landau")
    if p in ("landau", "two_stream"):
        v = 8.0 if p == "two_stream" else 6.0
        g.update(xlo=[0.0] * D, xhi=[4.0 * math.pi] * D, vlo=[-v] * D, vhi=[v] * D)
    elif p == "slab":
        g.update(xlo=[0.0], xhi=[1.0], vlo=[-1.0], vhi=[1.0], coupling=4.0 * math.pi)
    else:  # isolated: cubic cells, the longest axis spans the box
        half, v = (4.0, 1.5) if p == "plummer" else (3.0, 3.0)
        h = 2.0 * half / max(nx)
        g.update(xlo=[-0.5 * h * n for n in nx], xhi=[0.5 * h * n for n in nx], vlo=[-v] * D, vhi=[v] * D, xbc=1,
                 poisson=1, coupling=4.0 * math.pi, rho_bg=0.0)
    return g


def _axis(lo, hi, n, device):
    return lo + (torch.arange(n, dtype=torch.float64, device=device) + 0.5) * ((hi - lo) / n)


def _along(x, axis, dims):
    """x along one of `dims` axes, broadcastable over the others."""
    return x.view([-1 if k == axis else 1 for k in range(dims)])


def _fill(case, g, seed, out, dtype):
    """The initial state into `out` (a flat array), a block of x_1 rows at a time."""
    r = np.random.default_rng(seed)
    D, p, dev = g["dims"], case.get("profile", "landau"), out.device
    amp, phase = r.uniform(0.8, 1.2), r.uniform(0.0, 2.0 * math.pi, size=3)
    a = r.uniform(0.9, 1.1)
    xs = [_axis(g["xlo"][d], g["xhi"][d], g["nx"][d], dev) for d in range(D)]
    vs = [_axis(g["vlo"][d], g["vhi"][d], g["nv"][d], dev) for d in range(D)]
    if p in ("landau", "two_stream", "slab"):
        alpha = amp * {"landau": 0.01 if D == 1 and g["order"] == 5 else 0.05, "two_stream": 0.05, "slab": 0.01}[p]
        k = 4.0 * math.pi if p == "slab" else 0.5
        sigma = 0.5 * math.sqrt(4.0 * math.pi) / k if p == "slab" else 1.0
        m = [torch.exp(-v * v / (2.0 * sigma * sigma)) / math.sqrt(2.0 * math.pi * sigma * sigma) for v in vs]
        if p == "two_stream":
            m[0] = m[0] * vs[0] * vs[0]
        fv = m[0] if D == 1 else (m[0][:, None] * m[1]).reshape(-1)
        s = torch.ones([1] * D, dtype=torch.float64, device=dev)
        for d in range(D):
            s = s + alpha * torch.cos(k * _along(xs[d], d, D) + float(phase[d]))
        s = s.reshape(-1)
        rows = max(1, (1 << 24) // fv.numel())
        for i in range(0, s.numel(), rows):
            b = (s[i:i + rows, None] * fv).to(dtype).reshape(-1)
            out[i * fv.numel():i * fv.numel() + b.numel()] = b
        return
    v2 = sum(_along(v * v, d, 3) for d, v in enumerate(vs)).reshape(-1)
    x2 = sum(_along((x - 0.1 * float(phase[d] / math.pi - 1.0)) ** 2, d, 3) for d, x in enumerate(xs)).reshape(-1)
    rows = max(1, (1 << 25) // v2.numel())
    for i in range(0, x2.numel(), rows):
        xx = x2[i:i + rows, None]
        if p == "plummer":
            e = 1.0 / torch.sqrt(xx + a * a) - 0.5 * v2
            b = 24.0 * math.sqrt(2.0) * a * a / (7.0 * math.pi ** 3) * torch.clamp(e, min=0.0) ** 3.5
        else:
            s2 = amp / (20.0 * a)
            rho = amp / (4.0 * math.pi * 8.0 * a ** 3 / 3.0)
            b = torch.where(xx < 4.0 * a * a, rho * torch.exp(-v2 / (2.0 * s2)) / (2.0 * math.pi * s2) ** 1.5, 0.0)
        b = b.to(dtype).reshape(-1)
        out[i * v2.numel():i * v2.numel() + b.numel()] = b


_STREAM = []


def _stream():
    """The program's one stream (the library's step graphs need one of their own)."""
    if not _STREAM:
        _STREAM.append(torch.cuda.Stream())
    return _STREAM[0]


def _sim(case, g, seed):
    from paper_1702_08521_gb300 import vlasov as V
    f64 = case.get("precision", "f32") == "f64"
    sim = V.Simulation(g, precision=V.VP_F64 if f64 else V.VP_F32, stream=_stream())
    _fill(case, g, seed, sim.f, torch.float64 if f64 else torch.float32)
    torch.cuda.synchronize()
    sim.field()
    sim.sync()
    return sim


# ---- network and ensemble inputs -----------------------------------------------------

def _network(seed, last, device):
    """A network of the library's layout: He weights, small biases, the last layer
    scaled to corrections of a trained network's size."""
    r = np.random.default_rng([seed, 7])
    parts = []
    for rows, cols, scale in ((32, 25, 1.0), (32, 32, 1.0), (32, 32, 1.0), (1, 32, last)):
        parts += [r.standard_normal(rows * cols) * math.sqrt(2.0 / cols) * scale, r.standard_normal(rows) * 0.02 * scale]
    return torch.tensor(np.concatenate(parts), dtype=torch.float32, device=device)


def _batch(case, seed, device):
    """Feature rows as the sampler makes them: stencil differences with a zero at the
    upwind cell, velocity differences and curvatures, the CFL number; small targets;
    the two interfaces' coefficients of a cell pair."""
    n = 2 * case["pairs"]
    gen = torch.Generator(device=device)
    gen.manual_seed(seed)
    X = torch.randn(n, 25, generator=gen, device=device) * 0.3
    X[:, 3] = 0.0
    X[:, 16:24] *= 0.2
    X[:, 24] = torch.rand(n, generator=gen, device=device) * 0.5
    y = torch.randn(n, generator=gen, device=device) * 0.02
    c = 0.7 + 0.3 * torch.rand(n, generator=gen, device=device)
    c[0::2] *= -1.0
    m = torch.randn(2977, generator=gen, device=device) * 1e-3
    v = torch.rand(2977, generator=gen, device=device) * 1e-5 + 1e-6
    return X.contiguous(), y, c, m, v


def _ensemble(case, seed):
    """Run descriptions and states: sizes from the ensemble's own draw, states seeded."""
    from paper_1702_08521_gb300 import inputs
    r = np.random.default_rng([seed, 3])
    draws = inputs.ensemble_draws(case["n1d"], case["n2d"])
    return [dict(d, alpha=float(r.uniform(0.001, 0.5)), phase=r.uniform(0.0, 2.0 * math.pi, size=2)) for d in draws]


def _member(d, device):
    """f of one ensemble run at t = 0, float32, shaped [x..][v..]."""
    D = d["dims"]
    xs = [_axis(d["xlo"][k], d["xhi"][k], d["nx"][k], device) for k in range(D)]
    vs = [_axis(d["vlo"][k], d["vhi"][k], d["nv"][k], device) for k in range(D)]
    s = sum(d["alpha"] / D * torch.cos(d["k"][k] * _along(x, k, 2 * D) + float(d["phase"][k])) for k, x in enumerate(xs)) + 1.0
    f = s
    for k, v in enumerate(vs):
        w = torch.exp(-0.5 * v * v) / math.sqrt(2.0 * math.pi)
        if d["kind"] == "two_stream" and k == 0:
            w = w * v * v
        f = f * _along(w, D + k, 2 * D)
    return f.float()


def _sine(case, seed, device):
    """The two-dimensional sine of the advection test, seeded phases; [n1][n2][nv][nv]."""
    r = np.random.default_rng([seed, 5])
    ph, a = r.uniform(0.0, 1.0, size=2), r.uniform(0.7, 0.95)
    x1, x2 = _axis(0.0, 1.0, case["n1"], device), _axis(0.0, 1.0, case["n2"], device)
    f = 1.0 + 0.5 * a * (torch.sin(2.0 * math.pi * (x1 + ph[0]))[:, None] + torch.sin(2.0 * math.pi * (x2 + ph[1])))
    return f.float()[:, :, None, None].expand(-1, -1, case["nv"], case["nv"]).contiguous()


def _unsplit_grid(case):
    nv = case["nv"]
    return dict(dims=2, nx=[case["n1"], case["n2"]], nv=[nv, nv], xlo=[0.0, 0.0], xhi=[1.0, 1.0], vlo=[0.5, 0.0],
                vhi=[1.5, 1.0], order=7, mp=1, pp=1, alpha=4.0, xbc=0, poisson=0, pois_order=6, coupling=-1.0, rho_bg=1.0)


# ---- the cases --------------------------------------------------------------------------

def prepare(case, seed):
    from paper_1702_08521_gb300 import vlasov as V
    kind = case["kind"]
    if kind in ("step", "sweeps"):
        g = _grid(case)
        sim = _sim(case, g, seed)
        diag = None
        if kind == "step" and case["diag"]:
            diag = torch.zeros(case["steps"] * V.VP_NDIAG, dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        return dict(case=case, V=V, sim=sim, diag=diag, split=V.VP_SPLIT_DKD if g["dims"] == 3 else V.VP_SPLIT_KDK)
    if kind == "ensemble":
        draws = _ensemble(case, seed)
        runs = [V.make_run(**{**d, "order": 7}) for d in draws]
        ens = V.vp_ensemble_create(runs, 7, _stream())
        pool = torch.zeros(V.vp_ensemble_num_cells(ens), dtype=torch.float32, device="cuda")
        V.vp_ensemble_bind(ens, pool)
        for i, d in enumerate(draws):
            off, _ = V.vp_ensemble_run_layout(ens, i)
            f = _member(d, "cuda").reshape(-1)
            pool[off:off + f.numel()] = f
        torch.cuda.synchronize()
        V.vp_ensemble_field(ens)
        V.vp_ensemble_autotune(ens, case["dt"])
        return dict(case=case, V=V, ens=_Owned(V, ens), pool=pool)
    if kind == "learned":
        g = _grid(case)
        sim = _sim(case, g, seed)
        w = _network(seed, 0.01, "cuda")
        torch.cuda.synchronize()
        return dict(case=case, V=V, sim=sim, w=w)
    if kind == "train":
        X, y, c, m, v = _batch(case, seed, "cuda")
        w = _network(seed, 0.1, "cuda")
        return dict(case=case, V=V, X=X, y=y, c=c, m=m, v=v, w=w, grad=torch.zeros_like(w),
                    loss=torch.zeros(1, device="cuda"))
    if kind == "samples":
        g = _grid(case)
        gc = dict(g, nv=[n // 4 for n in g["nv"]])
        fine = _sim(case, g, seed)
        coarse = V.Simulation(gc, precision=V.VP_F32, stream=_stream())
        m, ncl, grp = V.vp_fluxnet_line_map(V.make_grid(**g), V.make_grid(**gc), 4, 0, case["dim"])
        L = g["nx"][case["dim"]]
        cells = int(np.prod(g["nx"], dtype=np.int64) * np.prod(g["nv"], dtype=np.int64))
        ns = ncl * (L + 1)
        s = dict(case=case, V=V, fine=fine, coarse=coarse, map=torch.tensor(m, dtype=torch.int64, device="cuda"), ncl=ncl,
                 grp=grp, nout=L + 1, Gf=torch.empty(cells // L * (L + 1), dtype=torch.float64, device="cuda"),
                 Gc=torch.empty(ns, dtype=torch.float64, device="cuda"), X=torch.empty(ns, 25, device="cuda"),
                 y=torch.empty(ns, device="cuda"), sc=torch.empty(ns, device="cuda"))
        torch.cuda.synchronize()
        return s
    g = _unsplit_grid(case)
    sim = V.Simulation(g, precision=V.VP_F32, stream=_stream())
    sim.f.copy_(_sine(case, seed, "cuda").reshape(-1))
    scratch = torch.empty_like(sim.f)
    torch.cuda.synchronize()
    return dict(case=case, V=V, sim=sim, scratch=scratch)


class _Owned:
    """An ensemble handle, destroyed with its owner."""

    def __init__(self, V, h):
        self.V, self.h = V, h

    def __del__(self):
        try:
            self.V.vp_ensemble_destroy(self.h)
        except Exception:
            pass


def run(s):
    case, V = s["case"], s["V"]
    kind, dt = case["kind"], case.get("dt")
    if kind == "step":
        s["sim"].step(dt, case["steps"], split=s["split"], mode=1, diag=s["diag"])
        return [s["sim"].f, s["sim"].accel] + ([s["diag"]] if s["diag"] is not None else [])
    if kind == "sweeps":
        sim = s["sim"]
        D, NX, ctx, acc = sim.dims, sim.NX, sim.ctx, sim.accel
        if s["split"] == V.VP_SPLIT_KDK:
            for d in range(D):
                V.vp_kick_sweep(ctx, d, 0.5 * dt, acc[d * NX:])
            for d in reversed(range(D)):
                V.vp_drift_sweep(ctx, d, dt)
            sim.field()
            for d in range(D):
                V.vp_kick_sweep(ctx, d, 0.5 * dt, acc[d * NX:])
        else:
            for d in reversed(range(D)):
                V.vp_drift_sweep(ctx, d, 0.5 * dt)
            sim.field()
            for d in range(D):
                V.vp_kick_sweep(ctx, d, dt, acc[d * NX:])
            for d in reversed(range(D)):
                V.vp_drift_sweep(ctx, d, 0.5 * dt)
        out = [sim.f, acc, sim.rho, sim.phi]
        if case["diag"]:
            q = sim.diagnostics(1)
            out.append(np.array([q[k] for k in V.DIAG_NAMES]))
        return out
    if kind == "ensemble":
        V.vp_ensemble_step(s["ens"].h, dt, case["steps"])
        return [s["pool"]]
    if kind == "learned":
        s["sim"].learned_step(dt, case["steps"], s["w"], split=V.VP_SPLIT_KDK)
        return [s["sim"].f, s["sim"].accel]
    if kind == "train":
        st = torch.cuda.current_stream()
        s["loss"].zero_()
        V.vp_net_grad(s["X"], s["y"], s["y"].numel(), s["w"], s["grad"], s["loss"], st, coef=s["c"], group=2)
        V.vp_net_adam(s["w"], s["m"], s["v"], s["grad"], 1000, 1e-3, st)
        return [s["w"], s["m"], s["v"], s["loss"]]
    if kind == "samples":
        fine, coarse, d = s["fine"], s["coarse"], case["dim"]
        V.vp_fine_flux(fine.ctx, 0, d, dt, None, 1, s["Gf"])
        V.vp_group_mean(s["Gf"], s["ncl"], s["nout"], s["map"], s["grp"], 1.0, s["Gc"], _stream())
        nv = _ints(case["nv"])
        V.vp_restrict_velocity(fine.f, coarse.f, fine.NX, nv[0], nv[1], 4, 4, _stream())
        V.vp_make_samples(coarse.ctx, 0, d, dt, None, s["Gc"], 0.0, s["X"], s["y"], s["sc"])
        return [s["Gf"], s["Gc"], coarse.f, s["X"], s["y"], s["sc"]]
    V.vp_drift_unsplit(s["sim"].ctx, case["cfl"] / max(case["n1"], case["n2"]), case["steps"], s["scratch"])
    return [s["sim"].f]


# operations of one cell-update: interpolant 13, bounds 40, limiter and update 8
_FLOPS = 61


def work(case):
    kind = case["kind"]
    if kind in ("step", "sweeps", "learned", "samples"):
        nx, nv = _ints(case["nx"]), _ints(case["nv"])
        D = len(nx)
        cells = float(np.prod(np.array(nx + nv, dtype=float)))
        es = 8 if case.get("precision") == "f64" else 4
        sweeps = 3 * D * case.get("steps", 1)
        if kind == "samples":
            fine, coarse = cells / nx[case["dim"]] * (nx[case["dim"]] + 1), cells / 16 / nx[case["dim"]] * (nx[case["dim"]] + 1)
            return {"bytes": cells * 4 + fine * 8 + coarse * (8 + 27 * 4) + cells / 16 * 4, "flops": fine * _FLOPS + coarse * 120}
        flops = cells * sweeps * _FLOPS * (3 if case.get("scheme") == "rk" else 1)
        if kind == "learned":
            flops += cells * D * case["steps"] * 2 * (25 * 32 + 2 * 32 * 32 + 32)
        return {"bytes": 2 * es * cells, "flops": flops}
    if kind == "ensemble":
        from paper_1702_08521_gb300 import inputs
        bytes_, flops = 0.0, 0.0
        for d in inputs.ensemble_draws(case["n1d"], case["n2d"]):
            cells = float(np.prod(np.array(d["nx"] + d["nv"], dtype=float)))
            bytes_ += 8 * cells
            flops += cells * 3 * d["dims"] * case["steps"] * _FLOPS
        return {"bytes": bytes_, "flops": flops}
    if kind == "train":
        n = 2 * case["pairs"]
        return {"bytes": n * 27 * 4.0 + 2977 * 4 * 6.0, "flops": n * 6.0 * 2880}
    cells = float(case["n1"]) * case["n2"] * case["nv"] ** 2
    return {"bytes": 8 * cells, "flops": cells * 2 * case["steps"] * _FLOPS}


# ---- the same in 64 bits ---------------------------------------------------------------

def _csl_polys(order):
    """Interface value of the semi-Lagrangian flux: the mean over the departure interval
    [1/2 - nu, 1/2] of the polynomial whose cell integrals are the stencil; returns the
    polynomial in nu (ascending) of each of the cells -3..3."""
    P = np.polynomial.Polynomial
    h = (order - 1) // 2
    nodes = np.arange(-h - 1, h + 1) + 0.5
    x = P([0.5, -1.0])  # 1/2 - nu
    lag = []
    for i, a in enumerate(nodes):
        q = P([1.0])
        for j, b in enumerate(nodes):
            if j != i:
                q = q * P([-b, 1.0]) / (a - b)
        lag.append(q(0.5) - q(x))
    out = [np.zeros(1)] * 7
    for k in range(-h, h + 1):
        t = sum((lag[i] for i, a in enumerate(nodes) if a > k), P([0.0]))
        out[k + 3] = t.coef[1:]  # divided by nu
    return out


def _weights(order, nu):
    return [sum((float(c) * nu ** j for j, c in enumerate(p)), torch.zeros_like(nu)) for p in _csl_polys(order)]


def _minmod4(a, b, c, d):
    lo = torch.minimum(torch.minimum(a, b), torch.minimum(c, d))
    hi = torch.maximum(torch.maximum(a, b), torch.maximum(c, d))
    return torch.clamp(lo, min=0.0) + torch.clamp(hi, max=0.0)


def _min3(a, b, c):
    return torch.minimum(torch.minimum(a, b), c)


def _max3(a, b, c):
    return torch.maximum(torch.maximum(a, b), c)


def _phi(u, w):
    """Interface value between u[3] and u[4] of the upwind-ordered cells u[0..6]: the
    interpolant, clamped into the monotonicity-preserving bounds."""
    v = sum(w[k] * u[k] for k in range(7))
    d = [u[k - 1] + u[k + 1] - 2.0 * u[k] for k in (2, 3, 4)]
    m4p = _minmod4(4.0 * d[1] - d[2], 4.0 * d[2] - d[1], d[1], d[2])
    m4m = _minmod4(4.0 * d[0] - d[1], 4.0 * d[1] - d[0], d[0], d[1])
    back = u[3] - u[2]
    ful, fmd = u[3] + 4.0 * back, 0.5 * (u[3] + u[4]) - 0.5 * m4p
    flc = u[3] + 0.5 * back + 4.0 / 3.0 * m4m
    lo = torch.maximum(_min3(u[3], u[4], fmd), _min3(u[3], ful, flc))
    hi = torch.minimum(_max3(u[3], u[4], fmd), _max3(u[3], ful, flc))
    return torch.minimum(torch.maximum(v, lo), hi)


def _positive(M, u0, u1, nu):
    """The positivity limiter on an interface mass M; next to a negative cell as the
    blend with the upwind mass."""
    out = torch.minimum(torch.maximum(M, -0.5 * u1), 0.5 * u0)
    bad = (u0 < 0) | (u1 < 0)
    if bool(bad.any()):
        phi = M / torch.where(nu > 0, nu, torch.ones_like(nu))
        up, um = u0 - 2 * nu * phi, u1 + 2 * nu * phi
        upu, umu = u0 - 2 * nu * u0, u1 + 2 * nu * u0
        one = torch.ones_like(M)

        def theta(full, upwind):
            den = upwind - full
            return torch.where(full < 0, torch.where(den > 0, upwind / torch.where(den > 0, den, one), 0.0 * one), one)
        th = torch.clamp(torch.minimum(theta(up, upu), theta(um, umu)), 0.0, 1.0)
        out = torch.where(bad, nu * (th * phi + (1.0 - th) * u0), out)
    return out


def _rows(f, r, periodic):
    """f[:, r] per line, zero outside a line that does not wrap; f [O][L][I]."""
    L = f.shape[1]
    if periodic:
        return torch.gather(f, 1, (r % L).expand(f.shape[0], -1, f.shape[2]))
    inside = (r >= 0) & (r < L)
    v = torch.gather(f, 1, r.clamp(0, L - 1).expand(f.shape[0], -1, f.shape[2]))
    return torch.where(inside, v, torch.zeros_like(v))


def _split_shift(s):
    n = torch.sign(s) * torch.floor(torch.abs(s) + 0.5)
    z = s - n
    return n.long(), torch.where(z < 0, -1, 1).long(), torch.abs(z)


def _euler(f, n, sg, nu, w, periodic):
    """One conservative update of the lines f [O][L][I]: whole cells n, then the
    limited fractional masses in direction sg."""
    L = f.shape[1]
    i = torch.arange(L, device=f.device).view(1, L, 1)
    u = [_rows(f, i - n + k * sg, periodic) for k in range(-4, 5)]  # u[4]: the cell's own source
    out = _positive(nu * _phi(u[1:8], w), u[4], u[5], nu)
    inn = _positive(nu * _phi(u[0:7], w), u[3], u[4], nu)
    return u[4] - out + inn


def _sweep(f, axis, s, periodic, order, scheme):
    """Advance f (full shape) along `axis` by s cells (broadcastable, size 1 there)."""
    shape = list(f.shape)
    O, L, I = int(np.prod(shape[:axis])), shape[axis], int(np.prod(shape[axis + 1:]))
    line = list(shape)
    line[axis] = 1
    s = s.expand(line).reshape(O, 1, I)
    v = f.view(O, L, I)
    out = torch.empty_like(v)
    most = 1 << 24
    ci = I if L * I <= most else max(1, most // L)
    co = max(1, most // (L * ci))
    for o in range(0, O, co):
        for c in range(0, I, ci):
            a, b = v[o:o + co, :, c:c + ci], s[o:o + co, :, c:c + ci]
            if scheme == "rk":
                sg, nu = torch.where(b < 0, -1, 1).long(), torch.abs(b)
                w = [torch.full_like(nu, x / 60.0) for x in (0.0, 2.0, -13.0, 47.0, 27.0, -3.0, 0.0)]
                n = torch.zeros_like(sg)
                f1 = _euler(a, n, sg, nu, w, periodic)
                f2 = 0.75 * a + 0.25 * _euler(f1, n, sg, nu, w, periodic)
                r = a / 3.0 + 2.0 / 3.0 * _euler(f2, n, sg, nu, w, periodic)
            else:
                n, sg, nu = _split_shift(b)
                r = _euler(a, n, sg, nu, _weights(order, nu), periodic)
            out[o:o + co, :, c:c + ci] = r
    return out.view(shape)


def _density(f, g):
    D = g["dims"]
    dv = np.prod([(g["vhi"][d] - g["vlo"][d]) / g["nv"][d] for d in range(D)])
    return f.flatten(D).sum(-1) * dv


def _field(rho, g):
    """Potential and acceleration on the mesh (Fourier convolution, central differences)."""
    D, n, dev = g["dims"], g["nx"], rho.device
    h = [(g["xhi"][d] - g["xlo"][d]) / n[d] for d in range(D)]
    if g["poisson"] == 0:
        lam = torch.zeros([1] * D, dtype=torch.float64, device=dev)
        for d in range(D):
            th = 2.0 * math.pi * torch.arange(n[d], dtype=torch.float64, device=dev) / n[d]
            e = sum(b * torch.sin(0.5 * m * th) ** 2 for m, b in ((1, 270.0), (2, -27.0), (3, 2.0)))
            lam = lam + _along(-4.0 * e / 180.0 / h[d] ** 2, d, D)
        hat = torch.fft.fftn(rho - g["rho_bg"])
        lam.view(-1)[0] = 1.0
        hat = g["coupling"] * hat / lam
        hat.view(-1)[0] = 0.0
        phi = torch.fft.ifftn(hat).real
    else:
        m = [2 * k for k in n]
        r2 = torch.zeros([1] * D, dtype=torch.float64, device=dev)
        for d in range(D):
            j = torch.arange(m[d], dtype=torch.float64, device=dev)
            r2 = r2 + _along(torch.minimum(j, m[d] - j) ** 2, d, D)
        inv = torch.where(r2 > 0, 1.0 / torch.sqrt(torch.clamp(r2, min=1.0)), 3.0 * math.log(2.0 + math.sqrt(3.0)) - 0.5 * math.pi)
        ker = -(g["coupling"] / (4.0 * math.pi)) * h[0] ** 2 * inv
        pad = torch.zeros(m, dtype=torch.float64, device=dev)
        pad[tuple(slice(0, k) for k in n)] = rho - g["rho_bg"]
        phi = torch.fft.ifftn(torch.fft.fftn(pad) * torch.fft.fftn(ker)).real
    box = tuple(slice(0, k) for k in n)
    acc = []
    for d in range(D):
        df = sum(c * (torch.roll(phi, -k, d) - torch.roll(phi, k, d)) for k, c in ((1, 45.0), (2, -9.0), (3, 1.0)))
        acc.append((-df / (60.0 * h[d]))[box])
    return phi[box], acc


def _diag(f, g):
    D = g["dims"]
    rho = _density(f, g)
    phi, acc = _field(rho, g)
    dX = np.prod([(g["xhi"][d] - g["xlo"][d]) / g["nx"][d] for d in range(D)])
    dV = np.prod([(g["vhi"][d] - g["vlo"][d]) / g["nv"][d] for d in range(D)])
    fx = f.flatten(0, D - 1).sum(0)
    ke = sum(float((fx * _along(_axis(g["vlo"][d], g["vhi"][d], g["nv"][d], f.device) ** 2, d, D)).sum()) for d in range(D))
    j = torch.arange(g["nx"][0], dtype=torch.float64, device=f.device)
    e = torch.exp(-2j * math.pi * j / g["nx"][0])
    amp = 2.0 / rho.numel() * abs(complex((acc[0].reshape(g["nx"][0], -1).sum(1) * e).sum()))
    return [float(f.sum()) * dX * dV, 0.5 * ke * dX * dV, 0.5 * sum(float((a * a).sum()) for a in acc) * dX,
            0.5 * float(((rho - g["rho_bg"]) * phi).sum()) * dX, float(f.min()), float(f.max()), amp,
            float(f.abs().sum()) * dX * dV, sum(float((b * b).sum()) for b in f.reshape(-1).split(1 << 26)) * dX * dV]


def _drift(f, d, dt, g, scheme="sl"):
    D = g["dims"]
    v = _axis(g["vlo"][d], g["vhi"][d], g["nv"][d], f.device)
    s = _along(v * dt / ((g["xhi"][d] - g["xlo"][d]) / g["nx"][d]), D + d, 2 * D)
    return _sweep(f, d, s, g["xbc"] == 0, g["order"], scheme)


def _kick(f, d, dt, acc, g, scheme="sl"):
    D = g["dims"]
    s = (acc[d] * dt / ((g["vhi"][d] - g["vlo"][d]) / g["nv"][d])).reshape(g["nx"] + [1] * D)
    return _sweep(f, D + d, s, False, g["order"], scheme)


def _strang(f, acc, g, dt, scheme, drift=_drift):
    D = g["dims"]
    if D < 3:
        for d in range(D):
            f = _kick(f, d, 0.5 * dt, acc, g, scheme)
        for d in reversed(range(D)):
            f = drift(f, d, dt, g, scheme)
        rho = _density(f, g)
        phi, acc = _field(rho, g)
        for d in range(D):
            f = _kick(f, d, 0.5 * dt, acc, g, scheme)
    else:
        for d in reversed(range(D)):
            f = drift(f, d, 0.5 * dt, g, scheme)
        rho = _density(f, g)
        phi, acc = _field(rho, g)
        for d in range(D):
            f = _kick(f, d, dt, acc, g, scheme)
        for d in reversed(range(D)):
            f = drift(f, d, 0.5 * dt, g, scheme)
    return f, acc, rho, phi


def _bf16(x):
    return x.to(torch.float32).to(torch.bfloat16).to(torch.float64)


def _layers(w):
    """Rounded matrices and the biases (as the sum of two bfloat16 numbers) of a network."""
    at, out = 0, []
    for rows, cols in ((32, 25), (32, 32), (32, 32), (1, 32)):
        W = _bf16(w[at:at + rows * cols]).view(rows, cols)
        at += rows * cols
        b = w[at:at + rows].double()
        at += rows
        out.append((W, b))
    return out


def _net(x, layers):
    """x [..., 25] -> [...]; inputs and activations rounded to bfloat16."""
    a = _bf16(x)
    for i, (W, b) in enumerate(layers):
        hi = _bf16(b)
        a = a @ W.T + (hi + _bf16(b - hi))
        if i < 3:
            a = _bf16(torch.relu(a))
    return a[..., 0]


def _learned_drift(w):
    layers = _layers(w)

    def drift(f, d, dt, g, scheme):
        D = g["dims"]
        J, L = g["nv"][d], g["nx"][d]
        v = _axis(g["vlo"][d], g["vhi"][d], J, f.device)
        s = _along(v * dt / ((g["xhi"][d] - g["xlo"][d]) / L), D + d, 2 * D)
        vax = D + d
        z = torch.zeros_like(f.narrow(vax, 0, 1))
        nxt = torch.cat([f.narrow(vax, 1, J - 1), z], vax)
        prv = torch.cat([z, f.narrow(vax, 0, J - 1)], vax)
        pos = _along(v >= 0, vax, 2 * D)
        fp, fm = torch.where(pos, nxt, prv), torch.where(pos, prv, nxt)
        shape = list(f.shape)
        O, I = int(np.prod(shape[:d])), int(np.prod(shape[d + 1:]))
        line = list(shape)
        line[d] = 1
        ss = s.expand(line).reshape(O, 1, I)
        a, ap, am = f.reshape(O, L, I), fp.reshape(O, L, I), fm.reshape(O, L, I)
        out = torch.empty_like(a)
        most = 1 << 21
        ci = I if L * I <= most else max(1, most // L)
        co = max(1, most // (L * ci))
        i = torch.arange(L, device=f.device).view(1, L, 1)
        for o in range(0, O, co):
            for c in range(0, I, ci):
                cut = (slice(o, o + co), slice(None), slice(c, c + ci))
                n, sg, nu = _split_shift(ss[cut])
                wt = _weights(7, nu)
                r = [i - n + k * sg for k in range(-4, 5)]
                u, p, m = ([_rows(t[cut].contiguous(), k, True) for k in r] for t in (a, ap, am))

                def mass(q):  # out of the cell whose source is u[q]
                    st = u[q - 3:q + 5]
                    sc = torch.stack([t.abs() for t in st]).amax(0) + 1e-30
                    x = [(t - u[q]) / sc for t in st] + [(p[k] - m[k]) / (2.0 * sc) for k in range(q - 3, q + 5)]
                    x += [(0.5 * (p[k] + m[k]) - u[k]) / sc for k in range(q - 3, q + 5)] + [nu.expand_as(sc)]
                    M = nu * _phi(st[:7], wt) + sc * _net(torch.stack(x, -1), layers)
                    return torch.minimum(torch.maximum(M, -0.5 * u[q + 1]), 0.5 * u[q])
                out[cut] = u[4] - mass(4) + mass(3)
        return out.view(shape)
    return drift


def _train(case, seed, device):
    """Gradient of the mean squared pair residual, straight through the roundings, and
    one Adam step; in 64 bits with the roundings of inputs, weights and activations."""
    X, y, c, m, v = _batch(case, seed, device)
    w32 = _network(seed, 0.1, device)
    layers = _layers(w32)
    n, groups = y.numel(), y.numel() // 2
    grad = [[torch.zeros_like(W), torch.zeros_like(b)] for W, b in layers]
    loss = 0.0
    for i in range(0, n, 1 << 19):
        x = _bf16(X[i:i + (1 << 19)])
        h = [x]
        for k, (W, b) in enumerate(layers):
            z = h[-1] @ W.T + b
            h.append(_bf16(torch.relu(z)) if k < 3 else z)
        a = c[i:i + (1 << 19)].double()
        r = (a * (h[4][:, 0] - y[i:i + (1 << 19)].double())).view(-1, 2).sum(1)
        loss += float((r * r).sum()) / groups
        d = (2.0 * r.repeat_interleave(2) * a / groups)[:, None]
        for k in (3, 2, 1, 0):
            grad[k][0] += d.T @ h[k]
            grad[k][1] += d.sum(0)
            if k:
                d = (d @ layers[k][0]) * (h[k] > 0)
    gr = torch.cat([t.reshape(-1) for pair in grad for t in pair])
    # the Adam coefficients as 32-bit numbers, as the call holds them
    b1, b2 = float(np.float32(0.9)), float(np.float32(0.999))
    m2 = b1 * m.double() + float(np.float32(1.0) - np.float32(0.9)) * gr
    v2 = b2 * v.double() + float(np.float32(1.0) - np.float32(0.999)) * gr * gr
    bc1, bc2 = 1.0 - b1 ** 1000, 1.0 - b2 ** 1000
    w = w32.double() - float(np.float32(1e-3)) * (m2 / bc1) / (torch.sqrt(v2 / bc2) + float(np.float32(1e-8)))
    return [w, m2, v2, torch.tensor([loss], dtype=torch.float64)]


def _interfaces(f, d, g, dt):
    """Fine-grid masses through every interface of the lines along x_d, before cells
    0..L, signed along +x_d; f [O][L][I] views; returns [O][L + 1][I] and the parts of
    the stencil at the shifted interface."""
    D, L = g["dims"], g["nx"][d]
    shape = list(f.shape)
    O, I = int(np.prod(shape[:d])), int(np.prod(shape[d + 1:]))
    v = _axis(g["vlo"][d], g["vhi"][d], g["nv"][d], f.device)
    line = list(shape)
    line[d] = 1
    s = _along(v * dt / ((g["xhi"][d] - g["xlo"][d]) / L), D + d, 2 * D).expand(line).reshape(O, 1, I)
    return f.reshape(O, L, I), s, torch.arange(L + 1, device=f.device).view(1, L + 1, 1)


def _samples(case, seed, device):
    """Fluxes, restriction, features and targets of one spatial sweep of a periodic grid."""
    g = _grid(case)
    d, D, dt = case["dim"], 2, case["dt"]
    shape = g["nx"] + g["nv"]
    f = torch.empty(int(np.prod(shape)), dtype=torch.float32, device=device)
    _fill(case, g, seed, f, torch.float32)
    L = g["nx"][d]

    def masses(a, s, i, limit):
        n, sg, nu = _split_shift(s)
        up = torch.where(sg > 0, i - 1 - n, i - n)  # upwind cell of the shifted interface
        u = [_rows(a, up + k * sg, True) for k in range(-3, 5)]
        phi = _phi(u[:7], _weights(7, nu))
        M = nu * phi
        if limit:
            M = torch.minimum(torch.maximum(M, -0.5 * u[4]), 0.5 * u[3])
        # whole cells between the interface and the shifted one, signed along +x
        S = torch.cat([torch.zeros_like(a[:, :1]), torch.cumsum(a, 1)], 1)
        total = S[:, L:L + 1]

        def upto(k):
            k = k.expand(a.shape[0], L + 1, a.shape[2])
            return torch.gather(S, 1, k % L) + torch.div(k, L, rounding_mode="floor") * total
        return upto(i) - upto(i - n), sg * M, u, sg, nu, up

    nvf, nvc = g["nv"], [k // 4 for k in g["nv"]]
    full = f.view(shape)
    Gf = torch.empty([0])
    a, s, i = _interfaces(full, d, g, dt)
    O, _, I = a.shape
    Gf = torch.empty(O, L + 1, I, dtype=torch.float64, device=device)
    co = max(1, (1 << 23) // (L * I))
    ci = I if L * I <= (1 << 23) else max(1, (1 << 23) // L)
    for o in range(0, O, co):
        for c in range(0, I, ci):
            q = a[o:o + co, :, c:c + ci].double()
            whole, M, *_ = masses(q, s[o:o + co, :, c:c + ci], i, True)
            Gf[o:o + co, :, c:c + ci] = whole + M
    rest = [g["nx"][1]] if d == 0 else []
    v6 = Gf.view([O, L + 1] + rest + [nvc[0], 4, nvc[1], 4])
    Gc = v6.mean((-1, -3)).reshape(O, L + 1, -1)
    fc = full.double().view(g["nx"] + [nvc[0], 4, nvc[1], 4]).mean((-1, -3)).float()
    gc = dict(g, nv=nvc)
    a, s, i = _interfaces(fc, d, gc, dt)
    a = a.double()
    whole, M, u, sg, nu, up = masses(a, s, i, False)
    vax = D + d
    J = nvc[d]
    z = torch.zeros_like(fc.narrow(vax, 0, 1))
    nxt, prv = torch.cat([fc.narrow(vax, 1, J - 1), z], vax), torch.cat([z, fc.narrow(vax, 0, J - 1)], vax)
    pos = _along(_axis(g["vlo"][d], g["vhi"][d], J, device) >= 0, vax, 2 * D)
    fp, fm = (torch.where(pos, x, y).reshape(a.shape).double() for x, y in ((nxt, prv), (prv, nxt)))
    p = [_rows(fp, up + k * sg, True) for k in range(-3, 5)]
    m = [_rows(fm, up + k * sg, True) for k in range(-3, 5)]
    sc = torch.stack([t.abs() for t in u]).amax(0) + 1e-30
    X = [(t - u[3]) / sc for t in u] + [(x - y) / (2.0 * sc) for x, y in zip(p, m)]
    X += [(0.5 * (x + y) - t) / sc for x, y, t in zip(p, m, u)] + [nu.expand_as(sc)]
    y = sg * (Gc - whole - M) / sc
    X = torch.stack(X, -1)
    X[:, L] = 0.0
    y[:, L] = float("nan")
    sc = sc.clone()
    sc[:, L] = 0.0
    t = lambda q: q.transpose(1, 2).contiguous()  # noqa: E731  [line][interface]
    return [t(Gf).reshape(-1), t(Gc).reshape(-1), fc.double().reshape(-1), t(X).reshape(-1, 25), t(y).reshape(-1), t(sc).reshape(-1)]


def exact(case, seed):
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    kind = case["kind"]
    if kind in ("step", "sweeps", "learned"):
        g = _grid(case)
        shape = g["nx"] + g["nv"]
        cells = float(np.prod(np.array(shape, dtype=float)))
        if cells * case.get("steps", 1) > 4e8:
            return None
        f = torch.empty(int(cells), dtype=torch.float64, device=dev)
        _fill(case, g, seed, f, torch.float64 if case.get("precision") == "f64" else torch.float32)
        f = f.view(shape)
        _, acc = _field(_density(f, g), g)
        drift = _learned_drift(_network(seed, 0.01, dev)) if kind == "learned" else _drift
        out = []
        for _ in range(case.get("steps", 1)):
            f, acc, rho, phi = _strang(f, acc, g, case["dt"], case.get("scheme", "sl"), drift)
            if case.get("diag"):
                out += _diag(f, g)
        r = [f.reshape(-1), torch.stack(acc).reshape(-1)]
        if kind == "sweeps":
            r += [rho.reshape(-1), phi.reshape(-1)]
        return r + ([torch.tensor(out, dtype=torch.float64)] if case.get("diag") else [])
    if kind == "ensemble":
        pool = []
        for d in _ensemble(case, seed):
            g = dict(d, order=7, xbc=0, poisson=0, coupling=-1.0, rho_bg=1.0)
            f = _member(d, dev).double()
            _, acc = _field(_density(f, g), g)
            for _ in range(case["steps"]):
                f, acc, _, _ = _strang(f, acc, g, case["dt"], "sl")
            f = f.reshape(-1)
            pool += [f, torch.zeros(-f.numel() % 32, dtype=torch.float64, device=dev)]
        return [torch.cat(pool)]
    if kind == "train":
        return _train(case, seed, dev)
    if kind == "samples":
        return _samples(case, seed, dev)
    g = _unsplit_grid(case)
    f = _sine(case, seed, dev).double()
    dt = case["cfl"] / max(case["n1"], case["n2"])
    for _ in range(case["steps"]):
        f = f + (_drift(f, 0, dt, g) - f) + (_drift(f, 1, dt, g) - f)
    return [f.reshape(-1)]
