"""Learned flux correction: training kernels against the FP64 reference,
the learned spatial sweep against the plain sweep and an oracle line update
(with the velocity-neighbour features),
conservation and positivity with the network on, the fine-flux extraction
used to build training data, and what a trained network gains."""
import math

import numpy as np
import pytest

import oracle as O
from oracle import flux_net as N
from paper_1702_08521_gb300 import inputs
from paper_1702_08521_gb300 import vlasov as V

from gpu_helpers import both, from_gpu, rel_l1, rel_max, snapshot, to_gpu

pytestmark = pytest.mark.gpu


def _t(a, dtype=None):
    import torch
    return torch.as_tensor(np.ascontiguousarray(a), dtype=dtype, device="cuda")


def _f32(a):
    return np.asarray(a, dtype=np.float32).astype(np.float64)


def _params(seed, scale=1.0):
    p = N.init_params(seed)
    rng = np.random.default_rng(seed + 100)
    for k in p:
        p[k] = _f32(p[k] * scale + 0.02 * rng.normal(size=p[k].shape))
    return p


def test_net_gradients_match_reference():
    import torch
    rng = np.random.default_rng(0)
    p = _params(1)
    B = 1000
    X = _f32(rng.normal(size=(B, N.NFEAT)))
    y = _f32(rng.normal(size=B))
    loss_ref, g_ref = N.loss_and_grad(p, X, y, round_bf16=True)
    w = _t(N.pack(p), torch.float32)
    grad = torch.zeros_like(w)
    loss = torch.zeros(1, dtype=torch.float32, device="cuda")
    V.vp_net_grad(_t(X.ravel(), torch.float32), _t(y, torch.float32), B, w, grad, loss)
    torch.cuda.synchronize()
    assert loss.item() == pytest.approx(loss_ref, rel=1e-4)
    gv = grad.double().cpu().numpy()
    rv = N.pack(g_ref)
    assert np.abs(gv - rv).max() <= 1e-2 * np.abs(rv).max()
    assert np.linalg.norm(gv - rv) <= 1e-3 * np.linalg.norm(rv)


def test_pair_loss_gradients_match_reference():
    import torch
    rng = np.random.default_rng(2)
    p = _params(3)
    B = 1000
    X = _f32(rng.normal(size=(B, N.NFEAT)))
    y = _f32(rng.normal(size=B))
    a = _f32(rng.uniform(-1, 1, size=B))
    loss_ref, g_ref = N.loss_and_grad(p, X, y, round_bf16=True, coef=a, group=2)
    w = _t(N.pack(p), torch.float32)
    grad = torch.zeros_like(w)
    loss = torch.zeros(1, dtype=torch.float32, device="cuda")
    V.vp_net_grad(_t(X.ravel(), torch.float32), _t(y, torch.float32), B, w, grad, loss,
                  coef=_t(a, torch.float32), group=2)
    torch.cuda.synchronize()
    assert loss.item() == pytest.approx(loss_ref, rel=1e-4)
    gv = grad.double().cpu().numpy()
    rv = N.pack(g_ref)
    assert np.abs(gv - rv).max() <= 1e-2 * np.abs(rv).max()
    assert np.linalg.norm(gv - rv) <= 1e-3 * np.linalg.norm(rv)


def test_adam_moves_against_the_gradient():
    import torch
    w = torch.zeros(V.VP_NET_NPARAM, dtype=torch.float32, device="cuda")
    g = torch.linspace(-1, 1, V.VP_NET_NPARAM, device="cuda")
    m, v = torch.zeros_like(w), torch.zeros_like(w)
    g0 = g.clone()
    V.vp_net_adam(w, m, v, g, 1, 1e-3)
    torch.cuda.synchronize()
    # first Adam step moves every parameter by -lr * g / (|g| + eps), i.e.
    # -lr * sign(g) wherever |g| >> eps
    nz = g0.abs() > 1e-4
    assert torch.allclose(w[nz], -1e-3 * torch.sign(g0[nz]), rtol=1e-3, atol=1e-7)
    assert torch.count_nonzero(g) == 0


def _grid2d(nx, nv):
    L = 4 * math.pi
    return dict(dims=2, nx=[nx, nx], nv=[nv, nv], xlo=[0.0, 0.0], xhi=[L, L], vlo=[-6.0, -6.0],
                vhi=[6.0, 6.0], order=7)


def test_learned_sweep_without_net_is_the_plain_sweep():
    import torch
    g = _grid2d(8, 16)
    sim, og = both(g, V.VP_F32)
    f0 = inputs.random_f(og.NX * og.NV, seed=3).astype(np.float32)
    acc = inputs.random_accel(og.NX, 2, seed=4, amax=3.0)
    w = torch.zeros(V.VP_NET_NPARAM, dtype=torch.float32, device="cuda")
    for kick in (0, 1):
        for d in range(2):
            to_gpu(sim, f0)
            a = _t(acc[d])
            if kick:
                V.vp_kick_sweep(sim.ctx, d, 0.4, a)
            else:
                V.vp_drift_sweep(sim.ctx, d, 0.4)
            ref = from_gpu(sim)
            to_gpu(sim, f0)
            V.vp_learned_sweep(sim.ctx, kick, d, 0.4, a, w, 0)
            got = from_gpu(sim)
            assert rel_max(got, ref) <= 1e-6, (kick, d)
    sim.close()


@pytest.mark.parametrize("use_net", [1, 2])
def test_learned_sweep_matches_oracle_line_update(use_net):
    """use_net 1: PP on the corrected mass; 2: the MP bounds of App. A on it
    first (the oracle's mp_bound)."""
    import torch
    g = dict(dims=1, nx=[24], nv=[20], xlo=[0.0], xhi=[2.0], vlo=[-3.0], vhi=[3.0], order=7)
    sim, og = both(g, V.VP_F32)
    f0 = _f32(inputs.random_f(og.NX * og.NV, seed=5))
    p = _params(7, scale=0.3)
    w = _t(N.pack(p), torch.float32)
    to_gpu(sim, f0)
    V.vp_learned_sweep(sim.ctx, 0, 0, 0.37, None, w, use_net, snapshot(sim))
    got = from_gpu(sim).reshape(24, 20)
    want = np.empty((24, 20))
    f2 = f0.reshape(24, 20)
    vc = og.v_centres(0)
    zero = np.zeros(24)
    for j in range(20):
        s = vc[j] * 0.37 / (2.0 / 24)
        sp = 1 if vc[j] >= 0 else -1
        up = f2[:, j + sp] if 0 <= j + sp < 20 else zero
        um = f2[:, j - sp] if 0 <= j - sp < 20 else zero
        want[:, j] = N.learned_line(f2[:, j], up, um, s, p, O.BC_PERIODIC, mp_bound=use_net == 2)
    # FP32 sums vs FP64 sums can move a bfloat16 rounding by one step
    assert rel_l1(got, want) <= 2e-3, rel_l1(got, want)
    sim.close()


def test_learned_sweep_integer_shift_is_exact_with_mp_bounds():
    """An integer shift (nu = 0 on every line) with the network on and the MP
    bounds applied to its correction (use_net = 2): in mass form they have
    zero width, so the learned sweep is the exact shift of every line, bit
    for bit, as in the oracle's learned update."""
    import torch
    g = dict(dims=1, nx=[24], nv=[20], xlo=[0.0], xhi=[24.0], vlo=[-5.0], vhi=[5.0], order=7)
    sim, og = both(g, V.VP_F32)
    f0 = _f32(inputs.random_f(og.NX * og.NV, seed=15))
    w = _t(N.pack(_params(9, scale=3.0)), torch.float32)
    to_gpu(sim, f0)
    # dx = 1, v_j = -4.75 + 0.5 j, dt = 4: shift v_j dt = -19 + 2 j cells
    dt = 4.0
    V.vp_learned_sweep(sim.ctx, 0, 0, dt, None, w, 2, snapshot(sim))
    got = from_gpu(sim).reshape(24, 20)
    f2 = f0.reshape(24, 20)
    for j, v in enumerate(og.v_centres(0)):
        n = int(round(v * dt))
        assert v * dt == n
        assert np.array_equal(got[:, j], np.roll(f2[:, j], n)), j
    sim.close()


def test_learned_sweep_conserves_mass_and_positivity():
    import torch
    g = _grid2d(8, 16)
    sim, og = both(g, V.VP_F32)
    f0 = (inputs.random_f(og.NX * og.NV, seed=9, zeros=0.4) ** 4).astype(np.float32)
    p = _params(11, scale=3.0)  # a large, untrained correction
    w = _t(N.pack(p), torch.float32)
    to_gpu(sim, f0)
    m0 = float(np.sum(f0, dtype=np.float64))
    for _ in range(3):
        for d in range(2):
            V.vp_learned_sweep(sim.ctx, 0, d, 0.3, None, w, 1, snapshot(sim))
    got = from_gpu(sim)
    assert got.min() >= 0.0
    assert abs(got.sum() - m0) / m0 <= 1e-6
    sim.close()


def test_fine_flux_reproduces_the_sweep():
    import torch
    g = _grid2d(8, 16)
    sim, og = both(g, V.VP_F32)
    f0 = inputs.random_f(og.NX * og.NV, seed=12).astype(np.float32)
    acc = inputs.random_accel(og.NX, 2, seed=13, amax=8.0)
    for kick, d in ((0, 0), (0, 1), (1, 0), (1, 1)):
        to_gpu(sim, f0)
        a = _t(acc[d])
        L = g["nv"][d] if kick else g["nx"][d]
        nlines = og.NX * og.NV // L
        G = torch.zeros(nlines * (L + 1), dtype=torch.float64, device="cuda")
        V.vp_fine_flux(sim.ctx, kick, d, 0.55, a, 1, G)
        if kick:
            V.vp_kick_sweep(sim.ctx, d, 0.55, a)
        else:
            V.vp_drift_sweep(sim.ctx, d, 0.55)
        ref = from_gpu(sim)
        Gh = G.cpu().numpy().reshape(nlines, L + 1)
        # rebuild f' = f + G_{i-1/2} - G_{i+1/2} along every line
        shp = og.shape
        axis = (2 + d) if kick else d
        fl = np.moveaxis(f0.reshape(shp).astype(np.float64), axis, -1)
        lines = fl.reshape(-1, L)
        order = np.arange(np.prod(shp)).reshape(shp)
        idx = np.moveaxis(order, axis, -1).reshape(-1, L)
        # G rows follow the library's line order: [outer][inner]
        outer = int(np.prod(shp[:axis]))
        inner = int(np.prod(shp[axis + 1:]))
        lib_first = (np.arange(outer)[:, None] * L * inner + np.arange(inner)[None, :]).ravel()
        pos = {v: k for k, v in enumerate(idx[:, 0])}
        rows = np.array([pos[v] for v in lib_first])
        new = lines[rows] + Gh[:, :-1] - Gh[:, 1:]
        got = np.empty(np.prod(shp))
        got[idx[rows].ravel()] = new.ravel()
        assert rel_max(got, ref) <= 1e-5, (kick, d, rel_max(got, ref))
    sim.close()


def test_learned_correction_rejects_velocity_sweeps():
    import torch
    g = _grid2d(8, 16)
    sim, og = both(g, V.VP_F32)
    w = torch.zeros(V.VP_NET_NPARAM, dtype=torch.float32, device="cuda")
    acc = _t(inputs.random_accel(og.NX, 2, seed=4, amax=3.0)[0])
    with pytest.raises(V.VpError):
        V.vp_learned_sweep(sim.ctx, 1, 0, 0.4, acc, w, 1, snapshot(sim))
    sim.close()


def test_learned_step_replays_the_sweep_sequence():
    """vp_learned_step (captured in a CUDA graph) gives, bit for bit, the f
    of the same KDK sequence issued sweep by sweep: plain kicks, learned
    drifts (library snapshot), field solve between; and a plain vp_step
    is unchanged by the learned path having run on the context."""
    import torch
    g = _grid2d(8, 16)
    f0 = (inputs.random_f(8 * 8 * 16 * 16, seed=21, zeros=0.3) ** 2).astype(np.float32)
    w = _t(N.pack(_params(5, scale=0.5)), torch.float32)
    dt = 0.2
    a, _ = both(g, V.VP_F32)
    b, _ = both(g, V.VP_F32)
    for sim in (a, b):
        to_gpu(sim, f0)
        sim.field()
    a.learned_step(dt, 3, w)
    a.sync()
    for _ in range(3):
        for d in range(2):
            V.vp_kick_sweep(b.ctx, d, 0.5 * dt, b.accel[d * b.NX:])
        for d in (1, 0):
            V.vp_learned_sweep(b.ctx, 0, d, dt, None, w, 1)
        b.field()
        for d in range(2):
            V.vp_kick_sweep(b.ctx, d, 0.5 * dt, b.accel[d * b.NX:])
    b.sync()
    fa, fb = from_gpu(a), from_gpu(b)
    assert np.array_equal(fa, fb)
    assert fa.min() >= 0.0
    # the plain step on the same contexts still matches sweep by sweep
    a.step(dt, 1)
    a.sync()
    for d in range(2):
        V.vp_kick_sweep(b.ctx, d, 0.5 * dt, b.accel[d * b.NX:])
    for d in (1, 0):
        V.vp_drift_sweep(b.ctx, d, dt)
    b.field()
    for d in range(2):
        V.vp_kick_sweep(b.ctx, d, 0.5 * dt, b.accel[d * b.NX:])
    b.sync()
    assert np.array_equal(from_gpu(a), from_gpu(b))
    a.close()
    b.close()


def test_learned_sweep_velocity_axis_limit():
    """One 128-row MMA operand per interface step: 128 velocity cells on the
    sweep's velocity axis run (mass kept, f >= 0), 129 are refused with
    VP_ENOTSUP and f is left as it was."""
    import torch
    w = _t(N.pack(_params(5, 0.3)), torch.float32)
    for nv, ok in ((128, True), (129, False)):
        g = dict(dims=1, nx=[16], nv=[nv], xlo=[0.0], xhi=[4.0], vlo=[-3.0], vhi=[3.0], order=7)
        sim, og = both(g, V.VP_F32)
        f0 = _f32(inputs.random_f(og.NX * og.NV, seed=nv))
        to_gpu(sim, f0)
        if ok:
            V.vp_learned_sweep(sim.ctx, 0, 0, 0.3, None, w, 1)
            f1 = from_gpu(sim)
            assert f1.min() >= 0.0
            assert abs(f1.sum() - f0.sum()) <= 1e-5 * f0.sum()
        else:
            with pytest.raises(V.VpError) as e:
                V.vp_learned_sweep(sim.ctx, 0, 0, 0.3, None, w, 1)
            assert e.value.code == V.VP_ENOTSUP
            assert np.array_equal(from_gpu(sim), f0)
        sim.close()


LINE_CASES = [
    # dims, nx, nv, xbc, kick, dim, dt: strided and contiguous lines, lines shorter than the
    # stencil, whole-cell shifts below and above the direct sum's limit, both boundaries
    (1, [40], [12], 0, 0, 0, 0.3),
    (1, [40], [70], 1, 0, 0, -3.1),
    (1, [3], [20], 0, 0, 0, 5.0),
    (1, [5], [7], 1, 0, 0, 2.9),
    (1, [9], [64], 1, 1, 0, 0.7),
    (1, [33], [40], 0, 1, 0, -4.0),
    (2, [6, 10], [8, 12], 0, 0, 0, 0.4),
    (2, [6, 10], [8, 12], 0, 0, 1, 1.3),
    (2, [5, 4], [16, 9], 1, 1, 0, 0.6),
    (2, [5, 4], [9, 16], 0, 1, 1, 0.8),
    # lines in fours on 16-byte boundaries: open and kicked ones, a ragged last tile
    (2, [6, 10], [8, 12], 1, 0, 0, 0.4),
    (2, [5, 4], [9, 16], 1, 1, 0, 0.6),
    (1, [33], [140], 0, 0, 0, 0.2),
]


@pytest.mark.parametrize("dims,nx,nv,xbc,kick,dim,dt", LINE_CASES)
def test_fluxes_and_samples_of_every_line_kind(dims, nx, nv, xbc, kick, dim, dt):
    """Fine fluxes against the sweep they describe (f' = f + G_left - G_right;
    two FP32 updates and the FP64 masses: 1e-6 of the cells of order one), and
    samples made from them on the same grid: with Gc = G the target is the
    difference of the limited and unlimited masses, zero (to FP32 rounding)
    where the PP limiter cannot bind (nu <= 0.4 on cells within 10%); scale and
    features against numpy's of the same cells."""
    import torch
    g = dict(dims=dims, nx=nx, nv=nv, xlo=[0.0] * dims, xhi=[2.0 + 0.3 * d for d in range(dims)],
             vlo=[-3.0 - 0.5 * d for d in range(dims)], vhi=[2.5] * dims, order=7, xbc=xbc)
    sim = V.Simulation(g, precision=V.VP_F32)
    rng = np.random.default_rng(dims + nx[0])
    f = (1.0 + 0.1 * rng.random(nx + nv)).astype(np.float32)
    acc = rng.uniform(-4.0, 4.0, size=sim.NX)
    axis = dims * kick + dim
    L = f.shape[axis]
    sim.upload(f.reshape(-1))
    a = torch.as_tensor(acc, device="cuda") if kick else None
    lines = f.size // L
    G = torch.empty(lines * (L + 1), dtype=torch.float64, device="cuda")
    V.vp_fine_flux(sim.ctx, kick, dim, dt, a, 1, G)
    X = torch.empty(lines * (L + 1), 25, device="cuda")
    y, sc = torch.empty(lines * (L + 1), device="cuda"), torch.empty(lines * (L + 1), device="cuda")
    torch.cuda.synchronize()
    V.vp_make_samples(sim.ctx, kick, dim, dt, a, G, 0.0, X, y, sc)
    every = 2 if L % 2 == 0 else L
    Ge = torch.empty(lines * (L // every + 1), dtype=torch.float64, device="cuda")
    V.vp_fine_flux(sim.ctx, kick, dim, dt, a, every, Ge)
    if kick:
        V.vp_kick_sweep(sim.ctx, dim, dt, a)
    else:
        V.vp_drift_sweep(sim.ctx, dim, dt)
    sim.sync()
    out = np.moveaxis(sim.f.cpu().numpy().reshape(f.shape), axis, -1).reshape(lines, L).astype(np.float64)
    fl = np.moveaxis(f, axis, -1).reshape(lines, L).astype(np.float64)
    G = G.cpu().numpy().reshape(lines, L + 1)
    assert np.abs(fl + G[:, :-1] - G[:, 1:] - out).max() <= 1e-6
    assert np.array_equal(Ge.cpu().numpy().reshape(lines, -1), G[:, ::every])
    X, y, sc = X.cpu().numpy().reshape(lines, L + 1, 25), y.cpu().numpy().reshape(lines, -1), sc.cpu().numpy().reshape(lines, -1)
    end = not kick and xbc == 0  # the duplicate interface of a periodic line
    if end:
        assert np.isnan(y[:, L]).all() and (X[:, L] == 0).all() and (sc[:, L] == 0).all()
    X, y, sc = X[:, :L], y[:, :L], sc[:, :L]
    ok = X[:, :, 24] <= 0.4
    assert ok.any() and np.abs(y[ok]).max() <= 2e-6
    # speeds, shifts and stencils of every line
    if kick:
        speed = np.repeat(acc, lines // sim.NX)
        h = (g["vhi"][dim] - g["vlo"][dim]) / nv[dim]
    else:
        vc = g["vlo"][dim] + (np.arange(nv[dim]) + 0.5) * (g["vhi"][dim] - g["vlo"][dim]) / nv[dim]
        shape = [1] * (2 * dims)
        shape[dims + dim] = nv[dim]
        speed = np.moveaxis(np.broadcast_to(vc.reshape(shape), f.shape), axis, -1).reshape(lines, L)[:, 0]
        h = (g["xhi"][dim] - g["xlo"][dim]) / nx[dim]
    s = speed * dt / h
    n = np.sign(s) * np.floor(np.abs(s) + 0.5)
    sg = np.where(s - n < 0, -1, 1)
    wrap = not kick and xbc == 0

    def stencil(lines_f):
        i = np.arange(L)[None, :, None]
        up = np.where(sg[:, None, None] > 0, i - 1 - n[:, None, None], i - n[:, None, None]).astype(int)
        r = up + sg[:, None, None] * np.arange(-3, 5)[None, None, :]
        v = np.take_along_axis(lines_f[:, None, :].repeat(L, 1), np.mod(r, L), axis=2)
        return v if wrap else np.where((r >= 0) & (r < L), v, 0.0)
    u = stencil(fl)
    scale = np.abs(u).max(-1) + 1e-30
    assert np.allclose(sc, scale, rtol=1e-6)
    want = np.zeros((lines, L, 25))
    want[:, :, :8] = (u - u[:, :, 3:4]) / scale[:, :, None]
    if not kick:
        z = np.zeros_like(np.take(f, [0], axis=dims + dim))
        hi = np.concatenate([np.take(f, range(1, nv[dim]), axis=dims + dim), z], axis=dims + dim)
        lo = np.concatenate([z, np.take(f, range(nv[dim] - 1), axis=dims + dim)], axis=dims + dim)
        hi, lo = (np.moveaxis(t, axis, -1).reshape(lines, L).astype(np.float64) for t in (hi, lo))
        pos = speed[:, None] >= 0
        p, m = stencil(np.where(pos, hi, lo)), stencil(np.where(pos, lo, hi))
        want[:, :, 8:16] = (p - m) / (2 * scale[:, :, None])
        want[:, :, 16:24] = (0.5 * (p + m) - u) / scale[:, :, None]
    else:
        want[:, :, 16:24] = -u / scale[:, :, None]
    want[:, :, 24] = np.abs(s - n)[:, None]
    assert np.abs(X - want).max() <= 2e-6
    sim.close()


@pytest.mark.parametrize("nf,factors", [((8, 12), (4, 4)), ((6, 15), (3, 5)), ((32, 1), (4, 1)), ((4, 6), (2, 3))])
def test_restriction_and_group_means(nf, factors):
    """Coarse cells and coarse masses against numpy's means: one FP32 rounding
    of an exact mean, and FP64 sums of a few terms."""
    import torch
    rng = np.random.default_rng(nf[0])
    NX, (a, b) = 7, factors
    f = (rng.random((NX, *nf)) * 10.0 ** rng.uniform(-40, 20, size=(NX, *nf))).astype(np.float32)
    ft = torch.as_tensor(f.reshape(-1), device="cuda")
    out = torch.empty(NX * nf[0] // a * (nf[1] // b), device="cuda")
    V.vp_restrict_velocity(ft, out, NX, nf[0], nf[1], a, b)
    want = f.astype(np.float64).reshape(NX, nf[0] // a, a, nf[1] // b, b).mean((2, 4)).reshape(-1)
    torch.cuda.synchronize()
    assert np.allclose(out.cpu().numpy(), want, rtol=2.0 ** -23, atol=1e-44)
    n, nout, grp = 23, 11, a * b
    Gf = rng.standard_normal((40, nout))
    m = rng.integers(0, 40, size=(n, grp))
    Gc = torch.empty(n * nout, dtype=torch.float64, device="cuda")
    V.vp_group_mean(torch.as_tensor(Gf.reshape(-1), device="cuda"), n, nout,
                    torch.as_tensor(m.reshape(-1), dtype=torch.int64, device="cuda"), grp, 0.25, Gc)
    torch.cuda.synchronize()
    assert np.abs(Gc.cpu().numpy().reshape(n, nout) - 0.25 * Gf[m].mean(1)).max() <= 1e-15 * grp


@pytest.mark.parametrize("power", [-112, -99, 60, 99, 112])
def test_sample_targets_at_every_scale_of_f(power):
    """Targets are masses over s, the stencil's largest cell (with a floor): the
    targets of masses Gc less those of no mass are Gc / s in the upwind frame,
    with f and Gc scaled by powers of two to within the fast division's range, to
    its ends and beyond.  FP32 roundings of masses of order s: 1e-6."""
    import torch
    rng = np.random.default_rng(5)
    f = ((1.0 + 0.5 * rng.random((12, 24))) * 2.0 ** power).astype(np.float32)
    G = rng.random((24, 13)) * 2.0 ** power
    sim = V.Simulation(dict(dims=1, nx=[12], nv=[24], xlo=[0.0], xhi=[1.0], vlo=[-3.0], vhi=[2.5], order=7),
                       precision=V.VP_F32)
    sim.upload(f.reshape(-1))

    def targets(Gc):
        X, y = torch.empty(24 * 13, 25, device="cuda"), torch.empty(24 * 13, device="cuda")
        s = torch.empty(24 * 13, device="cuda")
        torch.cuda.synchronize()
        V.vp_make_samples(sim.ctx, 0, 0, 0.02, None, torch.as_tensor(Gc, device="cuda"), 0.0, X, y, s)
        sim.sync()
        return y.cpu().numpy().reshape(24, 13), s.cpu().numpy().reshape(24, 13)
    y1, s = targets(G)
    y0, _ = targets(np.zeros_like(G))
    speed = -3.0 + 5.5 / 24 * (np.arange(24) + 0.5)  # |shift| < 1/2 at nx dt |v| = 0.72 for some, above for others
    shift = speed * 0.02 * 12
    sign = np.where(shift - np.round(shift) < 0, -1.0, 1.0)[:, None]
    ok = ~np.isnan(y1)
    assert ok.any() and np.array_equal(ok, ~np.isnan(y0))
    want = sign * G / np.where(ok, s, 1.0).astype(np.float64)
    size = np.abs(y1[ok]).max() + np.abs(y0[ok]).max()
    assert np.abs(y1.astype(np.float64) - y0 - want)[ok].max() <= 1e-6 * size
    sim.close()


@pytest.mark.parametrize("net", ["he", "positive", "biased"])
@pytest.mark.parametrize("n,group,coef", [(16, 2, True), (250, 1, False), (1003, 1, True), (4000, 2, True),
                                          (32768, 2, True), (100002, 2, False)])
def test_training_loss_and_gradient_to_fp32_rounding(n, group, coef, net):
    """Loss and gradient against the same network in 64 bits, whose activations are
    the bfloat16 roundings of its sums rounded to FP32: no activation may differ
    (one does with a probability of 1e-4 per FP32 sum, and moves the loss of a
    batch by up to 1e-5).  What is left: an output takes 13 FP32 roundings, each
    of at most u = 2^-24 of the sizes of its terms (S, against residuals R), the
    loss a chain of up to 214 additions, the deltas 16 roundings in each of three
    layers.  Independent roundings: six standard deviations."""
    import torch
    dev = "cuda"

    def bf(t):
        return t.to(torch.float32).to(torch.bfloat16).to(torch.float64)
    worst = []
    for seed in range(5):
        gen = torch.Generator(device=dev)
        gen.manual_seed(1000 * seed + n)
        X = 0.3 * torch.randn(n, 25, generator=gen, device=dev)
        X[:, 3] = 0.0
        X[:, 24] = 0.5 * torch.rand(n, generator=gen, device=dev)
        y = 0.02 * torch.randn(n, generator=gen, device=dev)
        c = 0.7 + 0.3 * torch.rand(n, generator=gen, device=dev)
        c[::2] *= -1.0
        w = torch.randn(V.VP_NET_NPARAM, generator=gen, device=dev) * 0.25
        if net == "positive":  # sums whose terms add up
            w, X = 0.25 * w.abs(), X.abs()
        layers, at = [], 0
        for rows, cols in ((32, 25), (32, 32), (32, 32), (1, 32)):
            b = w[at + rows * cols:at + rows * cols + rows]
            b *= 8.0 if net == "biased" else 0.1
            layers.append((bf(w[at:at + rows * cols]).view(rows, cols), b.double()))
            at += rows * cols + rows
        grad, loss = torch.zeros_like(w), torch.zeros(1, device=dev)
        V.vp_net_grad(X, y, n, w, grad, loss, torch.cuda.current_stream(), coef=c if coef else None, group=group)
        a, h = c.double() if coef else torch.ones(n, dtype=torch.float64, device=dev), [bf(X)]
        for k, (W, b) in enumerate(layers):
            z = h[-1] @ W.T + b
            h.append(bf(torch.relu(z)) if k < 3 else z)
        r = (a * (h[4][:, 0] - y.double())).view(-1, group).sum(1)
        want_loss = float((r * r).mean())
        d = (2.0 * r.repeat_interleave(group) * a / r.numel())[:, None]
        parts = []
        for k in (3, 2, 1, 0):
            parts = [(d.T @ h[k]).reshape(-1), d.sum(0)] + parts
            d = (d @ layers[k][0]) * (h[k] > 0) if k else d
        want = torch.cat(parts)
        S = float((a * (h[3] @ layers[3][0].abs().T + layers[3][1].abs())[:, 0].add(y.double().abs())).square().mean().sqrt())
        u, ratio = 2.0 ** -24, S / float(r.square().mean().sqrt())
        tol = 6 * u * (np.sqrt(214) / 3 + 2 * np.sqrt(13 * group / 3) * ratio / np.sqrt(n / group))
        tol_grad = 48 * u + 6 * u * np.sqrt(13 / 3) * ratio
        el = abs(float(loss) - want_loss) / want_loss
        eg = float((grad.double() - want).norm() / want.norm())
        worst.append((el / tol, eg / tol_grad))
    assert max(e for e, _ in worst) <= 1.0 and max(e for _, e in worst) <= 1.0, worst


@pytest.mark.parametrize("factors", [(4, 4), (3, 5), (8, 1)])
def test_restriction_of_cells_whose_sum_leaves_the_float_range(factors):
    """Means of cells up to FLT_MAX are finite: one FP32 rounding of sums in double.
    Cells that are not finite stay so."""
    import torch
    a, b = factors
    rng = np.random.default_rng(a)
    f = (rng.random((5, 2 * a, 3 * b)) * 3.4e38).astype(np.float32)
    f[3, 0, 0], f[4, 0, 0] = np.inf, np.nan
    out = torch.empty(5 * 6, device="cuda")
    V.vp_restrict_velocity(torch.as_tensor(f.reshape(-1), device="cuda"), out, 5, 2 * a, 3 * b, a, b)
    torch.cuda.synchronize()
    want = f.astype(np.float64).reshape(5, 2, a, 3, b).mean((2, 4)).reshape(-1)
    out = out.cpu().numpy().astype(np.float64)
    fine = np.isfinite(want)
    assert (~fine).sum() == 2 and np.isinf(out[18]) and np.isnan(out[24])
    assert (np.abs(out - want)[fine] <= 2.0 ** -23 * want[fine]).all()


@pytest.mark.parametrize("dt", [1.875, -1.875, 5.0])
def test_fine_flux_of_cells_whose_sum_leaves_the_float_range(dt):
    """Masses of several whole cells of 6e37 are finite doubles, as direct sums of a
    few cells and (longer shifts) as differences of prefix sums of a line: where a
    shift is a whole number of cells, the sum of the swept cells, to 40 roundings of
    the sum of a line in double and the rounding of the shift."""
    import torch
    nx, nv = 40, 17
    g = dict(dims=1, nx=[nx], nv=[nv], xlo=[0.0], xhi=[float(nx)], vlo=[-3.4], vhi=[3.4], order=7)
    sim = V.Simulation(g, precision=V.VP_F32)
    rng = np.random.default_rng(3)
    f = ((0.9 + 0.1 * rng.random((nx, nv))) * 6.5e37).astype(np.float32)
    sim.upload(f.reshape(-1))
    G = torch.empty(nv * (nx + 1), dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    V.vp_fine_flux(sim.ctx, 0, 0, dt, None, 1, G)
    sim.sync()
    G = G.cpu().numpy().reshape(nv, nx + 1)
    assert np.isfinite(G).all()
    f = f.astype(np.float64)
    seen = 0.0
    for k in range(nv):
        s = (-3.4 + 0.4 * (k + 0.5)) * dt
        n = int(round(s))
        if abs(s - n) > 1e-9:
            continue
        whole = np.array([sum(f[(j - 1 - m) % nx, k] for m in range(n)) - sum(f[(j + m) % nx, k] for m in range(-n))
                          for j in range(nx + 1)])
        assert np.abs(G[k] - whole).max() <= 40 * 40 * 2.0 ** -53 * 6.5e37 + 1e-13 * 6.5e37
        seen = max(seen, np.abs(whole).max())
    assert seen > 3.5e38
    sim.close()
