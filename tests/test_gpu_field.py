"""GPU parity of the velocity moment, the Poisson solver, the diagnostics and
initial conditions against the FP64 oracle."""
import math

import numpy as np
import pytest

import oracle as O
from paper_1702_08521_gb300 import inputs
from paper_1702_08521_gb300 import vlasov as V

from gpu_helpers import both, from_gpu, rel_max, to_gpu

pytestmark = pytest.mark.gpu


def _t(x):
    import torch
    return torch.as_tensor(np.ascontiguousarray(x, dtype=np.float64), device="cuda")


@pytest.mark.parametrize("precision", [V.VP_F32, V.VP_F64])
@pytest.mark.parametrize("dims,nx,nv", [(1, [33], [130]), (2, [6, 5], [12, 20]), (3, [3, 4, 2], [8, 6, 10])])
def test_density_moment(precision, dims, nx, nv):
    g = dict(dims=dims, nx=nx, nv=nv, xlo=[0.0] * dims, xhi=[1.0] * dims, vlo=[-2.0] * dims,
             vhi=[3.0] * dims)
    sim, og = both(g, precision)
    f0 = inputs.random_f(og.NX * og.NV, seed=2).astype(np.float32).astype(np.float64)
    to_gpu(sim, f0)
    V.vp_density_moment(sim.ctx, sim.rho)
    sim.sync()
    rho_g = sim.rho.cpu().numpy()
    rho_o = O.density_moment(og, f0)
    assert rel_max(rho_g, rho_o) <= 1e-13
    sim.close()


@pytest.mark.parametrize("order", [2, 4, 6])
@pytest.mark.parametrize("dims,nx", [(1, [64]), (1, [48]), (2, [16, 12]), (3, [8, 6, 4])])
def test_periodic_poisson(order, dims, nx):
    g = dict(dims=dims, nx=nx, nv=[1] * dims, xlo=[0.0] * dims, xhi=[2.0 + d for d in range(dims)],
             vlo=[-1.0] * dims, vhi=[1.0] * dims, pois_order=order, coupling=-1.0, rho_bg=1.0)
    sim, og = both(g, V.VP_F64)
    rng = np.random.default_rng(order)
    rho = 1.0 + 0.3 * rng.standard_normal(og.NX)
    acc = np.zeros(dims * og.NX)
    phi = np.zeros(og.NX)
    r_t, p_t, a_t = _t(rho), _t(phi), _t(acc)
    V.vp_poisson_solve(sim.ctx, r_t, p_t, a_t)
    sim.sync()
    phi_o, acc_o = O.poisson_solve(og, rho)
    assert rel_max(p_t.cpu().numpy(), phi_o) <= 1e-12
    assert rel_max(a_t.cpu().numpy(), acc_o.reshape(-1)) <= 1e-12
    sim.close()


@pytest.mark.parametrize("n", [6, 8])
def test_isolated_poisson(n):
    h = 0.5
    g = dict(dims=3, nx=[n] * 3, nv=[1] * 3, xlo=[0.0] * 3, xhi=[n * h] * 3, vlo=[-1.0] * 3,
             vhi=[1.0] * 3, poisson=V.VP_POIS_ISOLATED, pois_order=6, coupling=4 * math.pi, rho_bg=0.0)
    sim, og = both(g, V.VP_F64)
    rho = np.random.default_rng(n).random(og.NX)
    p_t, a_t = _t(np.zeros(og.NX)), _t(np.zeros(3 * og.NX))
    V.vp_poisson_solve(sim.ctx, _t(rho), p_t, a_t)
    sim.sync()
    phi_o, acc_o = O.poisson_solve(og, rho)
    assert rel_max(p_t.cpu().numpy(), phi_o) <= 1e-12
    assert rel_max(a_t.cpu().numpy(), acc_o.reshape(-1)) <= 1e-12
    sim.close()


@pytest.mark.parametrize("nx,iso", [([1], 0), ([2], 0), ([37], 0), ([99], 0), ([1024], 0), ([7, 22], 0), ([25, 64], 0),
                                    ([1, 130], 0), ([5, 14, 9], 0), ([16, 2, 33], 0), ([3, 5, 7], 1), ([11, 4, 1], 1)])
def test_poisson_axis_lengths(nx, iso):
    """Axis lengths of every kind the transforms take (1, powers of two and
    four, 3 and 5, larger primes) and the convolution of one dimension, with
    the potential requested, left out, and written over the density.  The
    force differences the potential over a cell, so rounding grows with the
    number of cells of an axis: 1e-12 up to 256 cells, in proportion above."""
    dims, h = len(nx), 0.5
    g = dict(dims=dims, nx=nx, nv=[1] * dims, xlo=[0.0] * dims, xhi=[n * h for n in nx], vlo=[-1.0] * dims,
             vhi=[1.0] * dims, pois_order=6, coupling=4 * math.pi, rho_bg=0.4, poisson=iso)
    sim, og = both(g, V.VP_F64)
    rho = np.random.default_rng(sum(nx)).random(og.NX)
    phi_o, acc_o = O.poisson_solve(og, rho)
    tol = 1e-12 * max(1.0, max(nx) / 256)

    def close(a, b):
        # an axis of one cell has no field: absolute against the density there
        assert np.abs(a.cpu().numpy() - b.reshape(-1)).max() <= tol * max(np.abs(b).max(), 1e-3), nx
    for phi_t in (_t(np.zeros(og.NX)), None, "rho"):
        r_t, a_t = _t(rho), _t(np.zeros(dims * og.NX))
        p_t = r_t if isinstance(phi_t, str) else phi_t
        V.vp_poisson_solve(sim.ctx, r_t, p_t, a_t)
        sim.sync()
        close(a_t, acc_o)
        if p_t is not None:
            close(p_t, phi_o)
    sim.close()


@pytest.mark.parametrize("cfg", [inputs.landau_linear(), inputs.two_stream(32, 64),
                                 inputs.plummer(6, 8)])
def test_initial_conditions_and_diagnostics(cfg):
    prec = V.VP_F64
    sim, og = both(cfg["grid"], prec)
    kind, params = cfg["ic"]
    V.vp_init_f(sim.ctx, kind, params)
    f_g = from_gpu(sim)
    f_o = O.init_f(og, kind, params)
    assert rel_max(f_g, f_o) <= 1e-13
    d_g = V.vp_diagnostics(sim.ctx, 1)
    d_o = O.diagnostics(og, f_o, 1)
    for k in O.DIAG_NAMES:
        assert d_g[k] == pytest.approx(d_o[k], rel=1e-11, abs=1e-14 * (1 + abs(d_o["mass"]))), k
    sim.close()


@pytest.mark.parametrize("cfg", [inputs.two_stream(32, 64), inputs.plummer(6, 8)])
def test_fp32_diagnostics_match_oracle_on_evolved_state(cfg):
    """FP32 f: the moments, energies, extrema and norms (FP64 sums of the FP32
    cells, compensated FP32 partial sums in the velocity moment) against the
    oracle's FP64 diagnostics of the same FP32-rounded state, after a few
    steps so that the state is not an analytic one."""
    sim, og = both(cfg["grid"], V.VP_F32)
    kind, params = cfg["ic"]
    V.vp_init_f(sim.ctx, kind, params)
    sim.field()
    sim.step(cfg["dt"], 3, split=cfg["split"])
    f_g = from_gpu(sim)
    d_g = V.vp_diagnostics(sim.ctx, 1)
    d_o = O.diagnostics(og, f_g, 1)
    for k in O.DIAG_NAMES:
        assert d_g[k] == pytest.approx(d_o[k], rel=1e-9, abs=1e-12 * (1 + abs(d_o["mass"]))), k
    sim.close()


@pytest.mark.parametrize("precision", [V.VP_F32, V.VP_F64])
@pytest.mark.parametrize("nx,nv", [([300], [300]), ([5], [1100]), ([3, 4], [7, 5]), ([4, 2], [3, 260]), ([2, 3, 2], [9, 1, 31])])
def test_diagnostic_sums_over_the_whole_float_range(precision, nx, nv):
    """Mass, kinetic energy, extrema and norms of cells spread over 1e-44 ..
    1e25, some negative, on velocity grids below and above a block, against
    FP64 sums of the same cells.  A thread's pair sum of m cells carries m
    roundings of its error term, m 2^-48 relative to the sum of the terms'
    sizes: below 1e-12 for the m <= 256 of these grids.  Also the density,
    whose cells stay below 1e25 / 1e13 here."""
    D = len(nx)
    g = dict(dims=D, nx=nx, nv=nv, xlo=[0.0] * D, xhi=[1.0] * D, vlo=[-2.0] * D, vhi=[3.0] * D)
    sim, og = both(g, precision)
    rng = np.random.default_rng(sum(nv))
    f = rng.random(og.NX * og.NV) * 10.0 ** rng.uniform(-44, 25, size=og.NX * og.NV)
    f = np.where(rng.random(f.size) < 0.1, -f, f).astype(np.float32).astype(np.float64)
    to_gpu(sim, f)
    d = V.vp_diagnostics(sim.ctx, 1)
    dX, dV = float(np.prod([1.0 / n for n in nx])), float(np.prod([5.0 / n for n in nv]))
    fx = f.reshape([og.NX] + list(nv))
    v2 = sum((np.asarray(og.v_centres(k)) ** 2).reshape([-1 if j == k else 1 for j in range(D)]) for k in range(D))
    terms = dict(mass=fx, ke=0.5 * fx * v2, l1=np.abs(fx), l2=fx ** 2)
    for k, t in terms.items():
        assert abs(d[k] - t.sum() * dX * dV) <= 1e-12 * np.abs(t).sum() * dX * dV, k
    assert d["min_f"] == f.min() and d["max_f"] == f.max()
    V.vp_density_moment(sim.ctx, sim.rho)
    sim.sync()
    rho, size = fx.reshape(og.NX, -1).sum(1) * dV, np.abs(fx).reshape(og.NX, -1).sum(1) * dV
    assert (np.abs(sim.rho.cpu().numpy() - rho) <= 1e-12 * size).all()
    sim.close()


def test_diagnostics_flags_nonfinite():
    g = dict(dims=1, nx=[8], nv=[8], xlo=[0.0], xhi=[1.0], vlo=[-1.0], vhi=[1.0])
    sim, _ = both(g, V.VP_F32)
    f = np.ones(64)
    f[5] = np.nan
    to_gpu(sim, f)
    with pytest.raises(V.VpError) as e:
        V.vp_diagnostics(sim.ctx)
    assert e.value.code == V.VP_ENONFINITE
    sim.close()


@pytest.mark.parametrize("spec", [inputs.plummer(6, 8), inputs.two_stream(64, 64)])
def test_overlapped_launches_on_every_kind_of_stream(spec):
    """The same kernels in the same order give the same bits: steps on a stream
    of their own (launches overlap the kernel before them) and on the default
    stream (they do not), and a solve captured behind a copy and replayed."""
    import torch
    out = []
    for stream in (torch.cuda.Stream(), torch.cuda.default_stream()):
        sim = V.Simulation(dict(spec["grid"]), V.VP_F64, stream=stream)
        V.vp_init_f(sim.ctx, *spec["ic"])
        sim.field()
        sim.step(spec["dt"], 4, split=spec["split"])
        sim.field()
        sim.sync()
        out.append((sim.f.clone(), sim.accel.clone(), sim.rho.clone()))
        grid = V.make_grid(**{**spec["grid"], "poisson": V.VP_POIS_PERIODIC, "precision": V.VP_F64})
        sim.close()
    for a, b in zip(*out):
        assert torch.equal(a, b)
    rho = out[0][2]
    src, phi, acc = torch.empty_like(rho), torch.zeros_like(rho), torch.zeros_like(out[0][1])
    s, graph = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    src.copy_(rho)
    assert V.vp_poisson_periodic_noalloc(grid, s, src, phi, acc) == V.VP_OK
    torch.cuda.synchronize()
    want = (phi.clone(), acc.clone())
    src.zero_(), phi.zero_(), acc.zero_()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph, stream=s):
        src.copy_(rho)
        assert V.vp_poisson_periodic_noalloc(grid, s, src, phi, acc) == V.VP_OK
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(phi, want[0]) and torch.equal(acc, want[1])


@pytest.mark.parametrize("nv", [[7], [128], [999], [2048], [2049], [33, 70], [128, 128]])
@pytest.mark.parametrize("scale", [1.0, 2.9e38, 1e-40])
def test_density_of_fp32_cells_of_any_size(nv, scale):
    """Densities of FP32 grids at scales whose sums leave the float range (and of
    subnormal cells), against exact sums.  A thread's float-pair sums of up to 16
    cells are off by at most 16 roundings of their error term, 16 2^-51 of the sum,
    its error terms of n cells by n / 16 such; doubles beyond that."""
    import math
    D, NX = len(nv), [3] * len(nv)
    g = dict(dims=D, nx=NX, nv=nv, xlo=[0.0] * D, xhi=[1.0] * D, vlo=[0.0] * D, vhi=[float(n) for n in nv])
    sim, og = both(g, V.VP_F32)
    rng = np.random.default_rng(nv[0])
    v = np.arange(og.NV) / og.NV - 0.5
    f = ((rng.random((og.NX, 1)) + 0.1) * np.exp(-20 * v * v) * (0.9 + 0.1 * rng.random((og.NX, og.NV))) / 1.1 * scale)
    f = f.astype(np.float32)
    to_gpu(sim, f)
    V.vp_density_moment(sim.ctx, sim.rho)
    sim.sync()
    rho = sim.rho.cpu().numpy()
    want = np.array([math.fsum(r) for r in f.astype(np.float64)])
    assert np.isfinite(rho).all()
    tol = max(16, og.NV // 32 / 16) * 2.0 ** -51 + 2.0 ** -50
    assert (np.abs(rho - want) <= tol * want).all(), np.abs(rho / want - 1).max()
    # independent roundings of every pair sum: 6 standard deviations of the mean square
    rms = np.sqrt(np.mean((rho / want - 1) ** 2))
    assert rms <= 6 * (2.0 ** -51 * 16 / np.sqrt(12 * max(1, min(og.NV, 32))) + 2.0 ** -53), rms
    f[1, 0] = np.inf
    to_gpu(sim, f)
    V.vp_density_moment(sim.ctx, sim.rho)
    sim.sync()
    bad = np.isnan(sim.rho.cpu().numpy())
    assert bad[1] and bad.sum() == 1
    sim.close()


@pytest.mark.parametrize("nx,nv", [([5], [128]), ([3], [5000]), ([2, 3], [64, 64]), ([4], [4099]), ([2, 2, 2], [32, 32, 32]), ([2, 1, 2], [9, 20, 33])])
@pytest.mark.parametrize("kind", ["large", "order one", "tiny", "straddling", "mixed points"])
def test_fp32_diagnostic_sums_as_float_pairs(nx, nv, kind):
    """Sums of FP32 cells that stay below the size at which a point is summed in
    double: all near that size (their squares leave the float range in sums of a few
    hundred), of order one, all tiny, on both sides of the scaled class's limit, and
    some points above it beside others below.  Pair sums of up to 19 cells: 19
    roundings of their error term, 2^-51 each, and weights of 48 bits; independent
    over the grid's runs of 16 cells where every term is positive: six standard
    deviations, and two roundings of the double result."""
    import math
    D = len(nx)
    g = dict(dims=D, nx=nx, nv=nv, xlo=[0.0] * D, xhi=[1.0] * D, vlo=[-2.0] * D, vhi=[3.0] * D)
    sim, og = both(g, V.VP_F32)
    rng = np.random.default_rng(sum(nv) + len(kind))
    shape = (og.NX, og.NV)
    f = rng.random(shape) + 0.1
    if kind == "large":
        f = 1e18 * f
    elif kind == "tiny":
        f = f * 10.0 ** rng.uniform(-40, -20, size=shape)
    elif kind == "straddling":
        f = np.where(rng.random(shape) < 0.2, -f, f) * 2.0 ** rng.uniform(-60, -40, size=shape)
    elif kind == "mixed points":
        f[::2] *= 10.0 ** rng.uniform(16, 25, size=(f[::2].shape[0], 1))
    f = f.astype(np.float32)
    to_gpu(sim, f)
    d = V.vp_diagnostics(sim.ctx, 1)
    dX, dV = float(np.prod([1.0 / n for n in nx])), float(np.prod([5.0 / n for n in nv]))
    fx = f.astype(np.float64).reshape([og.NX] + list(nv))
    v2 = sum((np.asarray(og.v_centres(k)) ** 2).reshape([-1 if j == k else 1 for j in range(D)]) for k in range(D))
    terms = dict(mass=fx, ke=0.5 * fx * v2, l1=np.abs(fx), l2=fx ** 2)
    for k, t in terms.items():
        size = math.fsum(np.abs(t).reshape(-1)) * dX * dV
        off = abs(d[k] - math.fsum(t.reshape(-1)) * dX * dV) / size
        assert off <= 19 * 2.0 ** -51 + 2.0 ** -47, (k, off)
        if kind == "order one":
            weights = 2.0 ** -48 if k == "ke" else 0.0
            assert off <= 6 * (16 * 2.0 ** -51 + weights) / np.sqrt(12 * max(1, fx.size / 16)) + 2.0 ** -51, (k, off)
    assert d["min_f"] == f.min() and d["max_f"] == f.max()
    sim.close()


@pytest.mark.parametrize("n", [7, 64, 300])
@pytest.mark.parametrize("order", [2, 6])
def test_field_of_a_density_on_a_large_background(n, order):
    """One dimension: a uniform density has no field at all, and a variation on a
    background 1e6 times as large has its own field to 1e-12 of the sizes of its
    convolution's terms (the kernels' own 2 n roundings of sums of n terms)."""
    ld = np.longdouble
    pi = ld("3.14159265358979323846264338327950288")
    L, S = 4.0, -1.5
    g = dict(dims=1, nx=[n], nv=[8], xlo=[0.0], xhi=[L], vlo=[-1.0], vhi=[1.0], pois_order=order, coupling=S, rho_bg=1.0)
    th, h = 2 * pi * np.arange(n).astype(ld) / n, ld(L) / n
    b, den = {2: ([1], 1), 6: ([270, -27, 2], 180)}[order]
    c, fden = {2: ([1], 2), 6: ([45, -9, 1], 60)}[order]
    lam = sum(-4 * ld(x) * np.sin((m + 1) * th / 2) ** 2 for m, x in enumerate(b)) / den / h ** 2
    green = np.concatenate([[ld(0)], ld(S) / lam[1:] / n])
    sym = sum(2 * ld(x) * np.sin((m + 1) * th) for m, x in enumerate(c)) / (fden * h)
    j = np.arange(n)
    ang = 2 * pi * ((j[:, None] * j) % n).astype(ld) / n
    shift = (j[:, None] - j) % n
    kernels = [(green * np.cos(ang)).sum(1)[shift], (green * sym * np.sin(ang)).sum(1)[shift]]
    rng = np.random.default_rng(n)
    sim, _ = both(g, V.VP_F64)
    for rho in (np.full(n, 1e6 + 0.1), 1e6 + np.cos(2 * np.pi * j / n) + 0.1 * rng.standard_normal(n)):
        sim.rho.copy_(sim.torch.as_tensor(rho))
        sim.torch.cuda.synchronize()
        V.vp_poisson_solve(sim.ctx, sim.rho, sim.phi, sim.accel)
        sim.sync()
        r = rho.astype(ld) - np.median(rho[[0, n // 3, 2 * (n // 3)]])
        for out, K in zip((sim.phi, sim.accel), kernels):
            off = np.abs(out.cpu().numpy() - K @ r)
            assert (off <= 1e-12 * (np.abs(K) @ np.abs(r))).all(), off.max()
    sim.close()
