"""GPU parity of the advection sweeps against the FP64 oracle (through the
C ABI).  FP64 sweeps must agree to 1e-12 relative per sweep; FP32 sweeps
within 2e-6 relative L1 per sweep (single rounding of f plus FP32
arithmetic); integer shifts are exact; f >= 0 is kept exactly."""
import math

import numpy as np
import pytest

import oracle as O
from paper_1702_08521_gb300 import inputs
from paper_1702_08521_gb300 import vlasov as V

from gpu_helpers import accel_tensor, both, from_gpu, rel_l1, rel_max, to_gpu

pytestmark = pytest.mark.gpu


def grid(dims, nx, nv, **kw):
    xhi = [2.0 + 0.37 * d for d in range(dims)]
    return dict(dims=dims, nx=nx, nv=nv, xlo=[0.0] * dims, xhi=xhi,
                vlo=[-3.0 - 0.5 * d for d in range(dims)], vhi=[2.5 + 0.25 * d for d in range(dims)],
                **kw)


CASES = [
    # ragged sizes spanning several tiles along both the line and across lines
    (1, [37], [45]),
    (1, [64], [130]),
    (1, [300], [33]),
    (1, [6], [1024]),  # long contiguous lines: few lines per CTA, many segments
    (1, [4096], [20]),  # long strided lines (the 4096-cell limit): tiles narrower than a warp
    (2, [9, 7], [10, 12]),
    (2, [16, 5], [33, 8]),
    (3, [5, 6, 4], [6, 5, 8]),
]


@pytest.mark.parametrize("dims,nx,nv", CASES)
@pytest.mark.parametrize("order", [5, 7])
@pytest.mark.parametrize("xbc", [0, 1])
def test_fp64_sweeps_match_oracle(dims, nx, nv, order, xbc):
    g = grid(dims, nx, nv, order=order, xbc=xbc)
    sim, og = both(g, V.VP_F64)
    f0 = inputs.random_f(og.NX * og.NV, seed=17 + dims)
    NX = og.NX
    acc = inputs.random_accel(NX, dims, seed=5, amax=7.0)
    rng = np.random.default_rng(3)
    for rep in range(2):
        for kick in (0, 1):
            for d in range(dims):
                dt = float(rng.uniform(-0.9, 0.9))
                f_o = f0.copy()
                to_gpu(sim, f0)
                if kick:
                    O.kick_sweep(og, f_o, d, dt, acc[d])
                    V.vp_kick_sweep(sim.ctx, d, dt, accel_tensor(sim, acc[d]))
                else:
                    O.drift_sweep(og, f_o, d, dt)
                    V.vp_drift_sweep(sim.ctx, d, dt)
                f_g = from_gpu(sim)
                assert rel_max(f_g, f_o) <= 1e-12, (kick, d, dt, rel_max(f_g, f_o))
    sim.close()


TMA_CASES = [
    # every strided sweep eligible for the TMA kernel (inner % 4 == 0), with
    # ragged column tiles and lines up to the 256-cell box limit
    (1, [37], [132]),
    (1, [256], [36]),
    (2, [9, 7], [12, 20]),
    (3, [5, 3, 4], [8, 4, 12]),
]


@pytest.mark.parametrize("dims,nx,nv", TMA_CASES)
@pytest.mark.parametrize("impl", [1, 2, 3])
@pytest.mark.parametrize("precision", [V.VP_F64, V.VP_F32])
def test_sweep_kernels_agree_with_oracle(dims, nx, nv, impl, precision):
    """The strided-axis kernels (staged loads, TMA pipeline, staged loads with
    two lines per thread) against the oracle, with the autotuner on (it must
    leave f untouched)."""
    g = grid(dims, nx, nv, order=7, xbc=1 if dims == 3 else 0)
    sim, og = both(g, precision)
    V.vp_set_option(sim.ctx, V.VP_OPT_SWEEP_IMPL, impl)
    f0 = inputs.random_f(og.NX * og.NV, seed=23).astype(np.float32).astype(np.float64)
    acc = inputs.random_accel(og.NX, dims, seed=8, amax=6.0)
    tol_max = 1e-12 if precision == V.VP_F64 else None
    for kick in (0, 1):
        for d in range(dims):
            f_o = f0.copy()
            to_gpu(sim, f0)
            if kick:
                O.kick_sweep(og, f_o, d, 0.53, acc[d])
                V.vp_kick_sweep(sim.ctx, d, 0.53, accel_tensor(sim, acc[d]))
            else:
                O.drift_sweep(og, f_o, d, 0.71)
                V.vp_drift_sweep(sim.ctx, d, 0.71)
            f_g = from_gpu(sim)
            if tol_max:
                assert rel_max(f_g, f_o) <= tol_max, (kick, d)
            else:
                assert rel_l1(f_g, f_o) <= 2e-6, (kick, d)
            tu = V.vp_get_tuning(sim.ctx, kick, d)
            assert tu["impl"] in (1, 2, 3)
            if impl == 1:
                assert tu["impl"] == 1
    sim.close()


@pytest.mark.parametrize("mp,pp", [(0, 0), (1, 0), (0, 1)])
def test_fp64_limiter_switches(mp, pp):
    g = grid(2, [12, 9], [20, 17], order=7, mp=mp, pp=pp)
    sim, og = both(g, V.VP_F64)
    f0 = inputs.random_f(og.NX * og.NV, seed=99)
    for d in range(2):
        f_o = f0.copy()
        to_gpu(sim, f0)
        O.drift_sweep(og, f_o, d, 0.37)
        V.vp_drift_sweep(sim.ctx, d, 0.37)
        assert rel_max(from_gpu(sim), f_o) <= 1e-12
    sim.close()


@pytest.mark.parametrize("dims,nx,nv", CASES[:5])
def test_fp32_sweeps_match_oracle(dims, nx, nv):
    g = grid(dims, nx, nv, order=7)
    sim, og = both(g, V.VP_F32)
    # inputs representable in float so both sides start from the same f
    f0 = inputs.random_f(og.NX * og.NV, seed=7).astype(np.float32).astype(np.float64)
    acc = inputs.random_accel(og.NX, dims, seed=6, amax=5.0)
    for kick in (0, 1):
        for d in range(dims):
            f_o = f0.copy()
            to_gpu(sim, f0)
            if kick:
                O.kick_sweep(og, f_o, d, 0.61, acc[d])
                V.vp_kick_sweep(sim.ctx, d, 0.61, accel_tensor(sim, acc[d]))
            else:
                O.drift_sweep(og, f_o, d, -0.43)
                V.vp_drift_sweep(sim.ctx, d, -0.43)
            f_g = from_gpu(sim)
            assert rel_l1(f_g, f_o) <= 2e-6, (kick, d, rel_l1(f_g, f_o))
            assert f_g.min() >= 0.0
    sim.close()


@pytest.mark.parametrize("precision", [V.VP_F32, V.VP_F64])
def test_integer_shift_is_exact_on_gpu(precision):
    # dyadic box and dt: s = v dt / h is an exact integer for every velocity
    n, nv = 32, 8
    g = dict(dims=1, nx=[n], nv=[nv], xlo=[0.0], xhi=[1.0], vlo=[-4.0], vhi=[4.0], order=7)
    sim, og = both(g, precision)
    f0 = inputs.random_f(n * nv, seed=1).astype(np.float32).astype(np.float64)
    to_gpu(sim, f0)
    # v = -3.5 .. 3.5 step 1; h = 1/32; dt = 1/16 -> s = 2 v: odd integers
    V.vp_drift_sweep(sim.ctx, 0, 1.0 / 16.0)
    f_g = from_gpu(sim).reshape(n, nv)
    v = og.v_centres(0)
    want = np.stack([np.roll(f0.reshape(n, nv)[:, j], int(round(2 * v[j]))) for j in range(nv)], axis=1)
    assert np.array_equal(f_g, want)
    sim.close()


def test_positivity_and_mass_fp32():
    g = grid(2, [24, 20], [40, 36], order=7)
    sim, og = both(g, V.VP_F32)
    f0 = (inputs.random_f(og.NX * og.NV, seed=44, zeros=0.5) ** 6).astype(np.float32)
    to_gpu(sim, f0)
    m0 = float(np.sum(f0, dtype=np.float64))
    for _ in range(5):
        for d in range(2):
            V.vp_drift_sweep(sim.ctx, d, 0.77)
    f_g = from_gpu(sim)
    assert f_g.min() >= 0.0
    assert abs(f_g.sum() - m0) / m0 < 1e-6
    sim.close()


def test_sweep_rejects_bad_arguments():
    g = grid(1, [16], [16])
    sim, _ = both(g, V.VP_F32)
    with pytest.raises(V.VpError):
        V.vp_drift_sweep(sim.ctx, 1, 0.1)
    with pytest.raises(V.VpError):
        V.vp_drift_sweep(sim.ctx, 0, float("nan"))
    with pytest.raises(V.VpError):
        V.vp_kick_sweep(sim.ctx, 0, 0.1, None)
    sim.close()


@pytest.mark.parametrize("dims,nx,nv", [(2, [8, 8], [16, 16]), (1, [64], [96]), (1, [2048], [64])])
def test_sweep_bits_do_not_depend_on_tuning(dims, nx, nv):
    """Every sweep gives the same bits whatever kernel, tile width and
    segment count runs it: each implementation with the default tiles, and
    three independently autotuned contexts (timing-based choices)."""
    L = 4 * math.pi
    g = dict(dims=dims, nx=nx, nv=nv, xlo=[0.0] * dims, xhi=[L] * dims, vlo=[-6.0] * dims, vhi=[6.0] * dims,
             order=7)
    n = int(np.prod(nx)) * int(np.prod(nv))
    f0 = (inputs.random_f(n, seed=21, zeros=0.3) ** 2).astype(np.float32)
    setups = [(0, 0), (1, 0), (2, 0), (3, 0), (0, 1), (0, 1), (1, 1), (3, 1)]  # (sweep impl, autotune)
    sweeps = [(1, d) for d in range(dims)] + [(0, d) for d in range(dims)]
    results = []
    for impl, tune in setups:
        out = []
        for kick, d in sweeps:
            sim, _ = both(g, V.VP_F32)
            V.vp_set_option(sim.ctx, V.VP_OPT_SWEEP_IMPL, impl)
            V.vp_set_option(sim.ctx, V.VP_OPT_AUTOTUNE, tune)
            to_gpu(sim, f0)
            sim.field()
            if kick:
                V.vp_kick_sweep(sim.ctx, d, 0.13, sim.accel[d * sim.NX:])
            else:
                V.vp_drift_sweep(sim.ctx, d, 0.37)
            out.append(from_gpu(sim))
            sim.close()
        results.append(out)
    for out in results[1:]:
        for a, b in zip(out, results[0]):
            assert np.array_equal(a, b)


@pytest.mark.parametrize("dims,nx,nv", [(1, [40], [48]), (2, [9, 8], [12, 16])])
def test_fp32_positivity_exact_down_to_subnormals(dims, nx, nv):
    """FP32 cells spread log-uniformly over 1e-45 .. 1 (many subnormal, some
    exactly 0) and lines of subnormals only: after 30 sweeps of every kind with
    random time steps f stays >= 0 exactly (the PP limiter in mass form with
    rounded-down half cells), and the state matches the FP64 oracle run from
    the same FP32 values within the FP32 sweep tolerance."""
    g = grid(dims, nx, nv, order=7, xbc=0)
    sim, og = both(g, V.VP_F32)
    rng = np.random.default_rng(71)
    n = og.NX * og.NV
    f0 = inputs.random_f(n, seed=72) * 10.0 ** rng.uniform(-45, 0, size=n)
    f0 = f0.reshape(og.shape)
    # whole spatial lines of subnormals only
    f0[0] = rng.random(f0[0].shape) * 1e-39
    f0 = f0.reshape(-1).astype(np.float32).astype(np.float64)
    acc = inputs.random_accel(og.NX, dims, seed=73, amax=5.0)
    to_gpu(sim, f0)
    f_o = f0.copy()
    for _ in range(30):
        kick = int(rng.integers(0, 2))
        d = int(rng.integers(0, dims))
        dt = float(rng.uniform(-0.8, 0.8))
        if kick:
            V.vp_kick_sweep(sim.ctx, d, dt, accel_tensor(sim, acc[d]))
            O.kick_sweep(og, f_o, d, dt, acc[d])
        else:
            V.vp_drift_sweep(sim.ctx, d, dt)
            O.drift_sweep(og, f_o, d, dt)
        f_g = from_gpu(sim)
        assert f_g.min() >= 0.0
    assert rel_l1(f_g, f_o) <= 1e-5
    sim.close()


def _with_specials(rng, shape):
    """Non-negative cells of every size, with zeros of both signs, numbers near
    both ends of the range, infinities and NaN scattered among them."""
    f = rng.random(shape) * 10.0 ** rng.uniform(-320, 299, size=shape)
    f[rng.random(shape) < 0.2] = 0.0
    for v in (-0.0, 5e-324, 1e299, 1e302, 1.7e308, np.inf, np.nan, -1e303):
        f[rng.random(shape) < 0.004] = v
    return f


@pytest.mark.parametrize("order", [5, 7])
@pytest.mark.parametrize("xbc", [0, 1])
@pytest.mark.parametrize("n,nv", [(40, 16), (64, 48)])
def test_fp64_integer_comparisons_give_the_plain_result(order, xbc, n, nv):
    """The staged FP64 kernels order doubles by their bits and repeat a segment
    in plain double where a cell is not finite or nearly overflows: the same
    numbers as the TMA kernel, which computes in plain double throughout, on
    ordinary data and on data full of special values.  Strided lines directly;
    contiguous lines against strided copies of them on a grid with a second
    velocity axis."""
    rng = np.random.default_rng(order + nv)
    g1 = dict(dims=1, nx=[n], nv=[nv], xlo=[0.0], xhi=[1.0], vlo=[-3.0], vhi=[2.5], order=order, xbc=xbc)
    g2 = dict(dims=2, nx=[n, 1], nv=[nv, 16], xlo=[0.0, 0.0], xhi=[1.0, 1.0], vlo=[-3.0, 0.0], vhi=[2.5, 1.0],
              order=order, xbc=xbc)
    acc = rng.uniform(-2.0, 2.0, size=n)

    def run(g, impl, f0, kick):
        sim, _ = both(g, V.VP_F64)
        V.vp_set_option(sim.ctx, V.VP_OPT_SWEEP_IMPL, impl)
        to_gpu(sim, f0)
        if kick:
            V.vp_kick_sweep(sim.ctx, 0, 0.31, accel_tensor(sim, acc))
        else:
            V.vp_drift_sweep(sim.ctx, 0, 0.017)
        out, impl_used = from_gpu(sim), V.vp_get_tuning(sim.ctx, kick, 0)["impl"]
        sim.close()
        return out, impl_used
    for f0 in (inputs.random_f(n * nv, seed=5).reshape(n, nv), _with_specials(rng, (n, nv))):
        wide = np.repeat(f0[:, :, None], 16, axis=2)
        ref, used = run(g1, 2, f0, 0)
        assert used == 2
        got, used = run(g1, 1, f0, 0)
        assert used == 1 and np.array_equal(got, ref, equal_nan=True)
        ref, used = run(g2, 2, wide, 1)
        assert used == 2
        ref = ref.reshape(n, nv, 16)[:, :, 0].reshape(-1)
        got, _ = run(g1, 1, f0, 1)
        assert np.array_equal(got, ref, equal_nan=True)


@pytest.mark.parametrize("precision", [V.VP_F32, V.VP_F64])
@pytest.mark.parametrize("dims,nx,nv", [(2, [12, 10], [40, 36]), (1, [200], [150])])
def test_flat_votes_of_blocks_give_the_same_bits(precision, dims, nx, nv):
    """The walkers vote once per block of steps on flat stencils, and tuned
    contexts may leave the vote out: data with empty regions, plateaus of every
    length down to one cell and steps between them give the same bits with the
    default kernels and with tuned ones, for every sweep (tuned on smooth data
    first, where leaving the vote out wins, then run on the plateaus)."""
    rng = np.random.default_rng(9)
    n = int(np.prod(nx)) * int(np.prod(nv))
    runs = np.repeat(rng.random(n), rng.integers(1, 30, size=n))[:n]
    runs[rng.random(n) < 0.02] = 0.0
    f0 = (runs * (rng.random(n) < 0.97) * np.repeat(rng.random(n // 50 + 1) < 0.6, 50)[:n]).astype(np.float32)
    f0 = f0.reshape(list(nx) + list(nv))
    smooth = np.ones(f0.shape)
    for k, m in enumerate(f0.shape):
        smooth = smooth * (1.5 + np.cos(2 * np.pi * (np.arange(m) + 0.5) / m)).reshape([-1 if j == k else 1 for j in range(f0.ndim)])
    g = grid(dims, nx, nv, order=7)
    acc = inputs.random_accel(int(np.prod(nx)), dims, seed=3, amax=3.0)
    for axis in range(2 * dims):
        kick, d = axis // dims, axis % dims
        f = np.ascontiguousarray(np.moveaxis(np.sort(np.moveaxis(f0, axis, -1), axis=-1)[..., ::-1], -1, axis)) if d else f0
        out = []
        for tune in (0, 1):
            sim, _ = both(g, precision)
            V.vp_set_option(sim.ctx, V.VP_OPT_AUTOTUNE, tune)
            for data in (smooth, f):
                to_gpu(sim, data)
                if kick:
                    V.vp_kick_sweep(sim.ctx, d, 0.21, accel_tensor(sim, acc[d]))
                else:
                    V.vp_drift_sweep(sim.ctx, d, 0.047)
            out.append(from_gpu(sim))
            sim.close()
        assert np.array_equal(out[0], out[1]), (kick, d)


@pytest.mark.parametrize("precision", [V.VP_F32, V.VP_F64])
@pytest.mark.parametrize("nx,nv", [([3, 5], [9, 6]), ([7, 1], [21, 2]), ([2, 3], [33, 30]), ([5, 3], [12, 7])])
def test_blocks_side_by_side_and_rows_of_every_width(precision, nx, nv):
    """Narrow outer blocks packed side by side in one tile (a last tile with
    fewer), rows of 16-, 8- and 4-byte pieces, contiguous lines whose 16-byte
    pieces straddle two lines: default and tuned kernels, one and two lines per
    thread, give the same bits, and those of FP64 match the oracle."""
    g = grid(2, nx, nv, order=7, xbc=1)
    og = O.grid(**g)
    f0 = inputs.random_f(og.NX * og.NV, seed=nv[0]).astype(np.float32).astype(np.float64)
    acc = inputs.random_accel(og.NX, 2, seed=2, amax=6.0)
    for kick in (0, 1):
        for d in range(2):
            out = []
            for impl, tune in ((0, 0), (1, 0), (0, 1), (1, 1)):
                sim, _ = both(g, precision)
                V.vp_set_option(sim.ctx, V.VP_OPT_SWEEP_IMPL, impl)
                V.vp_set_option(sim.ctx, V.VP_OPT_AUTOTUNE, tune)
                to_gpu(sim, f0)
                if kick:
                    V.vp_kick_sweep(sim.ctx, d, 0.43, accel_tensor(sim, acc[d]))
                else:
                    V.vp_drift_sweep(sim.ctx, d, 0.29)
                out.append(from_gpu(sim))
                sim.close()
            assert all(np.array_equal(a, out[0]) for a in out[1:]), (kick, d)
            f_o = f0.copy()
            if kick:
                O.kick_sweep(og, f_o, d, 0.43, acc[d])
            else:
                O.drift_sweep(og, f_o, d, 0.29)
            assert rel_l1(out[0], f_o) <= (2e-6 if precision == V.VP_F32 else 1e-12)


@pytest.mark.parametrize("precision,n", [(V.VP_F32, 12000), (V.VP_F32, 20000), (V.VP_F64, 5000), (V.VP_F64, 9000)])
@pytest.mark.parametrize("tune", [0, 1])
def test_long_lines_in_blocks_of_two_columns(precision, n, tune):
    """Strided lines whose tile of two columns fits shared memory but one of four does
    not (and ones where four just fit): the same cells as contiguous lines of a grid of
    one velocity dimension, kicked by the same accelerations."""
    import torch
    rng = np.random.default_rng(n)
    f = inputs.random_f(6 * n * 2, seed=n).reshape(6, n, 2)
    f = f.astype(np.float32 if precision == V.VP_F32 else np.float64)
    acc = rng.uniform(-3.0, 3.0, size=6)
    g2 = dict(dims=2, nx=[3, 2], nv=[n, 2], xlo=[0.0] * 2, xhi=[1.0] * 2, vlo=[-2.0] * 2, vhi=[3.0] * 2, order=7)
    sim = V.Simulation(g2, precision=precision)
    V.vp_set_option(sim.ctx, 2, tune)
    sim.upload(f.reshape(-1))
    V.vp_kick_sweep(sim.ctx, 0, 0.0021, torch.as_tensor(acc, device="cuda"))
    sim.sync()
    got = sim.f.cpu().numpy().reshape(6, n, 2)
    sim.close()
    g1 = dict(dims=1, nx=[12], nv=[n], xlo=[0.0], xhi=[1.0], vlo=[-2.0], vhi=[3.0], order=7)
    sim = V.Simulation(g1, precision=precision)
    V.vp_set_option(sim.ctx, 2, 0)
    sim.upload(np.ascontiguousarray(f.transpose(0, 2, 1)).reshape(-1))
    V.vp_kick_sweep(sim.ctx, 0, 0.0021, torch.as_tensor(np.repeat(acc, 2), device="cuda"))
    sim.sync()
    want = sim.f.cpu().numpy().reshape(6, 2, n).transpose(0, 2, 1)
    sim.close()
    assert not np.array_equal(want, f) and np.array_equal(got, want)
