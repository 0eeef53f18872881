"""Densities, populations and units far apart in FP64: the float-float arithmetic of the stage (csrc/olb_ff.cuh,
olb_stage64.cuh) and of the force is scaled into FP32's range tile by tile, and has to hold wherever FP64 does."""
import ctypes

import numpy as np
import pytest

from helpers import make_oracle
from paper_1702_01690_gb300 import inputs

pytestmark = pytest.mark.gpu
EPS = float(np.finfo(np.float64).eps)
SMALL, LARGE = (37, 19), (136, 88)  # 15 tiles: one launch a stage; 187 tiles, more than SMs: three


@pytest.fixture(scope="module")
def olb():
    from paper_1702_01690_gb300 import olb as m
    return m


def _ideal(nx, ny, **more):
    """No van der Waals terms (Delta p = 0): advection and collision only, however large a jump is."""
    ds = 1.0 / max(nx, ny)
    return inputs.RunParams(**{**dict(nx=nx, ny=ny, ds=ds, dt=inputs.stable_dt(ds), tau=5e-3, Tw=(0.9, 0.9), a=0.0, b=0.0,
                                      sigma=0.0), **more})


def _populations(olb, p, fields):
    ctx = olb.create(p)
    ctx.init_fields(*fields)
    return ctx.get_populations()


def _stepped(olb, p, f, steps, how="single", fields=None):
    if how == "batch":
        b = olb.Batch([p, p])
        for r in range(2):
            b.init_fields(r, *fields)
        b.step_async(steps)
        b.status()
        out = b.get_populations(1)
        assert np.array_equal(b.get_populations(0), out, equal_nan=True)
        return out
    if how == "static":
        import torch
        dev = torch.from_numpy(f).cuda().contiguous()
        stream = torch.cuda.current_stream()
        params = olb.params_from(p)
        olb.library().olb_step_static(ctypes.byref(params), ctypes.c_void_p(stream.cuda_stream),
                                      ctypes.c_void_p(dev.data_ptr()), steps)
        return dev.cpu().numpy()
    ctx = olb.create(p)
    ctx.set_populations(f)
    ctx.step_async(steps)
    ctx.status()
    return ctx.get_populations()


# one step, three stages, each of about 40 rounded FP64 operations on terms of at most the largest population
@pytest.mark.parametrize("how", ["single", "batch", "static"])
@pytest.mark.parametrize("nx,ny", [SMALL, LARGE])
@pytest.mark.parametrize("low", [1e-3, 1e-7, 1e-9, 1e-12, 1e-25])
def test_dilute_tiles_beside_dense_ones(olb, nx, ny, low, how):
    """Jumps at the edge of tiles (x = 16, the other across the periodic side) and along y: the faces of a tile reach
    three nodes into the next.  (The status is not asked for: at 1e-25 a stage's n is below the rounding of a node
    beside it, and may be negative.)"""
    p = _ideal(nx, ny)
    i, j = np.arange(nx) + 0 * np.arange(ny)[:, None], 0 * np.arange(nx) + np.arange(ny)[:, None]
    z = np.zeros((ny, nx))
    for dense in (i < 16, j >= 8):
        fields = (np.where(dense, 1.0, low), z + 0.01, z - 0.02, z + 0.9)
        f = _populations(olb, p, fields)
        o = make_oracle(p, (z + 1, z, z, z + 1))
        o.set_populations(f)
        o.step(1)
        assert np.max(np.abs(_stepped(olb, p, f, 1, how, fields) - o.get_populations())) <= 3 * 40 * EPS * np.max(f)


@pytest.mark.parametrize("nx,ny", [SMALL, LARGE])
def test_populations_far_above_their_density(olb, nx, ny):
    """2^30 n of w He_4(p_x) w He_4(p_y), which n, u, T and their fluxes along x do not see, varying along x: the
    populations, not the density, set the scale.  (tau large: no relaxation.)"""
    p = _ideal(nx, ny, tau=1e9)
    rng = np.random.default_rng(4)
    z = np.zeros((ny, nx))
    f = _populations(olb, p, (1.0 + 0.2 * rng.uniform(-1, 1, z.shape), z, z, z + 1.0))
    R = np.array([np.sqrt(5 + s * np.sqrt(10)) for s in (1, -1)] + [0.0])
    h = (np.array([(7 - 2 * np.sqrt(10)) / 60, (7 + 2 * np.sqrt(10)) / 60, 8 / 15]) * (R ** 4 - 6 * R ** 2 + 3))[
        [0, 1, 2, 1, 0]]
    f += np.outer(h, h).reshape(25, 1, 1) * (2.0 ** 30 * (1.0 + 0.2 * rng.uniform(-1, 1, nx)))
    o = make_oracle(p, (z + 1, z, z, z + 1))
    o.set_populations(f)
    o.step(1)
    assert np.max(np.abs(_stepped(olb, p, f, 1) - o.get_populations())) <= 3 * 40 * EPS * np.max(np.abs(f))


def _noisy(p, seed=3):
    rng = np.random.default_rng(seed)
    n, u, v, T = rng.uniform(-1, 1, (4, p.ny, p.nx))
    return 1.0 + 0.3 * n, 0.1 * u, 0.1 * v, 1.0 + 0.1 * T


@pytest.mark.parametrize("shift", [-101, -64, 64, 101, 125])
@pytest.mark.parametrize("nx,ny", [SMALL, LARGE])
def test_units_of_density(olb, nx, ny, shift):
    """The step with n, 1/a, 1/b and 1/sigma in another unit, a power of two: the same bits, capillary term included."""
    p = _ideal(nx, ny, a=9.0 / 8.0, b=1.0 / 3.0, sigma=1e-4)
    q = _ideal(nx, ny, a=np.ldexp(9.0 / 8.0, -shift), b=np.ldexp(1.0 / 3.0, -shift), sigma=np.ldexp(1e-4, -shift))
    f = _populations(olb, p, _noisy(p))
    one, other = _stepped(olb, p, f, 2), _stepped(olb, q, np.ldexp(f, shift), 2)
    assert np.isfinite(one).all()
    assert np.array_equal(np.ldexp(other, -shift), one)


@pytest.mark.parametrize("shift", [900, 950, 1000, 1020])
@pytest.mark.parametrize("nx,ny", [SMALL, LARGE])
def test_largest_densities(olb, nx, ny, shift):
    """An ideal gas up to the end of FP64's range: the same bits."""
    p = _ideal(nx, ny)
    f = _populations(olb, p, _noisy(p))
    one, other = _stepped(olb, p, f, 1), _stepped(olb, p, np.ldexp(f, shift), 1)
    assert np.array_equal(np.ldexp(other, -shift), one)


@pytest.mark.parametrize("precision,learned", [(0, False), (1, False), (0, True), (1, True)])
def test_grids_of_more_rows_than_a_launch_has(olb, precision, learned):
    """65537 tiles along y; the shape (32, 16, 1) has always taken them.  Uniform along y: the moments of eight rows."""
    from paper_1702_01690_gb300 import learned as weights
    out = []
    for ny in (8, 8 * 65535 + 11):
        ds = 1.0 / 64
        p = inputs.RunParams(nx=5, ny=ny, ds=ds, dt=inputs.stable_dt(ds), tau=5e-3, Tw=(0.9, 0.9))
        row = 1.5 + 0.1 * np.sin(2 * np.pi * np.arange(5) / 5)
        n = np.ascontiguousarray(np.broadcast_to(row, (ny, 5)))
        ctx = olb.create(p, precision, weno_mode=olb.WENO_LEARNED if learned else olb.WENO_JS)
        ctx.set_tile(32, 16, 1)
        if learned:
            ctx.set_weno_mlp(weights.load_theta())
        ctx.init_fields(n, 0 * n + 0.05, 0 * n - 0.02, 0 * n + 0.9)
        assert ctx.step(1) == 0
        out.append(ctx.moments())
        ctx.close()
    for small, tall in zip(*out):
        assert np.max(np.abs(tall - small[:1])) <= 1e-6 * np.max(np.abs(small))
        assert precision or learned or np.array_equal(tall, np.broadcast_to(small[:1], tall.shape))
