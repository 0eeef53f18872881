"""FP64 stage kernel: WENO-5 and the stage's increments in float-float arithmetic on the FP32 pipe.

What can go wrong there and nowhere else: the scaling that brings differences into FP32's range, differences and
indicators that are exactly zero (Table tab:weno), jumps next to rounding noise, and infinities and NaN among the
populations.
"""
import numpy as np
import pytest

from helpers import make_oracle
from paper_1702_01690_gb300 import inputs

pytestmark = pytest.mark.gpu
EPS = float(np.finfo(np.float64).eps)


@pytest.fixture(scope="module")
def olb():
    from paper_1702_01690_gb300 import olb as m
    return m


def _params(nx, ny, side_x=0, **more):
    ds = 1.0 / max(nx, ny)
    return inputs.RunParams(nx=nx, ny=ny, ds=ds, dt=inputs.stable_dt(ds, sigma=more.get("sigma", 1e-4)), tau=5e-3,
                            Tw=(0.9, 0.9), side_x=side_x, **more)


def _populations(olb, p, fields):
    ctx = olb.create(p)
    ctx.init_fields(*fields)
    return ctx.get_populations()


def _step(olb, p, f, steps=1):
    ctx = olb.create(p)
    ctx.set_populations(f)
    ctx.step_async(steps)
    ctx.status()
    return ctx.get_populations()


@pytest.mark.parametrize("shift", [-700, -150, -40, 40, 150, 300])
def test_ideal_gas_step_scales_exactly_with_the_density(olb, shift):
    """a = b = sigma = 0: the step is homogeneous in f, so a power of two goes through it bit for bit, far beyond
    FP32's range too."""
    p = _params(37, 19, a=0.0, b=0.0, sigma=0.0)
    rng = np.random.default_rng(3)
    n = 1.0 + 0.3 * rng.uniform(-1, 1, (p.ny, p.nx))
    u = 0.1 * rng.uniform(-1, 1, (2, p.ny, p.nx))
    f = _populations(olb, p, (n, u[0], u[1], 1.0 + 0.1 * rng.uniform(-1, 1, n.shape)))
    one, other = _step(olb, p, f, 2), _step(olb, p, np.ldexp(f, shift), 2)
    assert np.array_equal(np.ldexp(other, -shift), one)


# one step, three stages; each of about 40 rounded FP64 operations on terms of at most the largest population
# (corrections are good to 2^-42 of the largest difference, times a Courant number below 0.15: less than that)
@pytest.mark.parametrize("nx,ny,side_x", [(9, 8, 0), (8, 8, 1), (17, 3, 1), (65, 9, 0)])
@pytest.mark.parametrize("kind", ["uniform", "ramp", "jump", "jump in noise", "noise of an ulp"])
def test_zero_and_uneven_differences_match_the_oracle(olb, nx, ny, side_x, kind):
    p = _params(nx, ny, side_x)
    rng = np.random.default_rng(5)
    i = np.arange(nx) + 0 * np.arange(ny)[:, None]
    n = {"uniform": 1.0 + 0.0 * i, "ramp": 1.0 + 0.01 * i, "jump": np.where(i < nx // 2, 0.6, 1.4),
         "jump in noise": np.where(i < nx // 2, 0.6, 1.4) + 1e-9 * rng.uniform(-1, 1, i.shape),
         "noise of an ulp": 1.0 + EPS * rng.integers(-1, 2, i.shape)}[kind].astype(float)
    z = np.zeros_like(n)
    fields = (n, z + 0.01, z - 0.02, z + 0.9)
    f = _populations(olb, p, fields)
    o = make_oracle(p, fields)
    o.set_populations(f)
    o.step(1)
    assert np.max(np.abs(_step(olb, p, f) - o.get_populations())) <= 3 * 40 * EPS * np.max(f)


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
def test_infinities_and_nan_reach_their_neighbours(olb, bad):
    """A stencil that holds an infinity or a NaN gives no finite face: the state of a diverged run shows it."""
    p = _params(24, 24, sigma=0.0, a=0.0, b=0.0)
    one = np.ones((p.ny, p.nx))
    f = _populations(olb, p, (one, 0 * one, 0 * one, one))
    f[24, 12, 12] = bad  # xi_x, xi_y > 0: upwind of the faces that follow it
    ctx = olb.create(p)
    ctx.set_populations(f)
    ctx.step_async(1)
    assert ctx.status() == olb.ERR_DIVERGED
    g = ctx.get_populations()
    assert not np.isfinite(g[:, 12, 12]).any()
    assert not np.isfinite(g[24, 12, 10:15]).any() and not np.isfinite(g[24, 10:15, 12]).any()
    assert np.isfinite(g[:, 0, 0]).all()


@pytest.mark.parametrize("precision", [0, 1])
def test_learned_weights_take_their_three_shapes_only(olb, precision):
    ctx = olb.create(_params(24, 24), precision=precision, weno_mode=olb.WENO_LEARNED)
    for shape in ((8, 8, 4), (16, 8, 2), (32, 16, 1)):
        ctx.set_tile(*shape)
        assert ctx.get_tile() == shape
    for shape in ((8, 8, 5), (8, 8, 8), (7, 8, 8), (16, 8, 1), (32, 8, 1), (16, 16, 1)):
        with pytest.raises(olb.OlbError):
            ctx.set_tile(*shape)
        assert ctx.get_tile() == (32, 16, 1)


# a face's arithmetic is that of its stencil, whichever lane and warp takes it and whatever its neighbours are (a
# density within [1, 2) gives every tile one scale): no tolerance
@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("nx,ny", [(9, 8), (24, 16), (65, 9)])
@pytest.mark.parametrize("kind", ["wave", "jump", "jump in noise"])
def test_learned_step_does_not_depend_on_the_tiles(olb, nx, ny, kind, precision):
    from paper_1702_01690_gb300 import learned
    p = _params(nx, ny)
    rng = np.random.default_rng(6)
    i = np.arange(nx) + 0 * np.arange(ny)[:, None]
    n = {"wave": 1.5 + 0.1 * np.sin(2 * np.pi * i / nx), "jump": np.where(i < nx // 2, 1.2, 1.7),
         "jump in noise": np.where(i < nx // 2, 1.2, 1.7) + 1e-9 * rng.uniform(-1, 1, i.shape)}[kind].astype(float)
    z = np.zeros_like(n)

    def run(dx, dy):
        ctx = olb.create(p, precision=precision, weno_mode=olb.WENO_LEARNED)
        ctx.set_weno_mlp(learned.load_theta())
        ctx.init_fields(np.roll(n, (dy, dx), (0, 1)), z + 0.01, z - 0.02, z + 0.9)
        assert ctx.step(2) == 0
        return np.roll(ctx.get_populations(), (-dy, -dx), (1, 2))

    ref = run(0, 0)
    for dx, dy in ((1, 0), (0, 3), (5, 6)):
        assert np.array_equal(run(dx, dy), ref)
