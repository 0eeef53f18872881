"""The kernels that grids of more than one tile an SM take (three launches a stage; learned weights in 256 threads a
tile) against the oracle, on ragged grids with every kind of side."""
import numpy as np
import pytest

from helpers import field_rel, make_oracle, moments_rel
from paper_1702_01690_gb300 import inputs, learned

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def olb():
    from paper_1702_01690_gb300 import olb as m
    return m


def _run(nx, ny, side_x, side_y, jump):
    ds = 1.0 / max(nx, ny)
    p = inputs.RunParams(nx=nx, ny=ny, ds=ds, dt=inputs.stable_dt(ds, n_max=2.2), tau=0.01, Tw=(0.85, 0.95),
                         uw=(0.01, -0.02), side_x=side_x, side_y=side_y)
    rng = np.random.default_rng(nx)
    n, u, v, T = rng.uniform(-1, 1, (4, ny, nx))
    # a liquid and its vapour beside it (densities over several binades), or a fluid at one density
    n = np.where(np.arange(nx) < nx // 3, 1.6, 0.05) * (1 + 0.05 * n) if jump else 1.0 + 0.05 * n
    return p, (n, 0.01 * u, 0.01 * v, 0.95 + 0.02 * T)


SIDES = [(0, 0), (1, 0), (2, 2), (3, 2)]


# the tolerances of the oracle comparisons of small grids (test_parity_gpu, test_mlp_gpu); 252 and 255 tiles
@pytest.mark.parametrize("side_x,side_y", SIDES)
@pytest.mark.parametrize("nx,ny", [(141, 109), (35, 403)])
@pytest.mark.parametrize("precision", [0, 1])
def test_step_matches_oracle(olb, nx, ny, side_x, side_y, precision):
    p, fields = _run(nx, ny, side_x, side_y, False)
    ctx = olb.create(p, precision)
    ctx.init_fields(*fields)
    o = make_oracle(p, fields)
    assert ctx.step(3) == 0
    o.step(3)
    tol = 1e-11 if precision == 0 else 1e-5
    assert field_rel(ctx.get_populations(), o.get_populations()) < tol
    assert max(moments_rel(ctx.moments(), o.moments()).values()) < tol


@pytest.mark.parametrize("side_x", [0, 1])
@pytest.mark.parametrize("nx,ny", [(141, 109), (35, 403)])
@pytest.mark.parametrize("precision", [0, 1])
def test_learned_step_matches_oracle(olb, nx, ny, side_x, precision):
    p, fields = _run(nx, ny, side_x, 0, False)
    theta = learned.load_theta()
    ctx = olb.create(p, precision, weno_mode=olb.WENO_LEARNED)
    ctx.set_weno_mlp(theta)
    ctx.init_fields(*fields)
    o = make_oracle(p, fields)
    o.set_mlp(theta.astype(np.float64))
    assert ctx.step(3) == 0
    o.step(3)
    assert max(moments_rel(ctx.moments(), o.moments()).values()) < (1e-6 if precision == 0 else 1e-5)


# a run in its own context (small ones: one launch a stage) and in a batch beside a large one (three).  The scales of
# k_force's blocks differ from those of a tile, which moves what is rounded at 2^-105 of the largest value: one rounding
# of a population, amplified as the oracle's own roundings are (1e-11, the bound against the oracle)
@pytest.mark.parametrize("side_x,side_y", SIDES)
def test_one_launch_and_three_over_binades_of_density(olb, side_x, side_y):
    runs = [_run(nx, ny, side_x, side_y, True) for nx, ny in ((150, 120), (45, 19), (24, 40), (9, 4))]
    b = olb.Batch([p for p, _ in runs])
    for r, (_, f) in enumerate(runs):
        b.init_fields(r, *f)
    b.step(2)
    for r, (p, f) in enumerate(runs):
        ctx = olb.create(p)
        ctx.init_fields(*f)
        ctx.step_async(2)
        ctx.status()
        assert field_rel(ctx.get_populations(), b.get_populations(r)) < 1e-11, (p.nx, p.ny)
