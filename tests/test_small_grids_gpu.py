"""Grids of at most one tile per SM: one launch per stage, whose CTAs take the moments and the force of their tile and
its surroundings themselves, against the three launches of larger grids (a batch with one large run takes those)."""
import numpy as np
import pytest

from helpers import field_rel
from paper_1702_01690_gb300 import inputs

pytestmark = pytest.mark.gpu


# FP64: the same operations (a density within [1, 2) gives every tile one scale), bit for bit.  FP32: a batch rounds its
# stage coefficients on the device, the bound of test_batch_matches_single_contexts
@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("side_x,side_y", [(0, 0), (1, 0), (2, 0), (2, 2), (3, 0), (3, 2)])
def test_one_launch_equals_three(side_x, side_y, precision):
    from paper_1702_01690_gb300 import olb
    runs = []
    for nx, ny in ((192, 160), (3, 3), (8, 8), (9, 4), (24, 16), (37, 5), (5, 61)):
        ds = 1.0 / max(nx, 8)
        p = inputs.RunParams(nx=nx, ny=ny, ds=ds, dt=0.25 * ds / inputs.P_MAX, tau=0.01, Tw=(0.9, 0.95),
                             side_x=side_x, side_y=side_y)
        rng = np.random.default_rng(nx * ny)
        n, u, v, T = rng.uniform(-1, 1, (4, ny, nx))
        runs.append((p, (1.5 + 0.02 * n, 0.02 * u, 0.02 * v, 0.9 + 0.02 * T)))
    b = olb.Batch([p for p, _ in runs], precision)
    for r, (_, f) in enumerate(runs):
        b.init_fields(r, *f)
    assert b.step(3) == 0
    for r, (p, f) in enumerate(runs):
        ctx = olb.create(p, precision)
        ctx.init_fields(*f)
        assert ctx.step(3) == 0
        if precision == 0:
            assert np.array_equal(b.get_populations(r), ctx.get_populations()), (p.nx, p.ny)
        else:
            assert field_rel(b.get_populations(r), ctx.get_populations()) < 1e-6, (p.nx, p.ny)
