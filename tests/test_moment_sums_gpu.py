"""Moments of given populations: the sums over a node in fixed point (csrc/olb_kernels.cuh) round to nearest, so that
they have no bias."""
import math

import numpy as np
import pytest

from paper_1702_01690_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def olb():
    from paper_1702_01690_gb300 import olb as m
    return m


def _context(olb, precision, nx=128, ny=128):
    ds = 1.0 / nx
    return olb.create(inputs.RunParams(nx=nx, ny=ny, ds=ds, dt=inputs.stable_dt(ds), tau=5e-3), precision)


# Rounding to nearest: an error of each node of at most half an ulp of n (2^-53 n) for the sum as a double and 25
# times half of 2^-57 of the binade above the largest population, of either sign; its mean over N nodes is within six
# standard deviations, 6 x 2^-53 / sqrt(3 x 16384) = 0.027 x 2^-53.  Sums of cut populations lose 2^-55 n on average.
@pytest.mark.parametrize("precision", [0, 1])
def test_sums_have_no_bias(olb, precision):
    ctx = _context(olb, precision)
    rng = np.random.default_rng(2)
    w = np.array([0.0113, 0.2221, 0.5333, 0.2221, 0.0113])
    f = (np.outer(w, w).reshape(25, 1, 1) * rng.uniform(0.5, 1.5, (25, 128, 128)))
    f[7] *= 1e-3
    f[18] *= 1e-5
    ctx.set_populations(f)
    f = ctx.get_populations().reshape(25, -1)  # (FP32: the pairs, exact in FP64)
    n = ctx.moments()[0].ravel()
    err = np.array([math.fsum([n[q]] + [-v for v in f[:, q]]) / n[q] for q in range(n.size)])
    assert np.max(np.abs(err)) <= 2.0 ** -53 * 2.0
    assert abs(err.mean()) <= 0.027 * 2.0 ** -53
