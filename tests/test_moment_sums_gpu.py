"""Moments of given populations: the sums over a node in fixed point (csrc/olb_kernels.cuh) round to nearest, so that
they have no bias, and the quotients are those of a division."""
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


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("shift", [-30, 0, 40])
def test_quotients_are_those_of_a_division(olb, precision, shift):
    """One velocity a node: n and e are exact up to one rounding, and u = j / n and e / n two rounded operations."""
    ctx = _context(olb, precision)
    rng = np.random.default_rng(9)
    f = np.zeros((25, 128 * 128))
    v = np.ldexp(rng.uniform(1, 2, f.shape[1]).astype(np.float32).astype(np.float64), shift)
    k = rng.integers(0, 25, v.size)
    f[k, np.arange(v.size)] = v
    ctx.set_populations(f.reshape(25, 128, 128))
    n, ux, uy, T = (m.ravel() for m in ctx.moments())
    R = [math.sqrt(5 + s * math.sqrt(10)) for s in (1, -1)]
    R = np.array([-R[0], -R[1], 0.0, R[1], R[0]])
    assert np.array_equal(n, v)
    # (the library's roots may be an ulp off these)
    for u, at in ((ux, k // 5), (uy, k % 5)):
        for q in range(5):
            roots = (np.nextafter(R[q], -9), R[q], np.nextafter(R[q], 9)) if R[q] else (0.0,)
            assert any(np.array_equal(u[at == q], (r * v[at == q]) / v[at == q]) for r in roots), q


@pytest.mark.parametrize("precision", [0, 1])
def test_empty_nodes(olb, precision):
    """n = 0: j / 0, as a division gives it."""
    ctx = _context(olb, precision, 8, 8)
    f = np.zeros((25, 8, 8))
    f[:, 0, 0] = np.where(np.arange(25) // 5 == 4, 1.0, 0.0) - np.where(np.arange(25) // 5 == 0, 1.0, 0.0)
    f[12, 1, 1] = 1.0
    ctx.set_populations(f)
    n, ux, uy, T = ctx.moments()
    assert n[0, 0] == 0 and ux[0, 0] == np.inf and np.isnan(uy[0, 0])
    assert np.isnan(ux[2, 2]) and ux[1, 1] == 0 and T[1, 1] == 0
