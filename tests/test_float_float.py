"""The float-float WENO-5 of csrc/olb_ff.cuh, compiled for the host, against the paper's equations in long double:
single faces, flux differences across a node, and values that leave FP32's range at a given scale."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from helpers import ROOT
from paper_1702_01690_gb300 import build

LD = np.longdouble
SOURCE = r"""
#include <algorithm>
#include <cmath>
using std::max;
using std::min;
#include "olb_ff.cuh"
using namespace olb;
using F = ffv<vf1>;
static FfScale scale(double top) { return ff_scale(f64_hi(top) & 0x7fffffff); }
// the face between v[2] and v[3], upwind of v[2]
extern "C" void faces(const double *v, const double *top, int n, double *out)
{
    for (int i = 0; i < n; ++i, v += 5)
        out[i] = weno5_face(v[2], v[1] - v[0], v[2] - v[1], v[3] - v[2], v[4] - v[3], scale(top[i]));
}
// six times the flux difference across v[3]: the faces of v[1] .. v[5] and of v[0] .. v[4]
extern "C" void fluxes(const double *v, const double *top, int n, double *out)
{
    for (int i = 0; i < n; ++i, v += 6) {
        const FfScale s = scale(top[i]);
        F d[5], q[5], x[4], t[3];
        for (int k = 0; k < 5; ++k) {
            const double b[1] = {v[k + 1] - v[k]};
            d[k] = ff_split<vf1>(b, s);
            q[k] = ff_sqr(d[k]);
        }
        for (int k = 0; k < 4; ++k) x[k] = ff_mul(d[k], d[k + 1]);
        for (int k = 0; k < 3; ++k) t[k] = ff_diff2(d[k], d[k + 1], d[k + 2]);
        const F z0 = weno5_ff(q[0], q[1], q[2], q[3], x[0], x[1], x[2], t[0], t[1]);
        const F z1 = weno5_ff(q[1], q[2], q[3], q[4], x[1], x[2], x[3], t[1], t[2]);
        out[i] = ff_widen(ff_lane(weno5_flux6(d[1], d[2], d[3], z0, z1), 0), s);
    }
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("ff")
    src, so = d / "ff.cpp", d / "ff.so"
    src.write_text(SOURCE)
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(build.nvcc()))), "include")
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-fPIC", "-shared", "-isystem", cuda,
                    "-I", os.path.join(ROOT, "paper_1702_01690_gb300", "csrc"), str(src), "-o", str(so)], check=True)
    return ctypes.CDLL(str(so))


def _call(fn, v, top):
    v, top = np.ascontiguousarray(v), np.ascontiguousarray(top)
    out = np.empty(len(v))
    fn(v.ctypes.data_as(ctypes.c_void_p), top.ctypes.data_as(ctypes.c_void_p), len(v),
       out.ctypes.data_as(ctypes.c_void_p))
    return out


def _face_minus_upwind(v):
    """Eqs. weno5_flux, weno5_omega, weno5_delta, weno5_sigma and Table tab:weno from the stencils' differences."""
    d = (v[:, 1:] - v[:, :-1]).astype(LD)  # (rounded to FP64, as the kernel takes them)
    d0, d1, d2, d3 = d.T
    s = [13 * (d1 - d0) ** 2 + 3 * (3 * d1 - d0) ** 2, 13 * (d2 - d1) ** 2 + 3 * (d1 + d2) ** 2,
         13 * (d3 - d2) ** 2 + 3 * (3 * d2 - d3) ** 2]
    low = np.minimum(s[0], np.minimum(s[1], s[2]))
    w = [np.where(low == 0, g * (q == 0), g * (low / np.where(q == 0, 1, q)) ** 2) for g, q in zip((1, 6, 3), s)]
    F = [5 * d1 - 2 * d0, d1 + 2 * d2, 4 * d2 - d3]
    return (w[0] * F[0] + w[1] * F[1] + w[2] * F[2]) / (6 * (w[0] + w[1] + w[2])), np.max(np.abs(d), axis=1)


def _stencils(kind, width, count=40000):
    rng = np.random.default_rng(8)
    i = np.arange(width)
    if kind == "noise":
        return rng.uniform(-1, 1, (count, width))
    if kind == "smooth":
        k = 2 * np.pi / rng.uniform(8, 3000, (count, 1))
        return 1.0 + 0.1 * np.sin(k * i + rng.uniform(0, 6.3, (count, 1)))
    jump = 1.0 * (i >= rng.integers(1, width, (count, 1)))
    return 0.3 + jump + (1e-9 * rng.uniform(-1, 1, (count, width)) if kind == "jump in noise" else 0.0)


# The indicators are forms of condition number below 19 and the quotient has two of their squares, each in arithmetic
# with 2^-47 a step: some 60 x 2^-47, below 2^-40 of the largest difference (flux6: six times two of them)
@pytest.mark.parametrize("kind", ["noise", "smooth", "jump", "jump in noise"])
def test_faces_and_flux_differences_match_the_paper(lib, kind):
    v = _stencils(kind, 5)
    ref, size = _face_minus_upwind(v)
    got = _call(lib.faces, v, np.max(np.abs(v), axis=1))
    # (the face is rounded at the size of v[2])
    assert np.all(np.abs(got - (v[:, 2] + ref)) <= 2.0 ** -40 * size + 2.0 ** -52 * np.abs(v).max(1))
    v = _stencils(kind, 6)
    (behind, s0), (ahead, s1) = _face_minus_upwind(v[:, :5]), _face_minus_upwind(v[:, 1:])
    ref = 6 * ((v[:, 3] - v[:, 2]).astype(LD) + ahead - behind)
    got = _call(lib.fluxes, v, np.max(np.abs(v), axis=1))
    assert np.all(np.abs(got - ref) <= 12 * 2.0 ** -40 * np.maximum(s0, s1))


@pytest.mark.parametrize("low", [1e-6, 1e-7, 1e-9, 1e-12, 1e-20])
def test_what_the_scale_cannot_hold_is_not_finite(lib, low):
    """A scale far below the values: their squares overflow FP32.  A face is then right or no number, never a finite
    one that is wrong."""
    for at in range(1, 6):
        v = np.where(np.arange(6) < at, 1.0, low * (1 + 0.01 * np.arange(6)))[None]
        for fn, w, ref in ((lib.faces, v[:, :5], v[0, 2] + _face_minus_upwind(v[:, :5])[0][0]),
                           (lib.fluxes, v, 6 * (v[0, 3] - v[0, 2] + _face_minus_upwind(v[:, 1:])[0][0]
                                                - _face_minus_upwind(v[:, :5])[0][0]))):
            got = _call(fn, w, np.array([low]))[0]
            assert not np.isfinite(got) or abs(got - ref) <= 1e-9, (at, got, ref)


def test_parity_form_of_the_momentum_derivative_is_the_matrix():
    """dp_line (csrc/olb_stage64.cuh) takes (d_p f)_{2 +- m} = (E_m2 a_2 + E_m1 a_1) +- (O_m2 s_2 + O_m1 s_1 + O_m0 f_2)
    with a_q = f_{2+q} - f_{2-q}, s_q = f_{2+q} + f_{2-q} and E, O from D as fill_tab forms them: D f of Eq. derf,
    exactly, since D is odd under p -> -p."""
    sp = pytest.importorskip("sympy")
    x = sp.Symbol("x")
    He = [sp.Integer(1), x, x ** 2 - 1, x ** 3 - 3 * x, x ** 4 - 6 * x ** 2 + 3]
    R = [-sp.sqrt(5 + sp.sqrt(10)), -sp.sqrt(5 - sp.sqrt(10)), sp.Integer(0)]
    R += [-R[1], -R[0]]
    W = [(7 - 2 * sp.sqrt(10)) / 60, (7 + 2 * sp.sqrt(10)) / 60, sp.Rational(8, 15)]
    W += [W[1], W[0]]
    D = [[-W[k] * sum(He[q + 1].subs(x, R[k]) * He[q].subs(x, R[j]) / sp.factorial(q) for q in range(4))
          for j in range(5)] for k in range(5)]
    f = sp.symbols("f0:5")
    a, s = [None] + [f[2 + q] - f[2 - q] for q in (1, 2)], [f[2]] + [f[2 + q] + f[2 - q] for q in (1, 2)]
    for m in range(3):
        d = D[2 + m]
        E = [None] + [(d[2 + q] - d[2 - q]) / 2 for q in (1, 2)]
        Od = [d[2]] + [(d[2 + q] + d[2 - q]) / 2 for q in (1, 2)]
        even, odd = E[2] * a[2] + E[1] * a[1], Od[2] * s[2] + Od[1] * s[1] + Od[0] * s[0]
        for sign in (1, -1):
            row = sum(D[2 + sign * m][j] * f[j] for j in range(5))
            form = even + (sign * odd if m else 0)  # (the middle row has no part O)
            for j in range(5):
                assert abs(sp.N(sp.diff(row - form, f[j]), 50)) < sp.Float("1e-45")
