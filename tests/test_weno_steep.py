"""The integer WENO5 form of one axis (csrc/weno_int.cuh): the side it evaluates, and
its larger units (weno_steep12) for differences out of its range, as those of a
phi far from a distance are.

CPU: the host build.  The side is right if the value is the larger of the two
sides' exactly.  Larger units, against extended precision: the differences are
rounded by half a unit 2^(s-S) <= 2^-56 of the largest: 8 units through the centre
term, 16 + 4 through the linear part of 12 Phi, and through its weights, whose
smoothness terms move by at most 12 sqrt(s_k) units, 270; with the 4 units and
2^-52 of the terms that weno_phi12 allows itself: 512 units, and 2^-52.  And the
largest and the root-mean-square error against the FP64 form's on the same
values, but for a kink at the stencil's far end.
GPU: steps at slopes around and beyond the range, against the oracle at 1e-10 h.
"""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2209_15095_gb300", "csrc")
SRC = """
#include <math.h>
#include "weno_int.cuh"
using namespace etd;
extern "C" void steep(int n, double h, const double* f, int positive, double* out, int* took) {
  const WenoInt k = weno_int(h, 1e-6);
  for (int i = 0; i < n; ++i) {
    i64 F[7], q[6];
    unsigned top = 0;
    for (int j = 0; j < 7; ++j) {
      F[j] = to_fix(f[7 * i + j], k.eh, FIX_KMAX);
      top |= hi_mag(F[j]);
    }
    const unsigned big = fix_diffs(F, q);
    took[i] = top >= FIX_OWN_HI ? 0 : big < FIX_DIFF_HI ? 1 : 2;
    out[i] = took[i] ? weno_steep12(q, big, positive, k) : 0.0;
  }
}
// 1 where weno_axis gives the larger of both sides (differences in range)
extern "C" void side(int n, double h, const double* f, int positive, int* right) {
  const WenoInt k = weno_int(h, 1e-6);
  for (int i = 0; i < n; ++i) {
    i64 F[7], q[6], e[5];
    for (int j = 0; j < 7; ++j) F[j] = to_fix(f[7 * i + j], k.eh, FIX_KMAX);
    right[i] = fix_diffs(F, q) < FIX_DIFF_HI ? 0 : 2;
    if (right[i]) continue;
    for (int j = 0; j < 5; ++j) e[j] = q[j + 1] - q[j];
    const i64 cen = 7 * (q[2] + q[3]) - (q[1] + q[4]);
    const i64 dm = cen - weno_phi12(e[0], e[1], e[2], e[3], k), dp = cen + weno_phi12(e[4], e[3], e[2], e[1], k);
    const i64 a = positive ? dm : -dm, b = positive ? -dp : dp;
    const i64 m = a > b ? a : b;
    right[i] = weno_axis(q, positive, k) == (m > 0 ? m : 0);
  }
}
"""


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("wsteep")
    (d / "w.cpp").write_text(SRC)
    subprocess.run([cxx, "-O2", "-shared", "-fPIC", "-I" + CSRC, str(d / "w.cpp"), "-o", str(d / "w.so")], check=True)
    return ctypes.CDLL(str(d / "w.so"))


def _p(a):
    return a.ctypes.data_as(ctypes.c_void_p)


def _godunov(f, h, positive, T):
    """12 h max(d-, -d+, 0) or its mirror image, and the size of its terms."""
    q = np.diff(f.astype(T), axis=1)
    e = np.diff(q, axis=1)
    eps, k13 = T(4e-6) * T(h) ** 2, T(13) / T(3)

    def phi(a, b, c, d):
        s = [eps + k13 * (a - b) ** 2 + (a - 3 * b) ** 2, eps + k13 * (b - c) ** 2 + (b + c) ** 2,
             eps + k13 * (c - d) ** 2 + (3 * c - d) ** 2]
        A, B, C = (s[1] * s[2]) ** 2, (s[0] * s[2]) ** 2, (s[0] * s[1]) ** 2
        X, Y = a - 2 * b + c, b - 2 * c + d
        return (4 * A * X + (3 * C - A - 6 * B) * Y) / (A + 6 * B + 3 * C), 4 * np.abs(X) + np.abs(Y)

    cen = 7 * (q[:, 2] + q[:, 3]) - (q[:, 1] + q[:, 4])
    pm, tm = phi(e[:, 0], e[:, 1], e[:, 2], e[:, 3])
    pp, tp = phi(e[:, 4], e[:, 3], e[:, 2], e[:, 1])
    a, b = (cen - pm, -cen - pp) if positive else (pm - cen, cen + pp)
    return np.maximum(np.maximum(a, b), 0), tm + tp, np.max(np.abs(q), axis=1)


def _values(rng, h, kind, n):
    x = np.arange(-3, 4) * h
    r = lambda *s: 2.0 * rng.random(s) - 1.0
    if kind == "slope":
        return 15.0 * r(n, 1) * x + 6.0 * h * r(n, 1) + h * rng.random((n, 1)) * np.sin(x / h + 6.0 * r(n, 1))
    if kind == "rough":
        return 30.0 * h * r(n, 7)
    if kind == "jumps":
        return r(n, 1) * x + h * r(n, 1) + (rng.random((n, 7)) < 0.3) * 40.0 * h * r(n, 7)
    if kind == "curved":
        return 3.0 * r(n, 1) * x + 3.0 * rng.random((n, 1)) * x * x / h
    f = (1.0 + 7.0 * rng.random((n, 1))) * x + 0.01 * h * rng.random((n, 7))  # a kink at the stencil's end
    f[:, 6] += 40.0 * h * r(n)
    return f


@pytest.mark.parametrize("positive", [0, 1])
@pytest.mark.parametrize("kind", ["slope", "rough", "jumps", "curved", "far kink"])
@pytest.mark.parametrize("h", [1.0, 12.0 / 199.0, 1.9999])
def test_against_extended_precision_and_fp64(host, h, kind, positive):
    n = 20000
    f = np.ascontiguousarray(_values(np.random.default_rng(12), h, kind, n))
    got, took = np.empty(n), np.empty(n, dtype=np.int32)
    host.steep(n, ctypes.c_double(h), _p(f), positive, _p(got), _p(took))
    ref, terms, top = _godunov(f, h, positive, np.longdouble)
    U = np.ldexp(1.0, int(np.floor(np.log2(h))) - 54)
    unit = np.maximum(U, top * 2.0 ** -56)
    err = np.abs(got - ref)
    assert np.all((err <= 512 * unit + 2.0 ** -52 * terms + 2.0 ** -52 * ref)[took > 0])
    f64 = np.abs(_godunov(f, h, positive, np.float64)[0] - ref)
    s = took == 2
    assert np.count_nonzero(s) > n // 10
    if kind != "far kink":
        assert np.max(err[s]) <= np.max(f64[s]) and np.mean(err[s] ** 2) <= np.mean(f64[s] ** 2)


@pytest.mark.parametrize("positive", [0, 1])
@pytest.mark.parametrize("h", [1.0, 12.0 / 199.0, 1.9999])
@pytest.mark.parametrize("kind", ["slope", "rough", "jumps", "curved", "far kink", "ridge"])
def test_side(host, h, kind, positive):
    n = 50000
    rng = np.random.default_rng(13)
    if kind == "ridge":  # d- + d+ near 0 and of every size
        f = -np.abs(np.arange(-3, 4)) * h * rng.random((n, 1)) * np.sign(rng.random((n, 1)) - 0.5)
        f = f + h * 10.0 ** (-7.0 * rng.random((n, 1))) * (2.0 * rng.random((n, 7)) - 1.0)
    else:
        f = _values(rng, h, kind, n) * 10.0 ** (-1.0 - 4.0 * rng.random((n, 1)))
    right = np.empty(n, dtype=np.int32)
    host.side(n, ctypes.c_double(h), _p(np.ascontiguousarray(f)), positive, _p(right))
    assert np.count_nonzero(right == 1) > n // 2 and not np.count_nonzero(right == 0)


@pytest.mark.gpu
@pytest.mark.parametrize("ndim,n", [(2, 40), (3, 34), (3, 97), (4, 18)])
@pytest.mark.parametrize("slope", [4.5, 7.0, 20.0, 80.0])
def test_steep_step(ndim, n, slope):
    """Axes in range, in larger units and (slope 80) with values out of range, on few
    nodes (an axis per lane) and many (3D at 97)."""
    import torch

    from oracle import levelset
    from oracle.eb import EBOperator
    from oracle.grid import Grid
    from paper_2209_15095_gb300 import build

    build.build()
    from paper_2209_15095_gb300 import etd

    box = 2.0
    g = Grid((n,) * ndim, (-box,) * ndim, (box,) * ndim)
    x = g.coords()
    r = np.sqrt(sum(((x[d] - 0.02 * d) / (1.0 + 0.05 * d)) ** 2 for d in range(ndim)))
    phi = slope * (r - 0.55 * box)
    op = EBOperator(g, phi, 1.0)
    u = np.where(op.comp, np.cos(r), 0.0)
    T = levelset.tube(phi, g.h)
    ctx = etd.Context(g.n, g.lo, g.hi, precision="fp64")
    dphi, du = torch.tensor(phi, device="cuda"), torch.tensor(u, device="cuda")
    ctx.init_domain(0, dphi)
    dt = 0.05 * g.h / slope
    ctx.levelset_advance(0, dphi, du, dt, False)
    ctx.sync()
    ref, _, _ = levelset.levelset_advance(phi, u, op.comp, g, dt, 1.0, False)
    assert np.max(np.abs(dphi.cpu().numpy() - ref)[T]) <= 1e-10 * g.h
