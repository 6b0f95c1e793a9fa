"""The FP32 bounds of a point-triangle distance that choose the triangles of the
object grid (csrc/tri_f32.h, compiled here for the host): for triangles of every
shape, needles with the sharp corner at each vertex above all, the exact distance
lies between them.  Exact: closest point in extended precision."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2605_21398_gb300", "csrc")

SHIM = r"""
#include "tri_f32.h"
extern "C" void bounds(int n, const double *v, const double *p, double S, double cut, float *lo, float *hi)
{
    for (int i = 0; i < n; ++i) {
        double q[3][3];
        for (int k = 0; k < 9; ++k) q[k / 3][k % 3] = v[9 * i + k];
        const dock::TriF t = dock::tri_f32(q, (float)S, (float)cut, true);
        const float e = dock::tri_edge_tol((float)S), x = (float)p[3 * i], y = (float)p[3 * i + 1], z = (float)p[3 * i + 2];
        const bool sure = t.tol < INFINITY;
        const float skip = (float)cut * 1.00001f;
        lo[i] = sure ? dock::tri_bound_f32<false>(t, x, y, z, skip, e) : 0.f;
        hi[i] = sure ? dock::tri_bound_f32<true>(t, x, y, z, skip, e) + e : INFINITY;
    }
}
"""


@pytest.fixture(scope="module")
def bounds(tmp_path_factory):
    d = tmp_path_factory.mktemp("tri")
    src, so = str(d / "shim.cpp"), str(d / "shim.so")
    with open(src, "w") as f:
        f.write(SHIM)
    subprocess.run(["g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-ffp-contract=off", "-I", CSRC, "-o", so, src],
                   check=True)
    fn = ctypes.CDLL(so).bounds
    dp, fp = ctypes.POINTER(ctypes.c_double), ctypes.POINTER(ctypes.c_float)
    fn.argtypes = [ctypes.c_int, dp, dp, ctypes.c_double, ctypes.c_double, fp, fp]

    def run(v, p, S, cut):
        n = len(v)
        v, p = np.ascontiguousarray(v, dtype=np.float64), np.ascontiguousarray(p, dtype=np.float64)
        lo, hi = np.empty(n, np.float32), np.empty(n, np.float32)
        fn(n, v.ctypes.data_as(dp), p.ctypes.data_as(dp), S, cut, lo.ctypes.data_as(fp), hi.ctypes.data_as(fp))
        return lo, hi
    return run


def _distance(v, p):
    """Distances in extended precision: the three edges, the plane where the projection falls inside."""
    v, p = v.astype(np.longdouble), p.astype(np.longdouble)

    def dot(x, y):
        return np.sum(x * y, axis=-1)

    best = np.full(len(v), np.inf, dtype=np.longdouble)
    for k in range(3):
        a, b = v[:, k], v[:, (k + 1) % 3]
        e = b - a
        s = np.clip(dot(p - a, e) / np.maximum(dot(e, e), np.longdouble(1e-300)), 0, 1)
        best = np.minimum(best, np.sqrt(dot(p - a - s[:, None] * e, p - a - s[:, None] * e)))
    n = np.cross(v[:, 1] - v[:, 0], v[:, 2] - v[:, 0])
    nn = np.maximum(dot(n, n), np.longdouble(1e-300))
    inside = np.ones(len(v), dtype=bool)
    for k in range(3):
        inside &= dot(np.cross(v[:, (k + 1) % 3] - v[:, k], p - v[:, k]), n) >= 0
    h = np.abs(dot(p - v[:, 0], n)) / np.sqrt(nn)
    return np.where(inside, np.minimum(best, h), best)


@pytest.mark.parametrize("corner", [0, 1, 2])
@pytest.mark.parametrize("edge", [0.05, 0.5, 2.0, 8.0])
@pytest.mark.parametrize("S, cut", [(16.0, 0.5), (19.2, 0.2), (150.0, 1.2)])
def test_exact_distance_lies_between_the_bounds(bounds, S, cut, edge, corner):
    rng = np.random.default_rng([int(S), int(100 * edge), corner])
    n = 60000
    edge = edge * S / 16.0
    # needles: apex, an end at `edge`, another turned by s; s from flat to equilateral
    s = 10.0 ** rng.uniform(-5, 0, size=n)
    d = rng.normal(size=(n, 3))
    d /= np.linalg.norm(d, axis=1, keepdims=True)
    o = np.cross(d, rng.normal(size=(n, 3)))
    o /= np.linalg.norm(o, axis=1, keepdims=True)
    apex = S / 2 + rng.uniform(-0.05, 0.05, size=(n, 3)) * S - 0.5 * edge * d
    far = rng.uniform(0.3, 1.0, size=(n, 1))
    tri = np.stack([apex, apex + edge * d, apex + far * edge * (d * np.cos(s)[:, None] + o * np.sin(s)[:, None])], axis=1)
    v = np.roll(tri, corner, axis=1)
    # points in the plane and off it, near the body, the ends and beyond them
    w = rng.uniform(-0.3, 1.3, size=(n, 2))
    base = tri[:, 0] + w[:, :1] * (tri[:, 1] - tri[:, 0]) + w[:, 1:] * rng.choice([0.0, 1.0], size=(n, 1)) * (tri[:, 2] - tri[:, 1])
    p = base + rng.normal(size=(n, 3)) * cut * 10.0 ** rng.uniform(-4, 0, size=(n, 1))
    inside = np.all((v > 0) & (v < S), axis=(1, 2)) & np.all((p > 0) & (p < S), axis=1)
    v, p = v[inside], p[inside]
    assert len(v) > n // 4
    lo, hi = bounds(v, p, S, cut)
    want = _distance(v, p)
    assert np.all(lo[want < cut] <= want[want < cut])
    assert np.all(hi >= want)
    # and they are of use: most well-shaped triangles are known to a thousandth of the cut
    good = (s[inside] > 0.1) & (want < 0.5 * cut)
    assert np.mean(hi[good] - lo[good] < 2e-3 * cut) > 0.9
