"""The FP32 filters in front of the FP64 decisions (csrc/pm_filter.cuh), compiled for the host:
whatever a filter decides has to hold for the values in extended precision, and near ties have to
be left undecided.  Their bounds leave a relative margin of at least 2^-24 for the FP64 code's own
rounding, so agreement with the exact values (margin 2^-40) covers it.
"""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = r"""
#include <cstdint>
#include "pm_filter.cuh"
using namespace pm;
static VF vf(const double* p) { return make_vf(p[0], p[1], p[2], p[3], p[4]); }
// the metric at points x of the triangles, and the quality bound of (x, b, c) with it
extern "C" void at(const double* p, const double* x, int n, float* m, float* kx, float* up) {
  for (int i = 0; i < n; ++i) {
    const VF a = vf(p + 15 * i), b = vf(p + 15 * i + 5), c = vf(p + 15 * i + 10);
    VF o = make_vf_xy(x[2 * i], x[2 * i + 1]);
    kx[i] = f_metric_at(o, a, b, c, o);
    m[3 * i] = o.m00;
    m[3 * i + 1] = o.m01;
    m[3 * i + 2] = o.m11;
    int sign;
    up[i] = f_quality_up(o, b, c, sign, kx[i]);
  }
}
// both quality bounds of (x, b, c) with the metric at x
extern "C" void bounds(const double* p, const double* x, int n, float* lo, float* up,
                       int32_t* sign) {
  for (int i = 0; i < n; ++i) {
    const VF a = vf(p + 15 * i), b = vf(p + 15 * i + 5), c = vf(p + 15 * i + 10);
    VF o = make_vf_xy(x[2 * i], x[2 * i + 1]);
    const float kx = f_metric_at(o, a, b, c, o);
    const FQual q = f_quality(o, b, c, sign[i], kx);
    lo[i] = q.lo;
    up[i] = q.up;
  }
}
extern "C" void run(const double* p, const double* bound, int n, int32_t* orient, int32_t* len,
                    float* up, int32_t* osign, float* l2, float* el2) {
  for (int i = 0; i < n; ++i) {
    const VF a = vf(p + 15 * i), b = vf(p + 15 * i + 5), c = vf(p + 15 * i + 10);
    orient[i] = f_orient(a, b, c);
    const FLen l = f_edge2(a, b);
    l2[i] = l.L2;
    el2[i] = l.err;
    len[i] = f_len_cmp(l, nextafterf((float)bound[i], -INFINITY),
                       nextafterf((float)bound[i], INFINITY));
    up[i] = f_quality_up(a, b, c, osign[i]);
  }
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("filters")
    src, so = d / "f.cpp", d / "f.so"
    src.write_text(SRC)
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-ffp-contract=off", "-x", "c++",
                    "-I", os.path.join(ROOT, "paper_1505_04694_gb300", "csrc"), str(src), "-o",
                    str(so)], check=True)
    return C.CDLL(str(so))


def triangles(rng, n, scale, offset, aspect, flat):
    """n triangles (x, y, m00, m01, m11 per vertex): points within `scale` of a point at distance
    `offset`, metrics of aspect ratio up to `aspect`; a third of them nearly collinear (`flat` times
    the scale off the line), some exactly."""
    o = rng.uniform(-1, 1, (n, 1, 2)) * offset
    p = o + rng.uniform(-1, 1, (n, 3, 2)) * scale
    k = n // 3
    t = rng.uniform(-2, 2, (k, 1))
    p[:k, 2] = p[:k, 0] + t * (p[:k, 1] - p[:k, 0]) + rng.uniform(-1, 1, (k, 2)) * scale * flat
    p[:k // 4, 2] = 0.5 * (p[:k // 4, 0] + p[:k // 4, 1])  # a midpoint (rounded)
    th = rng.uniform(0, np.pi, (n, 1)) + rng.uniform(-0.1, 0.1, (n, 3))
    asp = np.exp(rng.uniform(0, np.log(aspect), (n, 1))) * np.ones((1, 3))
    a = np.exp(rng.uniform(-1, 1, (n, 3))) / scale / scale
    b = a / asp ** 2
    c, s = np.cos(th), np.sin(th)
    return np.ascontiguousarray(np.concatenate(
        [p, (a * c * c + b * s * s)[..., None], ((a - b) * c * s)[..., None],
         (a * s * s + b * c * c)[..., None]], axis=2))


CASES = [(1.0, 1.0, 10.0, 1e-7), (1e-3, 1.0, 100.0, 1e-6), (1e-4, 1.0, 3.0, 1e-3),
         (1e-3, 1e4, 30.0, 1e-5), (1e-12, 1e-10, 100.0, 1e-8), (1e6, 1e6, 1000.0, 1e-9),
         (1e-22, 1e-22, 10.0, 1e-3), (1e15, 1e15, 10.0, 1e-4), (1e25, 1e25, 10.0, 1e-4),
         (1e-45, 1e-45, 5.0, 1e-2), (1e160, 1e160, 5.0, 1e-2)]


@pytest.mark.parametrize("scale,offset,aspect,flat", CASES)
def test_filters_decide_only_what_is_certain(lib, scale, offset, aspect, flat):
    rng = np.random.default_rng(int(abs(np.log10(scale)) * 7 + aspect))
    n = 60000
    tri = triangles(rng, n, scale, offset, aspect, flat)
    L = np.longdouble
    with np.errstate(all="ignore"):
        a, b, c = (tri[:, k].astype(L) for k in range(3))
        det = ((b[:, 0] - a[:, 0]) * (c[:, 1] - a[:, 1])
               - (b[:, 1] - a[:, 1]) * (c[:, 0] - a[:, 0]))
        mag = (abs((b[:, 0] - a[:, 0]) * (c[:, 1] - a[:, 1]))
               + abs((b[:, 1] - a[:, 1]) * (c[:, 0] - a[:, 0])))

        def length2(m, p, q):
            dx, dy = q[:, 0] - p[:, 0], q[:, 1] - p[:, 1]
            return m[0] * dx * dx + 2 * m[1] * dx * dy + m[2] * dy * dy

        e2 = length2([(a[:, k] + b[:, k]) / 2 for k in (2, 3, 4)], a, b)
        k = [(a[:, j] + b[:, j] + c[:, j]) / 3 for j in (2, 3, 4)]
        P = sum(np.sqrt(length2(k, p, q)) for p, q in ((a, b), (b, c), (c, a)))
        x = P / 3
        s = np.minimum(x, 1 / x)
        q = (12 * np.sqrt(L(3)) * np.sqrt(k[0] * k[2] - k[1] ** 2) * (det / 2) / P ** 2
             * (s * (2 - s)) ** 3)
        # bounds around each edge's own squared length, some of them very near it
        near = 1.0 + rng.choice([1e-9, 1e-7, 1e-6, 1e-4, 0.1], n) * rng.choice([-1, 1], n)
        bound = np.ascontiguousarray((e2 * near).astype(np.float64))
        out = dict(orient=np.zeros(n, np.int32), len=np.zeros(n, np.int32),
                   up=np.zeros(n, np.float32), osign=np.zeros(n, np.int32),
                   l2=np.zeros(n, np.float32), el2=np.zeros(n, np.float32))
        vp = C.c_void_p
        lib.run(vp(tri.ctypes.data), vp(bound.ctypes.data), n,
                *(vp(v.ctypes.data) for v in out.values()))
        tie = mag * L(2.0) ** -40
        for sign in (out["orient"], out["osign"]):
            assert not np.any((sign > 0) & ~(det > tie))
            assert not np.any((sign < 0) & ~(det < -tie))
        assert not np.any((out["len"] > 0) & ~(e2 > bound * (1 + L(2.0) ** -40)))
        assert not np.any((out["len"] < 0) & ~(e2 < bound * (1 - L(2.0) ** -40)))
        known = np.isfinite(out["l2"]) & np.isfinite(out["el2"]) & np.isfinite(e2.astype(float))
        assert not np.any(known & (abs(out["l2"].astype(L) - e2) > out["el2"]))
        # the bound is an upper bound wherever it is one at all
        has = np.isfinite(out["up"]) & np.isfinite(q.astype(float))
        assert not np.any(has & ~(out["up"].astype(L) >= q + abs(q) * L(2.0) ** -40))
    if 1e-13 < scale < 1e10:  # and in the ordinary range the filters decide most cases
        fat = np.arange(n) >= n // 3
        assert np.mean(out["orient"][fat] != 0) > 0.98
        ok = has & (det > 0) & (x < 10) & fat
        if aspect <= 30 and offset <= 1.0:
            assert np.median((out["up"][ok] - q[ok]) / q[ok]) < 0.01


def quality_exact(a, b, c):
    """The quality of (a, b, c) (columns x, y, m00, m01, m11) in extended precision."""
    L = np.longdouble
    k = [(a[:, j] + b[:, j] + c[:, j]) / 3 for j in (2, 3, 4)]
    P = 0
    for p, q in ((a, b), (b, c), (c, a)):
        dx, dy = q[:, 0] - p[:, 0], q[:, 1] - p[:, 1]
        P = P + np.sqrt(k[0] * dx * dx + 2 * k[1] * dx * dy + k[2] * dy * dy)
    det = ((b[:, 0] - a[:, 0]) * (c[:, 1] - a[:, 1]) - (b[:, 1] - a[:, 1]) * (c[:, 0] - a[:, 0]))
    s = np.minimum(P / 3, 3 / P)
    return (12 * np.sqrt(L(3)) * np.sqrt(k[0] * k[2] - k[1] ** 2) * (det / 2) / P ** 2
            * (s * (2 - s)) ** 3)


@pytest.mark.parametrize("scale,offset,aspect,flat", CASES)
def test_interpolated_metric_and_its_quality_bound(lib, scale, offset, aspect, flat):
    """f_metric_at at points inside the triangles, on their edges and just outside: its error
    bound holds, and so does the quality bound that carries it."""
    rng = np.random.default_rng(int(abs(np.log10(scale)) * 11 + aspect))
    n = 40000
    tri = triangles(rng, n, scale, offset, aspect, flat)
    w = rng.dirichlet([1.0, 1.0, 1.0], n)
    w[: n // 4, 0] = rng.uniform(-1e-8, 1e-8, n // 4)  # on an edge line, within rounding
    with np.errstate(all="ignore"):
        x = np.ascontiguousarray(np.einsum("ij,ijk->ik", w, tri[:, :, :2]))
        L = np.longdouble
        a, b, c = (tri[:, k].astype(L) for k in range(3))
        X = x.astype(L)

        def det(p, q, r):
            return ((q[:, 0] - p[:, 0]) * (r[:, 1] - p[:, 1])
                    - (q[:, 1] - p[:, 1]) * (r[:, 0] - p[:, 0]))

        o = det(a, b, c)
        l0, l1, l2 = det(X, b, c) / o, det(a, X, c) / o, det(a, b, X) / o
        m = [l0 * a[:, k] + l1 * b[:, k] + l2 * c[:, k] for k in (2, 3, 4)]
        got, kx, up = np.zeros((n, 3), np.float32), np.zeros(n, np.float32), np.zeros(n, np.float32)
        vp = C.c_void_p
        lib.at(vp(tri.ctypes.data), vp(x.ctypes.data), n, vp(got.ctypes.data), vp(kx.ctypes.data),
               vp(up.ctypes.data))
        known = (kx < 0.05) & np.isfinite(o.astype(float))  # larger bounds are not used
        bound = kx.astype(L)
        root = np.sqrt(abs(m[0] * m[2]))
        for j, ref in ((0, m[0]), (1, root), (2, m[2])):
            assert not np.any(known & (abs(got[:, j].astype(L) - m[j]) > bound * abs(ref) * 1.01))
        q = quality_exact(np.stack([X[:, 0], X[:, 1], *m], axis=1), b, c)
        has = known & np.isfinite(up) & np.isfinite(q.astype(float))
        assert not np.any(has & ~(up.astype(L) >= q))
    if 1e-13 < scale < 1e10 and offset <= 1.0:
        assert np.mean(known[(np.arange(n) >= n // 3) & (o > 0)]) > 0.95


@pytest.mark.parametrize("scale,offset,aspect,flat", CASES)
def test_lower_quality_bound(lib, scale, offset, aspect, flat):
    """f_quality with an interpolated metric: the lower bound is -1 unless the element is certainly
    counter-clockwise, lies below the quality and close to it where the upper one is close."""
    rng = np.random.default_rng(int(abs(np.log10(scale)) * 13 + aspect))
    n = 40000
    tri = triangles(rng, n, scale, offset, aspect, flat)
    w = rng.dirichlet([1.0, 1.0, 1.0], n)
    with np.errstate(all="ignore"):
        x = np.ascontiguousarray(np.einsum("ij,ijk->ik", w, tri[:, :, :2]))
        L = np.longdouble
        a, b, c = (tri[:, k].astype(L) for k in range(3))
        X = x.astype(L)

        def det(p, q, r):
            return ((q[:, 0] - p[:, 0]) * (r[:, 1] - p[:, 1])
                    - (q[:, 1] - p[:, 1]) * (r[:, 0] - p[:, 0]))

        o = det(a, b, c)
        l0, l1, l2 = det(X, b, c) / o, det(a, X, c) / o, det(a, b, X) / o
        m = [l0 * a[:, k] + l1 * b[:, k] + l2 * c[:, k] for k in (2, 3, 4)]
        lo, up, sign = np.zeros(n, np.float32), np.zeros(n, np.float32), np.zeros(n, np.int32)
        vp = C.c_void_p
        lib.bounds(vp(tri.ctypes.data), vp(x.ctypes.data), n, vp(lo.ctypes.data),
                   vp(up.ctypes.data), vp(sign.ctypes.data))
        q = quality_exact(np.stack([X[:, 0], X[:, 1], *m], axis=1), b, c)
        has = lo > -1
        assert not np.any(has & (sign <= 0)) and not np.any(np.isnan(lo))
        assert not np.any(has & ~((lo.astype(L) < q) & (det(X, b, c) > 0)))
        ok = has & (q > 1e-3)
        width = (up[ok] - q[ok]) / q[ok]
        assert np.all((q[ok] - lo[ok]) / q[ok] <= 3 * width + 1e-5)
    if aspect <= 30 and offset <= 1.0 and 1e-13 < scale < 1e10:
        fat = (np.arange(n) >= n // 3) & (q > 1e-3)
        assert np.mean(has[fat]) > 0.95
