"""The FP32 filters' bounds over every unit of length that a record holds (metric entries from 1e-30
to 1e30).
"""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

import test_filters as F

CSRC = os.path.join(F.ROOT, "paper_1505_04694_gb300", "csrc")


def build(d, header=None):
    """The filters compiled for the host; `header` replaces pm_filter.cuh."""
    if header is not None:
        (d / "pm_filter.cuh").write_text(header)
    (d / "f.cpp").write_text(F.SRC)
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-ffp-contract=off", "-x", "c++",
                    "-I", CSRC if header is None else str(d), str(d / "f.cpp"), "-o",
                    str(d / "f.so")], check=True)
    return C.CDLL(str(d / "f.so"))


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    return build(tmp_path_factory.mktemp("units"))


def quality_bounds(lib, tri, x):
    n = len(tri)
    lo, up, sign = np.zeros(n, np.float32), np.zeros(n, np.float32), np.zeros(n, np.int32)
    vp = C.c_void_p
    lib.bounds(vp(tri.ctypes.data), vp(x.ctypes.data), n, vp(lo.ctypes.data), vp(up.ctypes.data),
               vp(sign.ctypes.data))
    return lo, up, sign


def near_equilateral(rng, n, aspect):
    """Triangles of about unit metric edges under one metric of aspect ratio up to `aspect` (long edges
    of unit length), and the place inside each to which its first vertex moves."""
    th = rng.uniform(0, np.pi, n)
    asp = np.exp(rng.uniform(0, np.log(aspect), n))
    c, s = np.cos(th), np.sin(th)
    a, b = np.ones(n), asp ** 2  # eigenvalues along and across (c, s)
    m = np.stack([a * c * c + b * s * s, (a - b) * c * s, a * s * s + b * c * c], axis=1)
    ref = np.array([[0, 0], [1, 0], [0.5, np.sqrt(0.75)]]) + rng.uniform(-0.15, 0.15, (n, 3, 2))
    p = np.stack([c[:, None] * ref[..., 0] - (s / asp)[:, None] * ref[..., 1],
                  s[:, None] * ref[..., 0] + (c / asp)[:, None] * ref[..., 1]], axis=2)
    # the metric of each vertex within a factor of about two of the triangle's
    tri = np.concatenate([p, m[:, None, :] * np.exp(rng.uniform(-0.5, 0.5, (n, 3, 1)))], axis=2)
    w = rng.dirichlet([6.0, 1.0, 1.0], n)
    return tri, np.einsum("ij,ijk->ik", w, tri[:, :, :2])


# Long edges from 6e-14 to 7e13 units (metric entries up to 1e30 at the smallest); powers of two, so that only the filters can tell the units apart.
@pytest.mark.parametrize("aspect", [1.5, 30.0, 100.0])
@pytest.mark.parametrize("e", [-44, -40, -34, -30, -20, 0, 20, 25, 30, 40, 46])
def test_quality_bounds_do_not_depend_on_the_unit(lib, e, aspect):
    tri, x = near_equilateral(np.random.default_rng(7), 20000, aspect)
    out = []
    for k in (0, e):
        t = tri.copy()
        t[..., :2] = np.ldexp(t[..., :2], k)
        t[..., 2:] = np.ldexp(t[..., 2:], -2 * k)
        t, xs = np.ascontiguousarray(t), np.ascontiguousarray(np.ldexp(x, k))
        L = np.longdouble
        a, b, c = (t[:, j].astype(L) for j in range(3))
        X = xs.astype(L)

        def det(p, q, r):
            return ((q[:, 0] - p[:, 0]) * (r[:, 1] - p[:, 1])
                    - (q[:, 1] - p[:, 1]) * (r[:, 0] - p[:, 0]))

        o = det(a, b, c)
        w = [det(X, b, c) / o, det(a, X, c) / o, det(a, b, X) / o]
        m = [w[0] * a[:, j] + w[1] * b[:, j] + w[2] * c[:, j] for j in (2, 3, 4)]
        q = F.quality_exact(np.stack([X[:, 0], X[:, 1], *m], axis=1), b, c)
        lo, up, sign = quality_bounds(lib, t, xs)
        has = np.isfinite(up)
        if aspect <= 30:  # (beyond, the bound of the lengths leaves some open at any unit)
            assert np.mean(has) > 0.99 and np.mean(lo > -1) > 0.99 and np.mean(sign > 0) > 0.99
        assert not np.any(has & ~(up.astype(L) >= q)) and not np.any((lo > -1) & ~(lo < q))
        ok = has & (lo > -1)
        # 30 u k11 against the Schur complement, at least k11 / aspect^2, and kx: under 1% in the mean
        assert np.median((up[ok] - q[ok]) / q[ok]) < 0.01
        assert np.median((q[ok] - lo[ok]) / q[ok]) < 0.01
        out.append((has, lo > -1, sign))
        held = np.all((t[:, :, (2, 4)] > 1e-30) & (t[:, :, (2, 4)] < 1e30), axis=(1, 2))
    for one, other in zip(*out):  # what is decided is the same but for the absolute terms (1e-36)
        assert np.mean((one != other)[held]) < 1e-3
