"""Builds tests/fixed_host.cu for the CPU and calls it."""
import ctypes as C
import functools
import os
import subprocess
import tempfile
from decimal import Decimal as D
from decimal import getcontext

import numpy as np

getcontext().prec = 60
HERE = os.path.dirname(os.path.abspath(__file__))


@functools.lru_cache(None)
def lib():
    from paper_2012_08221_gb300 import build
    out = os.path.join(tempfile.mkdtemp(prefix="fixed_host"), "libfixed_host.so")
    r = subprocess.run([build.nvcc(), "-shared", "-o", out, os.path.join(HERE, "fixed_host.cu"), "-O2", "-std=c++17",
                        "-Xcompiler", "-fPIC,-ffp-contract=off", "-I", build.INCLUDE, "-I", build.CSRC] + build.ARCH,
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return C.CDLL(out)


def _p(a):
    return a.ctypes.data_as(C.c_void_p)


def cells(lower, last, keys):
    """Cells of the keys (IEEE bits), and the size of the guide table used."""
    lower = np.ascontiguousarray(lower, dtype=np.float64).view(np.uint64)
    keys = np.ascontiguousarray(keys, dtype=np.uint64)
    out, guided = np.empty(keys.size, np.int32), C.c_int()
    lib().host_cells(_p(lower), lower.size, C.c_uint64(int(np.float64(last).view(np.uint64))), _p(keys), keys.size,
                     _p(out), C.byref(guided))
    return out, guided.value


def evaluate(x, q2, v, px, pq, x_linear=False, q_linear=False):
    """Columns: fixed-point value (NaN where FP64 serves), FP64 form at the same
    coordinates, the two fixed-point derivatives, FP64 form at coordinates from
    FP64 logarithms; and the coordinates as integers (value 2^62)."""
    a = [np.ascontiguousarray(z, np.float64) for z in (x, q2, v, px, pq)]
    n = a[3].size
    out, t = np.empty((n, 5)), np.empty((n, 2), np.int64)
    lib().host_eval(a[0].size, _p(a[0]), int(x_linear), a[1].size, _p(a[1]), int(q_linear), _p(a[2]), n, _p(a[3]),
                    _p(a[4]), _p(out), _p(t))
    return out, t


def _weights(z, k, t, linear):
    """Stencil weights of cell k at t and their derivatives, by knot (the
    definition: Hermite cubic with finite-difference slopes)."""
    w, d = {}, {}

    def add(i, a, b):
        w[i], d[i] = w.get(i, 0) + a, d.get(i, 0) + b
    if linear:
        return {k: 1 - t, k + 1: t}, {k: D(-1), k + 1: D(1)}
    dz = z[k + 1] - z[k]
    add(k, 1 - 3 * t * t + 2 * t ** 3, 6 * t * t - 6 * t)
    add(k + 1, 3 * t * t - 2 * t ** 3, 6 * t - 6 * t * t)
    for knot, h, dh in ((k, t - 2 * t * t + t ** 3, 1 - 4 * t + 3 * t * t), (k + 1, t ** 3 - t * t, 3 * t * t - 2 * t)):
        sides = [s for s in (knot - 1, knot) if s >= 0 and s + 1 < len(z)]
        for s in sides:                                       # mean of the adjacent secants
            f = dz / (z[s + 1] - z[s]) / len(sides)
            add(s, -f * h, -f * dh)
            add(s + 1, f * h, f * dh)
    return w, d


def exact(x, q2, v, px, pq, t=None, x_linear=False, q_linear=False):
    """Per point (value, sum of |weight value|, d/dt_x, d/dt_q) in 60 digits, at
    the coordinates t (value 2^62) or, without them, at the points' own."""
    ux, uq = [D(float(a)).ln() for a in x], [D(float(a)).ln() for a in q2]
    res = []
    for i in range(len(px)):
        ks, ts = [], []
        for z, u, p, j in ((x, ux, px[i], 0), (q2, uq, pq[i], 1)):
            k = int(np.clip(np.searchsorted(z[:-1], p, side="right") - 1, 0, len(z) - 2))
            ks.append(k)
            ts.append(D(int(t[i, j])) / (1 << 62) if t is not None else (D(float(p)).ln() - u[k]) / (u[k + 1] - u[k]))
        (wx, dx), (wq, dq) = _weights(ux, ks[0], ts[0], x_linear), _weights(uq, ks[1], ts[1], q_linear)
        r = [D(0)] * 4
        for a in wq:
            for b in wx:
                y = D(float(v[a][b]))
                term = wq[a] * wx[b] * y
                r = [r[0] + term, r[1] + abs(term), r[2] + wq[a] * dx[b] * y, r[3] + dq[a] * wx[b] * y]
        res.append(r)
    return res


def error(got, want):
    """|got - want| of a double against a decimal, as a double."""
    return np.array([abs(float(D(float(g)) - w)) if np.isfinite(g) else np.nan for g, w in zip(got, want)])


def alphas(q2, a, pq):
    """alpha_s in fixed point on one subgrid (NaN where FP64 serves), and the
    coordinates."""
    z = [np.ascontiguousarray(b, np.float64) for b in (q2, a, pq)]
    out, t = np.empty(z[2].size), np.empty(z[2].size, np.int64)
    lib().host_alphas(z[0].size, _p(z[0]), _p(z[1]), z[2].size, _p(z[2]), _p(out), _p(t))
    return out, t
