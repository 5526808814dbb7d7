"""Timed cases of the library: what its users have it do, at the sizes they do it.

``listed()`` names the standard cases, ``draw(rng)`` gives another one of the
same ranges; ``prepare`` makes what a caller holds before the call (grids
loaded on the GPU, query arrays, the tuned batch), ``run`` is one pass through
the public entry points, ``work`` counts what the pass cannot do without, and
``exact`` evaluates the same definition in plain float64 torch.

Every input comes from the case and the seed.  Query arrays are log-uniform
over the grid's range, as Monte Carlo phase space and the paper's benchmark
make them; ``outside`` is the share of points beyond the knots (low-x and
low-scale tails that real phase space reaches).
"""
import math

import numpy as np
import torch

from paper_2012_08221_gb300 import autograd, synth
from paper_2012_08221_gb300.batch import Batch
from paper_2012_08221_gb300.lumi import DeviceEvents, luminosity
from paper_2012_08221_gb300.pdf import PDF
from paper_2012_08221_gb300.vegas import Vegas

DEV = "cuda:0"
F64 = torch.float64


def listed():
    return [
        # The paper's usage: all flavours at a short list of points.  The call's latency counts.
        {"name": "xf_1e3", "form": "xf", "grid": "nnpdf", "n": 1000, "flavours": 13, "extrap": "linear",
         "outside": 0.0},
        # The small-grid workload: x*f and alpha_s at 1e5 points, half a wave of threads.
        {"name": "xf_alphas_1e5", "form": "xf_alphas", "grid": "small", "n": 100_000, "flavours": 11,
         "extrap": "linear", "outside": 0.0},
        # The headline: 13 flavours at 1e7 points of an NNPDF-shaped grid.
        {"name": "xf_1e7", "form": "xf", "grid": "nnpdf", "n": 10_000_000, "flavours": 13, "extrap": "linear",
         "outside": 0.0},
        # Three flavours in Q with LHAPDF-style continuation and a tail outside the knots; ragged.
        {"name": "xfq_tail_1e6", "form": "xfq", "grid": "set_b", "n": 1_000_003, "flavours": 3,
         "extrap": "continuation", "outside": 0.05},
        # The headline's second half: alpha_s at 1e7 scales.
        {"name": "alphas_1e7", "form": "alphas", "grid": "nnpdf", "n": 10_000_000, "outside": 0.0},
        # A fit on data points with one flavour each: value and gradients in x, Q^2 and the knots.
        {"name": "fit_pw_1e7", "form": "fit_pw", "grid": "small", "n": 10_000_000, "flavours": 13,
         "outside": 0.0},
        # A fit that needs every flavour at each point.
        {"name": "fit_1e6", "form": "fit", "grid": "small", "n": 1_000_000, "flavours": 13, "outside": 0.0},
        # PDF uncertainties: many uneven requests over replicas of three sets in one prepared launch.
        {"name": "batch_400", "form": "batch", "requests": 400, "smallest": 1000, "largest": 1_000_000},
        # Collider events: luminosity and alpha_s per event, 5 % of them in the low tail.
        {"name": "lumi_2e7", "form": "lumi", "grid": "nnpdf", "n": 20_000_000, "outside": 0.05},
        # The same as a fit's objective: the luminosity and its gradient in the knots.
        {"name": "lumi_fit_2e6", "form": "lumi_fit", "grid": "nnpdf", "n": 2_000_001, "outside": 0.05},
        # Monte Carlo integration around a user's integrand (the paper's single-top use).
        {"name": "vegas_1e6", "form": "vegas", "grid": "nnpdf", "n": 1_000_000, "iterations": 3, "bins": 50},
        # Arrays in host memory, in and out, through the library's own pipeline.
        {"name": "host_1e6", "form": "host", "grid": "nnpdf", "n": 1_000_000, "flavours": 13,
         "extrap": "linear", "outside": 0.0},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    form = rng.choice(["xf", "xf", "xfq", "xf_alphas", "alphas", "fit_pw", "fit", "batch", "lumi", "lumi_fit",
                       "vegas", "host"])
    grid = rng.choice(["small", "set_b", "nnpdf"])
    outside = rng.choice([0.0, 0.01, 0.05])
    if form in ("xf", "xfq", "xf_alphas", "host"):
        hi = {"xf": 9_000_000, "xfq": 9_000_000, "xf_alphas": 9_000_000, "host": 2_000_000}[form]
        return {"form": form, "grid": grid, "n": _log_int(rng, 1000, hi), "flavours": rng.randint(1, 11),
                "extrap": rng.choice(["linear", "linear", "freeze", "continuation"]), "outside": outside}
    if form == "alphas":
        return {"form": form, "grid": grid, "n": _log_int(rng, 1000, 9_000_000), "outside": outside}
    if form == "fit_pw":
        return {"form": form, "grid": grid, "n": _log_int(rng, 10_000, 9_000_000), "flavours": rng.randint(1, 11),
                "outside": outside}
    if form == "fit":
        return {"form": form, "grid": grid, "n": _log_int(rng, 1000, 900_000), "flavours": rng.randint(1, 11),
                "outside": outside}
    if form == "batch":
        return {"form": form, "requests": _log_int(rng, 10, 390), "smallest": 1000,
                "largest": _log_int(rng, 20_000, 900_000)}
    if form == "lumi":
        return {"form": form, "grid": grid, "n": _log_int(rng, 10_000, 18_000_000), "outside": outside}
    if form == "lumi_fit":
        return {"form": form, "grid": grid, "n": _log_int(rng, 10_000, 1_900_000), "outside": outside}
    return {"form": form, "grid": grid, "n": _log_int(rng, 10_000, 990_000), "iterations": 3,
            "bins": rng.randint(20, 100)}


# --------------------------------------------------------------------- inputs

def _grid(case, seed):
    """The set of the case; its knot values depend on the seed (a fit's start)."""
    name = case["grid"]
    if name == "small":
        return synth.grid_small(seed=seed, pids=synth.PIDS_13 if case.get("flavours", 0) > 11 else synth.PIDS_11)
    if name == "set_b":
        return synth.grid_set_b()
    return synth.grid_nnpdf(seeds=(seed,))


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _uniform(gen, n, lo, hi):
    return torch.rand(n, generator=gen, dtype=F64, device=DEV) * (hi - lo) + lo


def _scales(g, gen, n, outside):
    """Q^2 log-uniform over the grid, a share of them below or above it."""
    lo, hi = 2 * math.log(g.q_knots[0]), 2 * math.log(g.q_knots[-1])
    w = _uniform(gen, n, lo, hi)
    if outside:
        u = torch.rand(n, generator=gen, dtype=F64, device=DEV)
        w = torch.where(u < outside / 4, lo - 3.0 * u * 4 / outside, w)
        w = torch.where(u > 1 - outside / 4, hi + 2.0 * (1 - u) * 4 / outside, w)
    return torch.exp(w)


def _points(g, gen, n, outside):
    """x log-uniform over the grid's range up to 1, a share of them below it, and the scales."""
    lo = math.log(g.x_knots[0])
    u = _uniform(gen, n, lo, 0.0)
    if outside:
        v = torch.rand(n, generator=gen, dtype=F64, device=DEV)
        u = torch.where(v < outside / 2, lo - 4.0 * v * 2 / outside, u)
    return torch.exp(u).clamp_(max=1.0 - 2.0 ** -53), _scales(g, gen, n, outside)


def _events(g, gen, n, outside):
    """Events in log variables at sqrt(s) = 13 TeV; the tail takes a low scale, half of it a low x1."""
    lt = _uniform(gen, n, math.log(1e-6), 0.0)
    y = _uniform(gen, n, -1.0, 1.0) * (-0.5 * lt)
    r = torch.rand(n, generator=gen, dtype=F64, device=DEV)
    flags = (r < outside).to(torch.uint8) + 2 * (r < 0.5 * outside).to(torch.uint8)
    mu = _uniform(gen, n, math.log(0.04), 0.0)
    lx = _uniform(gen, n, math.log(1e-11), math.log(1e-9))
    return DeviceEvents(lt, y, flags, mu, lx, 2 * math.log(synth.SQRT_S))


def _pids(g, k, seed):
    """k of the grid's pids in ascending order, all of them where k is the set's size."""
    k = min(int(k), g.n_flav)
    return np.sort(np.random.default_rng(seed).choice(g.pids, size=k, replace=False)).astype(np.int32)


def _batch_sets():
    return [synth.grid_set_a(), synth.grid_set_b(), synth.grid_set_c()]


def _batch_requests(case, seed, sets):
    """(set, member, pids, x, Q^2) per request; sizes log-uniform, the same for every seed."""
    rng, gen = np.random.default_rng(case["requests"]), _gen(seed)
    for _ in range(case["requests"]):
        s = int(rng.integers(0, len(sets)))
        g = sets[s]
        m = int(rng.integers(0, g.n_members))
        pids = np.sort(rng.choice(g.pids, size=int(rng.integers(1, 4)), replace=False)).astype(np.int32)
        n = int(round(math.exp(rng.uniform(math.log(case["smallest"]), math.log(case["largest"])))))
        x, q2 = _points(g, gen, n, 0.0)
        yield s, m, pids, x, q2


def _uniforms(case, seed):
    gen = _gen(seed)
    return [torch.rand((case["n"], 3), generator=gen, dtype=F64, device=DEV) for _ in range(case["iterations"])]


def _row(n):
    """Doubles that an output of n doubles takes in the batch's buffer (64-byte rows)."""
    return (n + 7) // 8 * 8


def prepare(case, seed):
    form = case["form"]
    if form == "batch":
        sets = _batch_sets()
        pdfs = [PDF.from_grid(g, device=DEV) for g in sets]
        asked = list(_batch_requests(case, seed, sets))
        out = torch.zeros(sum(_row(r[3].numel() * r[2].size) for r in asked), dtype=F64, device=DEV)
        reqs, at = [], 0
        for s, m, pids, x, q2 in asked:
            k = x.numel() * pids.size
            reqs.append((pdfs[s], m, pids, x, q2, out[at:at + k].view(x.numel(), pids.size)))
            at += _row(k)
        return {"form": form, "batch": Batch(reqs), "out": out}
    g = _grid(case, seed)
    pdf = PDF.from_grid(g, device=DEV, extrap=case.get("extrap", "linear"))
    gen = _gen(seed)
    st = {"form": form, "pdf": pdf}
    if form in ("xf", "xfq", "xf_alphas", "host"):
        st["pids"] = _pids(g, case["flavours"], seed)
        x, q2 = _points(g, gen, case["n"], case["outside"])
        st["x"], st["q"] = x, torch.sqrt(q2) if form == "xfq" else q2
        if form == "host":
            st["x"], st["q"] = x.cpu().pin_memory(), q2.cpu().pin_memory()
            st["out"] = torch.empty((case["n"], st["pids"].size), dtype=F64, pin_memory=True)
    elif form == "alphas":
        st["q"] = _scales(g, gen, case["n"], case["outside"])
    elif form in ("fit", "fit_pw"):
        pids = _pids(g, case["flavours"], seed)
        x, q2 = _points(g, gen, case["n"], case["outside"])
        st["x"], st["q"] = x.requires_grad_(True), q2.requires_grad_(True)
        st["values"] = torch.as_tensor(g.values, device=DEV).requires_grad_(True)
        if form == "fit":
            st["pids"] = pids
            st["w"] = torch.randn((case["n"], pids.size), generator=gen, dtype=F64, device=DEV)
        else:
            at = torch.randint(pids.size, (case["n"],), generator=gen, device=DEV)
            st["pids"] = torch.as_tensor(pids, device=DEV)[at].contiguous()
            st["w"] = torch.randn(case["n"], generator=gen, dtype=F64, device=DEV)
    elif form in ("lumi", "lumi_fit"):
        st["events"] = _events(g, gen, case["n"], case["outside"])
        if form == "lumi_fit":
            st["values"] = torch.as_tensor(g.values, device=DEV).requires_grad_(True)
    else:
        st["bins"], st["iterations"], st["n"] = case["bins"], case["iterations"], case["n"]
        st["uniforms"] = _uniforms(case, seed)
    return st


# ------------------------------------------------------------------- the pass

TOP, W_MASS, S_HAD = 173.0, 80.4, synth.SQRT_S ** 2
QUARKS = np.array([2, 4, -1, -3], dtype=np.int32)
BOTTOM = np.array([5], dtype=np.int32)


def _single_top(r, xf):
    """A single-top-like LO integrand over (tau, y, cos theta), as user code; ``xf(pids, x, Q^2)``."""
    ln_tau_min = math.log(TOP * TOP / S_HAD)
    ln_tau = (1.0 - r[:, 0]) * ln_tau_min
    tau = torch.exp(ln_tau)
    y = (2.0 * r[:, 1] - 1.0) * (-0.5 * ln_tau)
    x1, x2 = torch.exp(0.5 * ln_tau + y).clamp_(max=1.0), torch.exp(0.5 * ln_tau - y).clamp_(max=1.0)
    shat = tau * S_HAD
    that = -(shat - TOP * TOP) * (1.0 - r[:, 2])
    me2 = shat * (shat - TOP * TOP) / (that - W_MASS * W_MASS) ** 2
    q2 = torch.full_like(x1, TOP * TOP)
    lum = xf(BOTTOM, x1, q2)[:, 0] * xf(QUARKS, x2, q2).sum(1) / (x1 * x2)
    return (-ln_tau_min) * tau * (-ln_tau) * 2.0 * me2 * lum / (2.0 * shat)


def run(st):
    form = st["form"]
    if form == "batch":
        st["batch"].run()
        return st["out"]
    pdf = st["pdf"]
    if form == "xf":
        return pdf.xfxQ2(st["pids"], st["x"], st["q"])
    if form == "xfq":
        return pdf.xfxQ(st["pids"], st["x"], st["q"])
    if form == "xf_alphas":
        return pdf.xfxQ2_alphasQ2(st["pids"], st["x"], st["q"])
    if form == "host":
        return pdf.xfxQ2_host(st["pids"], st["x"], st["q"], out=st["out"])
    if form == "alphas":
        return pdf.alphasQ2(st["q"])
    if form in ("fit", "fit_pw"):
        f = autograd.xfxQ2 if form == "fit" else autograd.xfxQ2_pw
        out = f(pdf, st["values"], st["pids"], st["x"], st["q"])
        return [out.detach(), *torch.autograd.grad(out, (st["values"], st["x"], st["q"]), st["w"])]
    if form == "lumi":
        return luminosity(pdf, st["events"])
    if form == "lumi_fit":
        L = autograd.lumi(pdf, st["values"], st["events"])
        return [L.detach(), *torch.autograd.grad(L, st["values"])]
    res = Vegas(3, n_bins=st["bins"], device=DEV).integrate(lambda r: _single_top(r, pdf.xfxQ2),
                                                            n_iter=st["iterations"], n_per_iter=st["n"],
                                                            uniforms=st["uniforms"])
    return [np.array([res.integral, res.error]), np.array(res.iterations), res.edges]


# ----------------------------------------------------------------------- work

LOG, PATCH, CUBIC, STENCIL = 15, 30, 6, 32      # flops: a logarithm, a bicubic patch, a cubic, 16 FMAs of a stencil


def work(case):
    """Bytes: inputs read once, outputs written once.  Flops: the interpolation's FP64 arithmetic."""
    form, n = case["form"], case.get("n", 0)
    if form == "batch":
        mean = (case["largest"] - case["smallest"]) / math.log(case["largest"] / case["smallest"])
        pts = case["requests"] * mean
        return {"bytes": pts * (16 + 2 * 8), "flops": pts * (2 * (LOG + 2) + 2 * PATCH)}
    F = case.get("flavours", 13)
    if form in ("xf", "xfq", "host"):
        return {"bytes": n * (16 + 8 * F), "flops": n * (2 * (LOG + 2) + F * PATCH)}
    if form == "xf_alphas":
        return {"bytes": n * (24 + 8 * F), "flops": n * (2 * (LOG + 2) + F * PATCH + CUBIC)}
    if form == "alphas":
        return {"bytes": n * 16, "flops": n * (LOG + 2 + CUBIC)}
    if form == "fit_pw":        # x, Q^2, pid, weight in; value and two derivatives out; two passes
        return {"bytes": n * (28 + 24), "flops": n * (2 * (LOG + 2) + 2 * PATCH + 8 + STENCIL)}
    if form == "fit":
        return {"bytes": n * (16 + 16 * F + 16), "flops": n * (2 * (LOG + 2) + F * (2 * PATCH + STENCIL) + 8)}
    F = 13 if case["grid"] == "nnpdf" else 11
    if form == "lumi":
        return {"bytes": n * (8 + 8 + 1 + 16), "flops": n * (10 + 2 * F * PATCH + 2 * F + CUBIC)}
    if form == "lumi_fit":
        return {"bytes": n * 17, "flops": n * (10 + 2 * F * PATCH + 2 * F + 2 * F * STENCIL)}
    it = case["iterations"]     # the uniforms in; the map, five flavours and the sums per point
    return {"bytes": it * n * 24, "flops": it * n * (3 * 4 + 4 * (LOG + 2) + 5 * PATCH + 60)}


# ---------------------------------------------------------------------- exact
#
# The definition in plain float64 torch: per axis the Hermite cubic on the
# interval with finite-difference knot derivatives (one-sided secant at the
# ends of the axis or subgrid, mean of the adjacent secants inside), first in
# ln x, then in ln Q^2 over the rows of the subgrid; outside the knots the
# continuation of the option.  Local coordinates come from log1p of the
# relative distance to the lower knot, which loses nothing next to a knot.

CHUNK = 1 << 19


class _Axis:
    """Knots z_0 < ... of one axis or several subgrids, cell by cell."""

    def __init__(self, parts):
        lo, dz, rho, sig, row, at = [], [], [], [], [], 0
        for z in parts:
            d = [math.log1p((z[k + 1] - z[k]) / z[k]) if z[k + 1] < 2 * z[k] else math.log(z[k + 1] / z[k])
                 for k in range(len(z) - 1)]
            for k in range(len(d)):
                lo.append(z[k])
                dz.append(d[k])
                rho.append(d[k] / d[k - 1] if k > 0 else math.nan)
                sig.append(d[k] / d[k + 1] if k + 1 < len(d) else math.nan)
                row.append(at + k)
            at += len(z)
        self.lo, self.dz, self.rho, self.sig = (torch.tensor(v, dtype=F64, device=DEV) for v in (lo, dz, rho, sig))
        self.row, self.rows = torch.tensor(row, device=DEV), at
        self.first, self.last = parts[0][0], parts[-1][-1]

    def locate(self, v=None, log=None):
        """Cell, local coordinate, inside?, below? of values v, or of their logarithms."""
        if v is None:
            lnlo = torch.log(self.lo)
            c = (torch.searchsorted(lnlo, log.contiguous(), right=True) - 1).clamp_(min=0)
            return c, (log - lnlo[c]) / self.dz[c], (log >= math.log(self.first)) & (log <= math.log(self.last)), \
                log < math.log(self.first)
        c = (torch.searchsorted(self.lo, v.contiguous(), right=True) - 1).clamp_(min=0)
        rel = (v - self.lo[c]) / self.lo[c]
        t = torch.where(rel.abs() < 0.5, torch.log1p(rel), torch.log(v / self.lo[c])) / self.dz[c]
        return c, t, (v >= self.first) & (v <= self.last), v < self.first

    def weights(self, c, t, inside, d=False):
        """Weights of the stencil (knots -1, 0, 1, 2 of the cell), or their derivatives in t."""
        if d:
            h00, h10, h01, h11 = 6 * t * (t - 1), (3 * t - 1) * (t - 1), 6 * t * (1 - t), t * (3 * t - 2)
            line = [torch.zeros_like(t), -torch.ones_like(t), torch.ones_like(t), torch.zeros_like(t)]
        else:
            s = 1 - t
            h00, h10, h01, h11 = s * s * (1 + 2 * t), t * s * s, t * t * (3 - 2 * t), -t * t * s
            line = [torch.zeros_like(t), s, t, torch.zeros_like(t)]
        r, g = self.rho[c], self.sig[c]
        e, f = torch.isnan(r), torch.isnan(g)
        r, g = torch.nan_to_num(r), torch.nan_to_num(g)
        p1 = torch.where(e, -1.0, 0.5 * r - 0.5)
        q1 = torch.where(f, 1.0, 0.5 - 0.5 * g)
        W = [-0.5 * r * h10,
             h00 + p1 * h10 + torch.where(f, -1.0, -0.5) * h11,
             h01 + torch.where(e, 1.0, 0.5) * h10 + q1 * h11,
             0.5 * g * h11]
        return [torch.where(inside, a, b) for a, b in zip(W, line)]


class _Exact:
    def __init__(self, g, extrap="linear", member=0):
        q2 = (g.q_knots * g.q_knots).tolist()
        parts, at = [], 0
        for n in g.n_q:
            parts.append(q2[at:at + int(n)])
            at += int(n)
        self.X, self.Q, self.extrap = _Axis([g.x_knots.tolist()]), _Axis(parts), extrap
        self.V = torch.as_tensor(g.values[member], device=DEV)
        self.A = torch.as_tensor(g.alphas, device=DEV)
        self.col = {int(p): i for i, p in enumerate(g.pids)}

    def at(self, axis, **kw):
        c, t, i, b = axis.locate(**kw)
        if self.extrap == "freeze":
            t = torch.where(i, t, torch.where(b, 0.0, 1.0))
        return c, t, i

    def _sum(self, x, q, wx, wq, cols):
        """sum_j wq_j sum_i wx_i V[row j][knot i][cols]: [n][F], or [n] for one column per point."""
        nx, out = self.V.shape[1], 0.0
        one = isinstance(cols, torch.Tensor)
        flat = self.V.reshape(-1, self.V.shape[2])
        for j in range(4):
            r = (self.Q.row[q[0]] + (j - 1)).clamp(0, self.Q.rows - 1)
            y = 0.0
            for i in range(4):
                k = r * nx + (x[0] + (i - 1)).clamp(0, nx - 1)
                v = flat.view(-1)[k * flat.shape[1] + cols] if one else flat[k][:, cols]
                y = y + (wx[i] if one else wx[i][:, None]) * v
            out = out + (wq[j] if one else wq[j][:, None]) * y
        return out

    def value(self, x, q, cols):
        wx, wq = self.X.weights(x[0], x[1], x[2]), self.Q.weights(q[0], q[1], q[2])
        v = self._sum(x, q, wx, wq, cols)
        if self.extrap != "continuation":
            return v
        out = torch.nonzero(~(x[2] & q[2])).view(-1)
        if out.numel():
            v[out] = self._continued([a[out] for a in x], [a[out] for a in q], cols)
        return v

    def _continued(self, x, q, cols):
        """The power law from the two edge values in Q, then in x (straight lines where one is small)."""
        def law(y0, y1, t):
            t, ok = t[:, None], (y0 > 1e-3) & (y1 > 1e-3)
            p = torch.where(ok, y0, 1.0) * torch.exp(t * torch.log(torch.where(ok, y1, 1.0) / torch.where(ok, y0, 1.0)))
            return torch.where(ok, p, y0 + t * (y1 - y0))

        def unit(k):
            z, o = torch.zeros_like(x[1]), torch.ones_like(x[1])
            return [o if i == k else z for i in range(4)]

        def in_q(wx):
            inner = self._sum(x, q, wx, self.Q.weights(q[0], q[1], torch.ones_like(q[2])), cols)
            edge = law(self._sum(x, q, wx, unit(1), cols), self._sum(x, q, wx, unit(2), cols), q[1])
            return torch.where(q[2][:, None], inner, edge)
        mid = in_q(self.X.weights(x[0], x[1], torch.ones_like(x[2])))
        edge = law(in_q(unit(1)), in_q(unit(2)), x[1])
        return torch.where(x[2][:, None], mid, edge)

    def alphas(self, q):
        w = self.Q.weights(q[0], q[1], q[2])
        return sum(w[j] * self.A[(self.Q.row[q[0]] + (j - 1)).clamp(0, self.Q.rows - 1)] for j in range(4))

    def scatter(self, G, x, q, wt, cols):
        """G[row j][knot i][cols] += wt Wq_j Wx_i."""
        wx, wq = self.X.weights(x[0], x[1], x[2]), self.Q.weights(q[0], q[1], q[2])
        nx, F = self.V.shape[1], self.V.shape[2]
        for j in range(4):
            r = (self.Q.row[q[0]] + (j - 1)).clamp(0, self.Q.rows - 1)
            for i in range(4):
                k = r * nx + (x[0] + (i - 1)).clamp(0, nx - 1)
                w = wq[j] * wx[i]
                if isinstance(cols, torch.Tensor):
                    G.view(-1).index_add_(0, k * F + cols, w * wt)
                else:
                    full = torch.zeros((k.numel(), F), dtype=F64, device=DEV)
                    full[:, cols] = w[:, None] * wt
                    G.view(-1, F).index_add_(0, k, full)

    def slopes(self, x, q, xv, qv, cols):
        """d/dx and d/dQ^2 of the value."""
        wx, wq = self.X.weights(x[0], x[1], x[2]), self.Q.weights(q[0], q[1], q[2])
        dx, dq = self.X.weights(x[0], x[1], x[2], d=True), self.Q.weights(q[0], q[1], q[2], d=True)
        gx, gq = self._sum(x, q, dx, wq, cols), self._sum(x, q, wx, dq, cols)
        sx, sq = 1.0 / (self.X.dz[x[0]] * xv), 1.0 / (self.Q.dz[q[0]] * qv)
        return (gx * sx, gq * sq) if gx.dim() == 1 else (gx * sx[:, None], gq * sq[:, None])


def _chunks(n):
    return [slice(a, min(n, a + CHUNK)) for a in range(0, n, CHUNK)]


def _exact_vegas(case, seed, E):
    nb, dim = case["bins"], 3
    edges, shift, ests = np.tile(np.linspace(0.0, 1.0, nb + 1), (dim, 1)), 0.0, []

    def xf(pids, x, q2):
        return E.value(E.at(E.X, v=x), E.at(E.Q, v=q2), [E.col[int(p)] for p in pids])
    for v in _uniforms(case, seed):
        e = torch.as_tensor(edges, device=DEV)
        s1 = s2 = 0.0
        sums = torch.zeros(dim, nb, dtype=F64, device=DEV)
        for sl in _chunks(case["n"]):
            vn = v[sl] * nb
            b = vn.long().clamp_(0, nb - 1)
            r, jac = torch.empty_like(vn), 1.0
            for d in range(dim):
                width = e[d, b[:, d] + 1] - e[d, b[:, d]]
                r[:, d] = e[d, b[:, d]] + (vn[:, d] - b[:, d]) * width
                jac = jac * (nb * width)
            w = _single_top(r, xf) * jac
            s1, s2 = s1 + float(w.sum()), s2 + float(((w - shift) ** 2).sum())
            for d in range(dim):
                sums[d].index_add_(0, b[:, d], w * w)
        n = case["n"]
        mean = s1 / n
        var = max(s2 / n - (mean - shift) ** 2, 0.0) / (n - 1)
        ests.append([mean, math.sqrt(var)])
        shift = mean
        for d in range(dim):            # smooth, damp, and move the edges to equal shares
            w2, old = sums[d].cpu().numpy(), edges[d].copy()
            sm = np.empty(nb)
            sm[0], sm[-1] = 0.5 * (w2[0] + w2[1]), 0.5 * (w2[-2] + w2[-1])
            sm[1:-1] = (w2[:-2] + w2[1:-1] + w2[2:]) / 3.0
            f = sm / sm.sum()
            damp = ((1.0 - f) / np.log(1.0 / f)) ** 1.5
            acc, k, share = 0.0, 0, damp.sum() / nb
            for j in range(1, nb):
                while acc + damp[k] <= j * share:
                    acc, k = acc + damp[k], k + 1
                edges[d, j] = old[k] + (j * share - acc) / damp[k] * (old[k + 1] - old[k])
    m, s = (np.array([e[i] for e in ests]) for i in (0, 1))
    wt = 1.0 / s ** 2
    return [np.array([(wt * m).sum() / wt.sum(), 1.0 / math.sqrt(wt.sum())]), np.array(ests), edges]


def exact(case, seed):
    form = case["form"]
    if form == "batch":
        sets = _batch_sets()
        outs = []
        for s, m, pids, x, q2 in _batch_requests(case, seed, sets):
            E = _Exact(sets[s], member=m)
            v = torch.cat([E.value(E.at(E.X, v=x[sl]), E.at(E.Q, v=q2[sl]), [E.col[int(p)] for p in pids])
                           for sl in _chunks(x.numel())]).reshape(-1)
            outs.append(torch.nn.functional.pad(v, (0, _row(v.numel()) - v.numel())))
        return torch.cat(outs)
    g = _grid(case, seed)
    E = _Exact(g, case.get("extrap", "linear"))
    gen, n = _gen(seed), case["n"]
    if form in ("xf", "xfq", "xf_alphas", "host"):
        cols = [E.col[int(p)] for p in _pids(g, case["flavours"], seed)]
        x, q2 = _points(g, gen, n, case["outside"])
        if form == "xfq":
            q2 = torch.sqrt(q2) ** 2
        out, a = torch.empty((n, len(cols)), dtype=F64, device=DEV), torch.empty(n, dtype=F64, device=DEV)
        for sl in _chunks(n):
            X, Q = E.at(E.X, v=x[sl]), E.at(E.Q, v=q2[sl])
            out[sl], a[sl] = E.value(X, Q, cols), E.alphas(Q)
        if form != "xf_alphas":
            return out
        return out, None if E.extrap == "continuation" else a
    if form == "alphas":
        q2 = _scales(g, gen, n, case["outside"])
        return torch.cat([E.alphas(E.at(E.Q, v=q2[sl])) for sl in _chunks(n)])
    if form in ("fit", "fit_pw"):
        pids = _pids(g, case["flavours"], seed)
        x, q2 = _points(g, gen, n, case["outside"])
        G = torch.zeros_like(E.V)
        out, gx, gq = [], [], []
        cols = [E.col[int(p)] for p in pids]
        if form == "fit":
            w = torch.randn((n, pids.size), generator=gen, dtype=F64, device=DEV)
        else:
            at = torch.randint(pids.size, (n,), generator=gen, device=DEV)
            every = torch.tensor(cols, device=DEV)[at]
            w = torch.randn(n, generator=gen, dtype=F64, device=DEV)
        for sl in _chunks(n):
            c = cols if form == "fit" else every[sl]
            X, Q = E.at(E.X, v=x[sl]), E.at(E.Q, v=q2[sl])
            out.append(E.value(X, Q, c))
            dx, dq = E.slopes(X, Q, x[sl], q2[sl], c)
            gx.append((dx * w[sl]).sum(1) if form == "fit" else dx * w[sl])
            gq.append((dq * w[sl]).sum(1) if form == "fit" else dq * w[sl])
            E.scatter(G, X, Q, w[sl], c)
        return [torch.cat(out), G[None], torch.cat(gx), torch.cat(gq)]
    if form in ("lumi", "lumi_fit"):
        ev = _events(g, gen, n, case["outside"])
        every = list(range(g.n_flav))           # ascending, symmetric pids: column a pairs with F - 1 - a
        G, lum, a = torch.zeros_like(E.V), [], []
        for sl in _chunks(n):
            h, f = 0.5 * ev.ln_tau[sl], ev.flags[sl]
            w = torch.where((f & 1) > 0, ev.ln_mu2[sl], ev.ln_tau[sl] + ev.ln_s)
            u1 = torch.where((f & 2) > 0, ev.ln_x1[sl], h + ev.y[sl])
            X1, X2, Q = E.at(E.X, log=u1), E.at(E.X, log=h - ev.y[sl]), E.at(E.Q, log=w)
            p1, p2 = E.value(X1, Q, every), E.value(X2, Q, every)
            lum.append((p1 * p2.flip(1)).sum(1))
            a.append(E.alphas(Q))
            if form == "lumi_fit":
                E.scatter(G, X1, Q, p2.flip(1) / n, every)
                E.scatter(G, X2, Q, p1.flip(1) / n, every)
        lum = torch.cat(lum)
        return [lum.mean(), G[None]] if form == "lumi_fit" else (lum.mean(), lum, torch.cat(a))
    return _exact_vegas(case, seed, E)
