"""The calls that users of this framework make, as cases that can be timed and compared.

One case is one geometry and one kind of call on it:

  form     the Toeplitz quadratic form of a field that the caller has, by itself
  eval     a new design: set_design, factor, averaged intensity
  grad     a new design with the adjoint gradient (one step of a design loop)
  relight  another objective and light on a design that is already factored
  angles   the brute-force angle average on a design that is already factored
  multi    several output spots on a design that is already factored
  serve    a burst of requests of mixed widths through the evaluation server

A case is a dict of plain values; the geometry follows the workloads of this repository
(20 points per wavelength, pillars of permittivity 5.3 on a substrate of 2.1, widths uniform
in [0.08, 0.36] of a wavelength at the 8-column period, 20 PML cells; thinner ones where
the grid is low).
"""
import math

import numpy as np
import torch

import paper_2207_10701_gb300 as P
import workloads as W

DEV = "cuda" if torch.cuda.is_available() else "cpu"


def listed():
    return [
        # The smallest call: a caller with its own field on the source plane of the 50-cell
        # concentrator wants the quadratic form alone.  Latency and launches are what counts.
        {"name": "form-400", "kind": "form", "n": 400},
        # The 20-wavelength concentrator in double precision (the default precision), one new
        # design: small blocks, few of them, many launches.
        {"name": "eval64-50x128", "kind": "eval", "prec": 64, "cells": 50, "px": 8, "ny": 128,
         "obj": "point", "light": "cone"},
        # Its brute-force average over 201 angles: several right-hand sides in double.
        {"name": "angles64-50x128", "kind": "angles", "prec": 64, "cells": 50, "px": 8, "ny": 128,
         "obj": "point", "light": "cone", "nq": 201},
        # The 200-wavelength collimator in double: the plain form that the others are judged by.
        {"name": "eval64-500x160", "kind": "eval", "prec": 64, "cells": 500, "px": 8, "ny": 160,
         "obj": "plane", "light": "annulus"},
        # The same in the precision form (single with refinement): the headline call.
        {"name": "eval32-500x160", "kind": "eval", "prec": 32, "cells": 500, "px": 8, "ny": 160,
         "obj": "plane", "light": "annulus"},
        # The comparison of the reciprocal value with the brute-force average, 1000 angles.
        {"name": "angles32-500x160", "kind": "angles", "prec": 32, "cells": 500, "px": 8, "ny": 160,
         "obj": "plane", "light": "annulus", "nq": 1000},
        # A designer who compares light sources on one finished design.
        {"name": "relight32-500x160", "kind": "relight", "prec": 32, "cells": 500, "px": 8,
         "ny": 160, "obj": "virtual", "light": "cone"},
        # One iteration of the design loop on the 200-wavelength concentrator.
        {"name": "grad32-500x160", "kind": "grad", "prec": 32, "cells": 500, "px": 8, "ny": 160,
         "obj": "virtual", "light": "cone"},
        # A gradient in double on a grid whose sizes are no multiples of anything: 5-column
        # cells, an odd number of rows.
        {"name": "grad64-77x131", "kind": "grad", "prec": 64, "cells": 77, "px": 5, "ny": 131,
         "obj": "virtual", "light": "annulus"},
        # The 1000-wavelength concentrator in the precision form: 4.5 million unknowns, blocks
        # of 224 rows, 33 GB.
        {"name": "eval32-2500x224", "kind": "eval", "prec": 32, "cells": 2500, "px": 8, "ny": 224,
         "obj": "virtual", "light": "cone"},
        # Twelve output spots of one design at once: a few right-hand sides.
        {"name": "multi32-250x160", "kind": "multi", "prec": 32, "cells": 250, "px": 8, "ny": 160,
         "obj": "virtual", "light": "cone", "outputs": 12},
        # Serving: a burst of requests, 50 to 400 cells, a third of them with the gradient.
        {"name": "serve-24", "kind": "serve", "prec": 32, "requests": 24, "most_cells": 400,
         "ny": 160},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["form", "eval", "eval", "grad", "relight", "angles", "multi", "serve"])
    if kind == "form":
        return {"kind": "form", "n": _log(rng, 100, 20000)}
    if kind == "serve":
        return {"kind": "serve", "prec": 32, "requests": rng.randint(6, 24),
                "most_cells": rng.randint(100, 400), "ny": 2 * rng.randint(56, 88)}
    prec = rng.choice([64, 32])
    ny = rng.randint(48, 224)
    if prec == 32:
        ny += ny & 1  # rows are read in pairs
    px = rng.choice([5, 8, 8, 10])
    # no more work than the largest listed case of the precision: unknowns x ny^2
    most = 500 * 8 * 160 ** 3 if prec == 64 else 2500 * 8 * 224 ** 3
    if kind in ("angles", "multi"):
        most = min(most, 500 * 8 * 160 ** 3) // (20 if prec == 64 else 1)
    cells = max(3, min(_log(rng, 8, 2500), int(0.8 * most / (px * ny ** 3))))
    c = {"kind": kind, "prec": prec, "cells": cells, "px": px, "ny": ny,
         "obj": rng.choice(["point", "plane", "virtual"]), "light": rng.choice(["cone", "annulus"])}
    if kind == "angles":
        c["nq"] = 2 * rng.randint(16, 400)
    if kind == "multi":
        c["outputs"] = rng.randint(2, 24)
    return c


# ---- the problem that a case stands for ------------------------------------------------------


def _desc(c, cells=None):
    # low grids take the thinner layers of the repository's small workloads
    low = c["ny"] < 96
    return W.GridDesc(n_cells=cells or c["cells"], ny=c["ny"], cell_px=c.get("px", 8),
                      npml=10 if low else 20, rows_sub=8 if low else 12, rows_pillar=12,
                      prec=P.FP64 if c["prec"] == 64 else P.FP32_REFINE)


def _objectives(c, d, rng, count=1):
    top = d.npml + d.rows_sub + d.rows_pillar
    width = d.n_cells * d.cell_px / d.ppl
    row = top + (6 if d.ny < 96 else 10)
    nx = d.n_cells * d.cell_px + 2 * d.npml
    out = []
    for k in range(count):
        at = (k + 1) / (count + 1)
        if c["obj"] == "point":
            out.append(W.Objective(W.OBJ_POINT, i_f=int(nx * at),
                                   j_f=min(top + 3 * d.ppl, d.ny - d.npml - 4)))
        elif c["obj"] == "plane":
            out.append(W.Objective(W.OBJ_PLANEWAVE, monitor_row=row,
                                   theta_out=W.deg(rng.uniform(0.0, 10.0))))
        else:
            out.append(W.Objective(W.OBJ_VIRTUAL_FOCUS, monitor_row=row, x_f=width * at,
                                   d_rows=int(round(rng.uniform(5.0, 20.0) * d.ppl))))
    return out


def _light(kind, rng):
    if kind == "cone":
        return W.Light(W.LIGHT_CONE, c=W.deg(rng.uniform(5.0, 40.0)))
    th1 = rng.uniform(5.0, 20.0)
    return W.Light(W.LIGHT_ANNULUS, th1=W.deg(th1), th2=W.deg(th1 + rng.uniform(5.0, 20.0)))


def _widths(d, rng):
    period = d.cell_px / d.ppl
    return rng.uniform(0.2, 0.9, d.n_cells) * period  # [0.08, 0.36] at the 0.4 period


def _problem(c, seed):
    rng = np.random.default_rng(seed)
    d = _desc(c)
    return d, _widths(d, rng), _objectives(c, d, rng, c.get("outputs", 1)), _light(c["light"], rng)


def _burst(c, seed):
    """Widths spread over the logarithm of 50 .. most_cells, in no order (every seed the same);
    designs, objectives and lights from the seed."""
    rng = np.random.default_rng(seed)
    n = c["requests"]
    out = []
    for k in np.random.default_rng(n).permutation(n):
        d = _desc(c, int(round(50 * (c["most_cells"] / 50) ** ((k + 0.5) / n))))
        obj = _objectives({"obj": "virtual" if k % 2 else "plane", "ny": c["ny"]}, d, rng)[0]
        light = _light("cone" if (k // 2) % 2 else "annulus", rng)
        out.append((d, _widths(d, rng), obj, light, k % 3 == 2))
    return out


def _field(c, seed):
    """A field on the source plane and the light's lags, as the quadratic form takes them."""
    rng = np.random.default_rng(seed)
    n = c["n"]
    v = rng.standard_normal(n) + 1j * rng.standard_normal(n)
    lags = _lags(_light("cone", rng), 2 * math.pi * math.sqrt(2.1), 1 / 20, n)
    return torch.from_numpy(v).to(DEV), lags.to(DEV)


# ---- what a user's program has in hand, and its call -----------------------------------------


def prepare(case, seed):
    kind = case["kind"]
    if kind == "form":
        v, lags = _field(case, seed)
        return {"kind": kind, "v": v, "lags": lags}
    if kind == "serve":
        return {"kind": kind, "requests": _burst(case, seed),
                "server": P.Server(slots=6, arena_bytes=24 << 30, lookahead=8)}
    d, widths, objs, light = _problem(case, seed)
    grid = P.Grid(d)
    s = {"kind": kind, "grid": grid, "widths": torch.from_numpy(widths).to(DEV), "obj": objs[0],
         "objs": objs, "light": light, "nq": case.get("nq")}
    if kind == "grad":
        s["widths"] = widths  # the design loop keeps its widths on the host
    if kind in ("relight", "angles", "multi"):
        grid.set_design(s["widths"])
        grid.factor()
    return s


def run(state):
    kind = state["kind"]
    if kind == "form":
        return np.float64(P.qform_toeplitz(state["v"], state["lags"]))
    if kind == "serve":
        s = state["server"]
        tickets = [s.submit(d, w, o, light, want_grad=g) for d, w, o, light, g in state["requests"]]
        got = [s.wait(t) for t in tickets]
        return [[np.float64(r["value"])] + ([] if r["grad"] is None else [r["grad"]]) for r in got]
    g = state["grid"]
    if kind in ("eval", "grad"):
        g.set_design(state["widths"])
        g.factor()
    if kind == "grad":
        value, grad, _ = g.avg_intensity_grad(state["obj"], state["light"])
        return [np.float64(value), grad]
    if kind == "angles":
        value, per_angle, _ = g.avg_bruteforce(state["obj"], state["light"], state["nq"])
        return [np.float64(value), per_angle]
    if kind == "multi":
        per_output, total, _ = g.avg_intensity_multi(state["objs"], state["light"])
        return [per_output, np.float64(total)]
    return np.float64(g.avg_intensity(state["obj"], state["light"])[0])


def work(case):
    """Multiply-adds of a complex number count 8.  Half of the columns are eliminated with a
    tridiagonal matrix; of the other half each costs one inverse and five products of ny x ny
    blocks; a solve with q columns reads (and a factorisation writes) three blocks for each
    of them and multiplies with them five times in all."""
    kind = case["kind"]
    if kind == "form":
        n = case["n"]
        return {"bytes": 24 * n, "flops": 2 * n * n}
    if kind == "serve":
        mean = (case["most_cells"] - 50) / math.log(case["most_cells"] / 50)
        one = dict(case, kind="eval", cells=int(mean), px=8)
        w = work(one)
        return {k: case["requests"] * v for k, v in w.items()}
    d = _desc(case)
    nx, ny = d.n_cells * d.cell_px + 2 * d.npml, d.ny
    size = 16 if case["prec"] == 64 else 8
    kept = nx // 2
    store = kept * 3 * ny * ny * size
    q = case.get("nq", case.get("outputs", 2 if kind == "grad" else 1))
    flops = kept * 5 * 8 * ny ** 2 * q
    moved = store + 2 * 16 * nx * ny * q
    if kind in ("eval", "grad"):
        flops += kept * (6 * 8 * ny ** 3 + 48 * ny ** 2)
        moved += store
    return {"bytes": moved, "flops": flops}


# ---- the same numbers in 64 bits, by plain torch and numpy -------------------------------------


def exact(case, seed):
    kind = case["kind"]
    if kind == "form":
        v, lags = _field(case, seed)
        return _toeplitz_form(v, lags)
    if kind == "serve":
        # the smaller requests only: each takes a factorisation of its own
        out = []
        for d, widths, obj, light, grad in _burst(case, seed):
            if d.n_cells > 120:
                out.append([None, None] if grad else [None])
                continue
            out.append(_Exact(d, widths).value(obj, light, grad))
        return out
    d, widths, objs, light = _problem(case, seed)
    nx = d.n_cells * d.cell_px + 2 * d.npml
    if nx * d.ny ** 3 > 1e11:
        return None
    e = _Exact(d, widths)
    if kind == "grad":
        return e.value(objs[0], light, True)
    if kind == "angles":
        return e.angles(objs[0], light, case["nq"])
    if kind == "multi":
        each = [e.value(o, light, False)[0] for o in objs]
        return [np.array(each), np.float64(sum(each))]
    return e.value(objs[0], light, False)[0]


def _sinc(z):
    return torch.sinc(z / math.pi)


def _lags(light, k_s, h, n):
    x = k_s * h * torch.arange(n, dtype=torch.float64)
    if light.kind == W.LIGHT_CONE:
        s = math.sin(light.c)
        return s / light.c * _sinc(x * s)
    s1, s2 = math.sin(light.th1), math.sin(light.th2)
    return (s2 * _sinc(x * s2) - s1 * _sinc(x * s1)) / (light.th2 - light.th1)


def _toeplitz_times(v, lags):
    n = v.numel()
    at = torch.arange(n, device=v.device)
    out = torch.empty_like(v)
    for i in range(0, n, 1024):
        rows = lags[(at[i:i + 1024, None] - at[None, :]).abs()].to(v.dtype)
        out[i:i + 1024] = rows @ v
    return out


def _toeplitz_form(v, lags):
    return np.float64(torch.vdot(v, _toeplitz_times(v, lags)).real.item())


def _focus_row(d, rows, offsets):
    """K(offset) = h/pi int_0^{pi/h} exp(i q(k) D) cos(k offset) dk through homogeneous air."""
    h, k0, D = 1 / d.ppl, 2 * math.pi, rows
    a = k0 * k0 * h * h * d.eps_air / 2
    kc = math.acos(1 - a) / h
    x, w = (torch.from_numpy(t) for t in np.polynomial.legendre.leggauss(32))
    out = torch.zeros(offsets.numel(), dtype=torch.complex128, device=offsets.device)
    for top, sign in ((math.sqrt(kc), -1), (math.sqrt(math.pi / h - kc), 1)):
        half = top / 512
        mid = (torch.arange(256, dtype=torch.float64) * 2 + 1) * half
        t = (mid[:, None] + half * x).reshape(-1).to(offsets.device)
        wt = (half * w).repeat(256).to(offsets.device)
        k = kc + sign * t * t
        cq = 2 - torch.cos(k * h) - a
        f = torch.exp(1j * D * torch.acos(cq.clamp(-1, 1))) if sign < 0 else \
            torch.exp(-D * torch.acosh(cq.clamp(min=1))).to(torch.complex128)
        f = f * (2 * t * wt)
        for i in range(0, offsets.numel(), 512):
            c = torch.cos(offsets[i:i + 512, None] * k[None, :])
            out[i:i + 512] += torch.complex(c @ f.real, c @ f.imag)
    return out * (h / math.pi)


class _Exact:
    """One design of one geometry: the five-point operator, factored by odd-even reduction over
    the columns in complex128, solves refined once with the operator itself."""

    def __init__(self, d, widths):
        self.d = d
        self.h, self.k0 = 1 / d.ppl, 2 * math.pi
        self.k_s = self.k0 * math.sqrt(d.eps_sub)
        self.n_src = d.n_cells * d.cell_px
        self.nx, self.ny = self.n_src + 2 * d.npml, d.ny
        self.j_src = d.npml + d.src_offset
        self.j0 = d.npml + d.rows_sub
        self.j1 = self.j0 + d.rows_pillar
        self.cols = slice(d.npml, self.nx - d.npml)
        f64 = dict(dtype=torch.float64, device=DEV)
        self.xs = (torch.arange(self.n_src, **f64) + 0.5) * self.h
        h, npml, wide = self.h, d.npml, self.n_src * self.h
        deep = npml * h
        smax = -(d.pml_m + 1) * math.log(d.pml_R0) / (2 * deep)

        def stretch(x, lo, hi):
            depth = torch.clamp(torch.maximum(lo - x, x - hi), min=0)
            return torch.complex(torch.ones_like(depth), smax * (depth / deep) ** d.pml_m / self.k0)

        i, j = torch.arange(self.nx + 1, **f64), torch.arange(self.ny + 1, **f64)
        sx = stretch((i[:-1] - npml + 0.5) * h, 0.0, wide)
        sxh = stretch((i - npml) * h, 0.0, wide)
        sy = stretch((j[:-1] + 0.5) * h, deep, (self.ny - npml) * h)
        syh = stretch(j * h, deep, (self.ny - npml) * h)
        # permittivity: the pillars' share of each column, and its derivative by each width
        w = torch.as_tensor(widths, **f64)
        px, p = d.cell_px, d.cell_px * h
        m = torch.arange(d.n_cells, **f64)
        lo = (torch.arange(self.n_src, **f64)).reshape(d.n_cells, px) * h
        hi = lo + h
        a = ((m + 0.5) * p - w / 2)[:, None]
        b = ((m + 0.5) * p + w / 2)[:, None]
        share = (torch.minimum(hi, b) - torch.maximum(lo, a)).clamp(min=0) / h
        self.dshare = (((lo <= b) & (b < hi)).double() + ((lo < a) & (a <= hi)).double()) / (2 * h)
        eps = torch.full((self.nx, self.ny), d.eps_air, **f64)
        eps[:, :self.j0] = d.eps_sub
        eps[self.cols, self.j0:self.j1] = (d.eps_air + share.reshape(-1) * (d.eps_pillar - d.eps_air))[:, None]
        self.kss = self.k0 ** 2 * sx[:, None] * sy[None, :]
        self.diag = (-sy[None, :] / h ** 2 * (1 / sxh[1:] + 1 / sxh[:-1])[:, None]
                     - sx[:, None] / h ** 2 * (1 / syh[1:] + 1 / syh[:-1])[None, :]
                     + self.kss * eps)
        self.cx = sy[None, :] / h ** 2 / sxh[1:-1, None]
        self.cy = sx[:, None] / h ** 2 / syh[None, 1:-1]
        self._factor()

    def times(self, u):
        out = self.diag * u
        out[:-1] += self.cx * u[1:]
        out[1:] += self.cx * u[:-1]
        out[:, :-1] += self.cy * u[:, 1:]
        out[:, 1:] += self.cy * u[:, :-1]
        return out

    def _factor(self):
        D = torch.diag_embed(self.diag) + torch.diag_embed(self.cy, 1) + torch.diag_embed(self.cy, -1)
        L = torch.diag_embed(self.cx)  # L[i] couples block i+1 to block i; the other side is L[i]^T
        self.levels = []
        while D.shape[0] > 1:
            n = D.shape[0]
            inv = torch.linalg.inv(D[1::2])               # the odd blocks go
            left = inv @ L[0::2]                          # inv(D_k) L_{k-1}: to the block before
            right = inv[:(n - 1) // 2] @ L[1::2].mT       # inv(D_k) L_k^T: to the block after
            E = D[0::2].clone()
            E[:left.shape[0]] -= L[0::2].mT @ left
            if right.shape[0]:
                E[1:1 + right.shape[0]] -= L[1::2] @ right
            M = -(L[1::2] @ left[:right.shape[0]])
            self.levels.append((inv, left, right))
            D, L = E, M
        self.last = torch.linalg.inv(D[0])

    def _once(self, b):
        kept = []
        for inv, left, right in self.levels:
            odd, even = b[1::2], b[0::2].clone()
            even[:left.shape[0]] -= torch.einsum("kij,ki->kj", left, odd)
            if right.shape[0]:
                even[1:1 + right.shape[0]] -= torch.einsum("kij,ki->kj", right, odd[:right.shape[0]])
            kept.append(torch.einsum("kij,kj->ki", inv, odd))
            b = even
        x = (self.last @ b[0])[None]
        for (inv, left, right), y in zip(reversed(self.levels), reversed(kept)):
            y = y - torch.einsum("kij,kj->ki", left, x[:left.shape[0]])
            if right.shape[0]:
                y[:right.shape[0]] -= torch.einsum("kij,kj->ki", right, x[1:1 + right.shape[0]])
            whole = torch.empty(x.shape[0] + y.shape[0], self.ny, dtype=x.dtype, device=x.device)
            whole[0::2], whole[1::2] = x, y
            x = whole
        return x

    def solve(self, b):
        x = self._once(b)
        for _ in range(2):
            x = x + self._once(b - self.times(x))
        return x

    def reciprocal(self, obj):
        """z = A^-1 conj(w)."""
        b = torch.zeros(self.nx, self.ny, dtype=torch.complex128, device=DEV)
        if obj.kind == W.OBJ_POINT:
            b[obj.i_f, obj.j_f] = 1
        elif obj.kind == W.OBJ_PLANEWAVE:
            b[self.cols, obj.monitor_row] = torch.exp(-1j * self.k0 * math.sin(obj.theta_out) * self.xs)
        else:
            b[self.cols, obj.monitor_row] = _focus_row(self.d, obj.d_rows, obj.x_f - self.xs)
        return self.solve(b)

    def value(self, obj, light, grad):
        z = self.reciprocal(obj)
        v = z[self.cols, self.j_src].conj()
        lags = _lags(light, self.k_s, self.h, self.n_src).to(DEV)
        g = _toeplitz_times(v, lags)
        F = np.float64(torch.vdot(v, g).real.item())
        if not grad:
            return [F]
        b = torch.zeros_like(z)
        b[self.cols, self.j_src] = g
        dF = -2 * (self.solve(b) * z * self.kss).real[self.cols, self.j0:self.j1].sum(1)
        dF = dF.reshape(self.dshare.shape) * self.dshare * (self.d.eps_pillar - self.d.eps_air)
        return [F, dF.sum(1).cpu().numpy()]

    def angles(self, obj, light, nq):
        """Since A is symmetric, w^dag A^-1 b0 = z^T b0 for every angle, with one solve."""
        z = self.reciprocal(obj)[self.cols, self.j_src]
        if light.kind == W.LIGHT_CONE:
            x, w = np.polynomial.legendre.leggauss(nq)
            theta, weight = light.c * x, w / 2
        else:
            x, w = np.polynomial.legendre.leggauss(nq // 2)
            half, mid = (light.th2 - light.th1) / 2, (light.th2 + light.th1) / 2
            theta = np.concatenate([half * x - mid, half * x + mid])
            weight = np.concatenate([w, w]) / 4
        t = torch.from_numpy(theta).to(DEV)
        b0 = torch.exp(1j * self.k_s * torch.sin(t)[:, None] * self.xs[None, :])
        f = (torch.cos(t) * (b0 @ z).abs() ** 2).cpu().numpy()
        return [np.float64(np.dot(weight, f)), f]
