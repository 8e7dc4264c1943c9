"""The work a user of this framework has it do, as measurable cases.

A case is one call of a public entry point: the nonlinear-interference
coefficient eta (``Engine.eta``), the SNR of every channel (``Engine.snr``),
eta of many launch-power profiles (``Engine.eta_batched``) and the throughput
with its gradient (``optim.throughput`` and ``backward``), over the plans,
grids and options of this repository's workloads, tests and benchmark.

The FP32 path's results are held as float32, the precision that path computes
in (``optim.throughput`` takes and returns float32 powers and gradients by
itself); the FP64 path's stay float64.

``exact`` evaluates the same Riemann sums in 64 bits with plain torch, written
from the model's definitions: every grid point, every z-step, the profile
rho(z, F) tabulated per channel as ln rho = a + b (F - f_c).
"""
import math

import numpy as np
import torch

from paper_2401_18022_gb300 import api, optim
from paper_2401_18022_gb300 import workloads as W

C_NM_PER_PS = 299792.458
PLANCK = 6.62607015e-34

DEFAULTS = {"plan": "uwb", "n": 589, "plan_seed": 1, "G": 64, "edges": 113, "cells": 0, "g_mci": 0, "raman": 0,
            "spans": 1, "trx": 0.0, "fp64": 0, "host": 0, "profiles": 1}


def listed():
    return [
        # The smallest call: an interactive SNR query on a 5-channel link, host arrays in and out.
        {"name": "tiny_snr_host", "kind": "snr", "plan": "tiny", "n": 5, "cells": 1, "host": 1},
        # The smallest gradient: one step of a launch-power optimiser on the same link with transceiver noise.
        {"name": "tiny_grad", "kind": "grad", "plan": "tiny", "n": 5, "cells": 1, "trx": 20.0},
        # The plain FP64 path, used to check the FP32 path on a small plan.
        {"name": "tiny_eta_fp64", "kind": "eta", "plan": "tiny", "n": 5, "cells": 1, "fp64": 1},
        # The O band at zero dispersion, every cell of the plane on the full grid (piece lists with MCI cells).
        {"name": "oband_eta", "kind": "eta", "plan": "oband", "n": 41, "cells": 1},
        # The same band with the Raman-ODE profile, as an optimiser differentiates it, on a coarse grid.
        {"name": "oband_raman_grad", "kind": "grad", "plan": "oband", "n": 41, "cells": 1, "G": 32, "raman": 1},
        # One band's worth of neighbouring channels over three spans with transceiver noise, an odd grid.
        {"name": "band65_snr_3spans", "kind": "snr", "plan": "block", "n": 65, "plan_seed": 3, "G": 127, "edges": 97,
         "spans": 3, "trx": 20.0},
        # The headline evaluation: 589 channels over 1260-1675 nm on the benchmark's grid.
        {"name": "uwb589_snr", "kind": "snr", "G": 256},
        # The fine stage of the power-segment optimiser: 557 channels with guard bands, adjoint gradient.
        {"name": "uwb557_grad", "kind": "grad", "plan": "guarded", "n": 557, "G": 128},
        # Many launch-power profiles over three uneven plans in one persistent launch.
        {"name": "batch12_eta", "kind": "batch", "profiles": 12},
        # The whole band with the Raman-ODE profile and every MCI cell on its own grid.
        {"name": "uwb557_raman_mci_snr", "kind": "snr", "plan": "guarded", "n": 557, "cells": 1, "g_mci": 8, "raman": 1},
        # The coarse stage of the optimiser with the Raman-ODE profile.
        {"name": "uwb557_raman_grad", "kind": "grad", "plan": "guarded", "n": 557, "raman": 1},
        # The gradient through the MCI cells of a separate grid, on a thinned-out plan.
        {"name": "subset295_mci_grad", "kind": "grad", "plan": "subset", "n": 295, "cells": 1, "g_mci": 8},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """A call of one of the listed forms: plan, grid, options drawn over the listed ranges."""
    while True:
        kind = rng.choice(["snr", "snr", "grad", "grad", "eta", "batch"])
        case = {"kind": kind, "G": _log_int(rng, 16, 256), "edges": rng.choice([41, 77, 97, 113, 113, 113]),
                "plan": rng.choice(["block", "subset", "subset"]), "n": _log_int(rng, 5, 589),
                "plan_seed": rng.randrange(1 << 20)}
        if kind == "batch":
            case.update(plan="uwb", n=589, profiles=rng.randrange(3, 25), G=_log_int(rng, 16, 96))
        elif kind == "eta" and rng.random() < 0.5:
            case.update(fp64=1, plan="block", n=rng.randrange(3, 10), G=_log_int(rng, 16, 64), cells=rng.randrange(2))
        else:
            case["raman"] = int(rng.random() < 0.35)
            case["spans"] = rng.choice([1, 1, 1, 3, 10])
            case["trx"] = rng.choice([0.0, 0.0, 20.0])
            if case["n"] <= 41 and rng.random() < 0.5:
                case.update(cells=1, plan="block")
            elif rng.random() < 0.3 and not (kind == "grad" and case["raman"]):
                case.update(cells=1, g_mci=rng.randrange(3, 17))
            if kind == "snr" and rng.random() < 0.2:
                case["host"] = 1
        if _cost(case) <= _cost(listed()[6]):
            return case


# ---------------------------------------------------------------------------
# sizes
# ---------------------------------------------------------------------------
def _full(case):
    return {**DEFAULTS, **case}


def _sizes(case):
    """(pieces with G rows, MCI cells with g_mci rows) of one pass, mirror cells counted once."""
    c = _full(case)
    if c["kind"] == "batch":
        sizes = [(589, 295, 147)[p % 3] for p in range(c["profiles"])]
    else:
        sizes = [c["n"]]
    pieces = sum(n * (3 + 2 * (n - 1)) for n in sizes)
    mci = 0
    if c["cells"]:
        cells = c["n"] * (c["n"] - 1) * c["n"] // 2
        if c["g_mci"]:
            mci = cells
        else:
            pieces += cells
    return pieces, mci


def _cost(case):
    """Grid points of one pass, weighted by how much more a point of that form takes."""
    c = _full(case)
    pieces, mci = _sizes(c)
    grad = c["kind"] == "grad"
    points = pieces * c["G"] ** 2 * (2.3 if grad else 1.0) + mci * c["g_mci"] ** 2 * (5.0 if grad else 2.5)
    return points * (600 if c["fp64"] else 1) * (1.6 if c["raman"] else 1.0)


def work(case):
    """Along one grid row (constant upsilon1) the integrand is a function of F_c alone, and the rows of a piece have
    phases far apart, so a z-sum of every row is the least that the Riemann sums take: 8 operations per row and
    z-step (one complex multiply-add with its weight), twice that with the gradient."""
    c = _full(case)
    pieces, mci = _sizes(c)
    rows = pieces * c["G"] + mci * c["g_mci"]
    per_ch = 8 * (2 + 6)                          # powers and plan in, up to three outputs
    n = sum((589, 295, 147)[p % 3] for p in range(c["profiles"])) if c["kind"] == "batch" else c["n"]
    return {"bytes": per_ch * n, "flops": (16 if c["kind"] == "grad" else 8) * rows * (c["edges"] - 1)}


# ---------------------------------------------------------------------------
# what a user's program has in hand
# ---------------------------------------------------------------------------
def _scenario(c):
    kw = {"G": c["G"], "n_edges": c["edges"], "cell_set": c["cells"]}
    if c["plan"] == "tiny":
        wl = W.tiny(**kw)
    elif c["plan"] == "oband":
        wl = W.oband(**kw)
    elif c["plan"] == "guarded":
        wl = W.uwb_guarded(**kw)
    else:
        wl = W.uwb(**kw)
        rng = np.random.default_rng(c["plan_seed"])
        if c["plan"] == "block":                  # neighbouring slots
            lo = int(rng.integers(0, wl.n_ch - c["n"] + 1))
            wl = W.subset_plan(wl, np.arange(lo, lo + c["n"]), "block")
        elif c["plan"] == "subset":               # slots picked at random
            wl = W.subset_plan(wl, rng.choice(wl.n_ch, size=c["n"], replace=False), "subset")
    if c["raman"]:
        wl = W.raman(wl)
    return wl.with_(n_spans=c["spans"], snr_trx_dB=c["trx"], G_mci=c["g_mci"])


def _powers(n, seed):
    """Launch powers [W] as the batched workload draws them: dBm ~ N(1, 1.5^2) clipped to [-4, 5]."""
    rng = np.random.default_rng([int(seed), n])
    return W.dbm_to_w(np.clip(rng.normal(1.0, 1.5, size=n), -4.0, 5.0))


def _inputs(c, seed):
    """(workload, powers as a numpy array of the type the call takes)."""
    if c["kind"] == "batch":
        bw = W.batched(n_prof=c["profiles"], G=c["G"], n_edges=c["edges"])
        return bw, np.concatenate([_powers(bw.plans[k].n_ch, seed * 64 + p) for p, k in enumerate(bw.plan_of_profile)])
    wl = _scenario(c)
    P = _powers(wl.n_ch, seed)
    return wl, P.astype(np.float32) if c["kind"] == "grad" else P


def prepare(case, seed):
    c = _full(case)
    wl, P = _inputs(c, seed)
    if not c["host"]:
        P = torch.from_numpy(P).cuda()
        if c["kind"] == "grad":
            P.requires_grad_(True)
    return {"engine": api.engine(0), "kind": c["kind"], "wl": wl, "P": P,
            "precision": api.PREC_FP64 if c["fp64"] else api.PREC_FP32}


def _f32(x):
    return x.astype(np.float32) if isinstance(x, np.ndarray) else x.float()


def run(state):
    eng, wl, P, prec = state["engine"], state["wl"], state["P"], state["precision"]
    if state["kind"] == "grad":
        T = optim.throughput(P, eng, wl)
        (g,) = torch.autograd.grad(T, P)
        return {"T": T.detach(), "dT_dP": g}
    if state["kind"] == "batch":
        return {"eta": _f32(eng.eta_batched(wl, P))}
    if state["kind"] == "snr":
        r = eng.snr(wl, P, precision=prec)
        return {"snr": _f32(r["snr"]), "eta": _f32(r["eta"]), "T": r["T"]}
    r = eng.eta(wl, P, precision=prec)
    return r if prec == api.PREC_FP64 else {k: _f32(v) for k, v in r.items()}


# ---------------------------------------------------------------------------
# the same sums in 64 bits
# ---------------------------------------------------------------------------
EXACT_POINT_STEPS = 2e10          # a few seconds of FP64 work on the GPU; a gradient takes about four times as much


def exact(case, seed):
    c = _full(case)
    pieces, mci = _sizes(c)
    steps = (pieces * c["G"] ** 2 + mci * c["g_mci"] ** 2) * (c["edges"] - 1) * (4 if c["kind"] == "grad" else 1)
    if steps > EXACT_POINT_STEPS:
        return None
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    wl, P = _inputs(c, seed)
    if c["kind"] == "batch":
        out, off = [], 0
        for k in wl.plan_of_profile:
            n = wl.plans[k].n_ch
            out.append(_Model(wl.plans[k], P[off:off + n], dev).eta()[0])
            off += n
        return {"eta": torch.cat(out)}
    m = _Model(wl, P, dev)
    if c["kind"] == "grad":
        return m.gradient()
    eta, pnli, sigma = m.eta()
    if c["kind"] == "eta":
        return {"eta": eta, "pnli": pnli, "sigma": sigma}
    snr, T = m.snr(sigma)
    return {"snr": snr, "eta": eta, "T": float(T)}


class _Model:
    """One plan and one launch-power profile in float64 torch."""

    def __init__(self, wl, P, dev):
        t = lambda x: torch.as_tensor(np.asarray(x, dtype=np.float64), device=dev)  # noqa: E731
        self.wl, self.dev, self.n = wl, dev, wl.n_ch
        self.f, self.B, self.alpha, self.nf = t(wl.f_THz), t(wl.B_THz), t(wl.alpha_per_km), t(wl.nf_dB)
        self.P = t(P)
        lam = C_NM_PER_PS / wl.f_ref_THz
        w = 2.0 * math.pi * C_NM_PER_PS
        self.b2 = -wl.D_ref * lam ** 2 / w
        self.b3 = lam ** 3 / w ** 2 * (2.0 * wl.D_ref + wl.S_ref * lam)
        self.b4 = -lam ** 4 / w ** 3 * (6.0 * wl.D_ref + 6.0 * wl.S_ref * lam + wl.Sdot_ref * lam ** 2)
        if wl.gamma_fixed is not None:
            self.gamma = torch.full_like(self.f, wl.gamma_fixed)
        else:
            self.gamma = t(2e3 * math.pi * wl.n2_m2_per_W / (wl.lambda_nm * 1e-9 * wl.aeff_um2 * 1e-12))
        M, a = wl.n_edges - 1, wl.alpha_R_per_km
        ze = t(-np.log(1.0 - np.arange(M + 1) / M * (1.0 - math.exp(-a * wl.L_km))) / a)
        ze[-1] = wl.L_km
        self.ze, self.z, self.dz = ze, 0.5 * (ze[1:] + ze[:-1]), ze[1:] - ze[:-1]

    # -- the power profile: ln rho(z_m, F) = a[c, m] + b[c, m] (F - f_c) and ln rho(L, f_c)
    def tables(self, P):
        if self.wl.profile == 1:
            return self._raman(P)
        z = torch.cat([self.z, self.ze[-1:]])
        kap = P.sum() * self.wl.Cr * (-torch.expm1(-self.wl.alpha_R_per_km * z)) / self.wl.alpha_R_per_km
        x = 0.5 * kap[None] * self.B[:, None]
        rel = (self.f - self.wl.f_ref_THz)[:, None]
        small = x.abs() < 1e-4
        xs = torch.where(small, torch.ones_like(x), x)
        sinhc = torch.where(small, 1.0 + x * x / 6.0, torch.sinh(xs) / xs)
        lnN = torch.logsumexp(torch.log(P)[:, None] - kap[None] * rel + torch.log(sinhc), 0)
        a = -self.alpha[:, None] * z[None] + torch.log(P.sum()) - lnN[None] - kap[None] * rel
        return a[:, :-1], (-kap[None] * torch.ones_like(rel))[:, :-1], a[:, -1]

    def _raman(self, P):
        wl, f = self.wl, self.f
        d = f[None, :] - f[:, None]                       # f_k - f_i
        h = torch.where(d > 0, d, d * (f[:, None] / f[None, :]) if wl.raman_photon else d)
        if wl.raman_max_THz > 0:
            h = torch.where(d.abs() <= wl.raman_max_THz, h, torch.zeros_like(h))
        if wl.raman_scale is not None:
            h = h * torch.as_tensor(np.asarray(wl.raman_scale), device=self.dev)[:, None]
        h = h * wl.Cr
        rhs = lambda y: h @ torch.exp(y) - self.alpha  # noqa: E731
        y0 = y = torch.log(P)
        mid = []
        for dz in self.dz.tolist():
            ns = max(1, math.ceil(0.5 * dz / wl.ode_h_km - 1e-9))
            for half in range(2):
                s = 0.5 * dz / ns
                for _ in range(ns):
                    k1 = rhs(y)
                    k2 = rhs(y + 0.5 * s * k1)
                    k3 = rhs(y + 0.5 * s * k2)
                    k4 = rhs(y + s * k3)
                    y = y + s / 6.0 * (k1 + 2.0 * k2 + 2.0 * k3 + k4)
                if half == 0:
                    mid.append(y - y0)
        a = torch.stack(mid, 1)
        if self.n == 1:
            return a, torch.zeros_like(a), y - y0
        r = a + self.alpha[:, None] * self.z[None]
        idx = torch.arange(self.n, device=self.dev)
        lo, hi = (idx - 1).clamp(min=0), (idx + 1).clamp(max=self.n - 1)
        return a, (r[hi] - r[lo]) / (f[hi] - f[lo])[:, None], y - y0

    # -- the cells of one CUT cut into quadrants, each with its grid; mirror cells (b, a) counted in the weight
    def pieces(self, i):
        f, B, wl = self.f.tolist(), self.B.tolist(), self.wl

        def split(c):
            lo, hi = f[c] - 0.5 * B[c] - f[i], f[c] + 0.5 * B[c] - f[i]
            out = []
            if hi > 0:
                out.append((1.0, max(lo, 0.0), hi))
            if lo < 0:
                out.append((-1.0, max(-hi, 0.0), -lo))
            return out

        parts = [split(c) for c in range(self.n)]
        by_grid = {}
        if wl.cell_set == 0:
            cells = [(min(a, i), max(a, i)) for a in range(self.n)]
        else:
            cells = [(a, b) for a in range(self.n) for b in range(a, self.n)]
        for a, b in cells:
            G = wl.G if a == i or b == i or wl.G_mci == 0 else wl.G_mci
            for s1, xl, xh in parts[a]:
                for s2, yl, yh in parts[b]:
                    by_grid.setdefault(G, []).append((a, b, s1, s2, xl, xh, yl, yh, 1.0 if a == b else 2.0))
        return by_grid

    def chunk_sum(self, i, G, ps, a, b, psd):
        """Sum over the grids of some pieces of CUT i."""
        wl = self.wl
        cols = list(zip(*ps))
        ia, ib = (torch.tensor(v, device=self.dev) for v in cols[:2])
        s1, s2, xl, xh, yl, yh, mult = (torch.tensor(v, dtype=torch.float64, device=self.dev)[:, None] for v in cols[2:])
        lhi = torch.log(xh * yh)
        llo = torch.log(torch.maximum(xl * yl, wl.eps_v1 * xh * yh))
        k = torch.arange(G, dtype=torch.float64, device=self.dev) + 0.5
        ds = (lhi - llo) / G
        u1 = torch.exp(llo + k[None] * ds)                                       # [piece, row]
        ymin = torch.maximum(yl, u1 / xh)
        ymax = torch.where(xl > 0, torch.minimum(yh, u1 / xl.clamp(min=1e-300)), yh)
        live = ymax > ymin
        ymax = torch.where(live, ymax, 2 * ymin)
        du2 = torch.log(ymax / ymin) / G
        w = torch.where(live, u1 * ds * du2, torch.zeros_like(u1)) * mult
        y = ymax[..., None] * torch.exp(-k * du2[..., None])                     # [piece, row, column]
        f1 = s1[..., None] * (u1[..., None] / y)
        f2 = s2[..., None] * y
        fi = float(self.f[i])
        Fc = fi + f1 + f2
        cc = torch.searchsorted(self.f - 0.5 * self.B, Fc, right=True) - 1
        ok = (cc >= 0) & (Fc < (self.f + 0.5 * self.B)[cc.clamp(min=0)]) & live[..., None]
        p, r, j = torch.nonzero(ok, as_tuple=True)
        f1, f2, Fc, cc = f1[p, r, j], f2[p, r, j], Fc[p, r, j], cc[p, r, j]
        ca, cb, fo = ia[p], ib[p], fi - wl.f_ref_THz
        br = self.b2 + math.pi * self.b3 * (f1 + f2 + 2 * fo) + 2 * math.pi ** 2 / 3 * self.b4 * (
            f1 * f1 + 1.5 * f1 * f2 + 3 * f1 * fo + f2 * f2 + 3 * f2 * fo + 3 * fo * fo)
        phi = -4 * math.pi ** 2 * f1 * f2 * br
        lnp = 0.5 * (a[ca] + b[ca] * (fi + f1 - self.f[ca])[:, None] + a[cb] + b[cb] * (fi + f2 - self.f[cb])[:, None]
                     + a[cc] + b[cc] * (Fc - self.f[cc])[:, None] - a[i])
        amp = torch.exp(lnp) * (self.dz * torch.sinc(phi[:, None] * self.dz / (2 * math.pi)))
        arg = phi[:, None] * self.z
        S2 = (amp * torch.cos(arg)).sum(1) ** 2 + (amp * torch.sin(arg)).sum(1) ** 2
        if wl.n_spans > 1:
            k = torch.arange(wl.n_spans, dtype=torch.float64, device=self.dev) * wl.L_km
            S2 = S2 * (torch.cos(phi[:, None] * k).sum(1) ** 2 + torch.sin(phi[:, None] * k).sum(1) ** 2)
        return (w[p, r] * psd[ca] * psd[cb] * psd[cc] * S2).sum()

    def chunks(self, i, budget=1 << 24):
        for G, ps in self.pieces(i).items():
            step = max(1, budget // (G * G * (self.wl.n_edges - 1)))
            for k in range(0, len(ps), step):
                yield G, ps[k:k + step]

    def sigma(self):
        with torch.no_grad():
            a, b, _ = self.tables(self.P)
            psd = self.P / self.B
            return torch.stack([sum(self.chunk_sum(i, G, ps, a, b, psd) for G, ps in self.chunks(i))
                                for i in range(self.n)])

    def eta(self):
        sigma = self.sigma()
        pnli = 16.0 / 27.0 * self.gamma ** 2 * self.B * sigma
        return pnli / self.P ** 3, pnli, sigma

    def loss(self, sigma, P, aL):
        pnli = 16.0 / 27.0 * self.gamma ** 2 * self.B * sigma
        pase = self.wl.n_spans * 10 ** (self.nf / 10) * PLANCK * (self.f * 1e12) * torch.expm1(-aL) * (self.B * 1e12)
        snr = P / (pnli + pase)
        if self.wl.snr_trx_dB > 0:
            snr = 1.0 / (1.0 / snr + 10 ** (-self.wl.snr_trx_dB / 10))
        return snr, (2 * self.B * torch.log2(1 + snr)).sum()

    def snr(self, sigma):
        with torch.no_grad():
            return self.loss(sigma, self.P, self.tables(self.P)[2])

    def gradient(self):
        P = self.P.clone().requires_grad_(True)
        a, b, aL = self.tables(P)
        psd = P / self.B
        leaf = [t.detach().clone().requires_grad_(True) for t in (a, b, psd)]
        sigma, grads = [], []
        for i in range(self.n):
            tot, g = 0.0, [torch.zeros_like(t) for t in leaf]
            for G, ps in self.chunks(i, 1 << 23):
                s = self.chunk_sum(i, G, ps, *leaf)
                for acc, d in zip(g, torch.autograd.grad(s, leaf)):
                    acc += d
                tot = tot + s.detach()
            sigma.append(tot)
            grads.append(g)
        sg = torch.stack(sigma).requires_grad_(True)
        _, T = self.loss(sg, P, aL)
        (c,) = torch.autograd.grad(T, sg, retain_graph=True)
        back = [sum(ci * g[k] for ci, g in zip(c, grads)) for k in range(3)]
        (gP,) = torch.autograd.grad([T, a, b, psd], [P], [torch.ones_like(T)] + back)
        return {"T": T.detach(), "dT_dP": gP}
