"""The node rule of the FP32 row sums (quad_nodes.cuh) in 64 bits: Sigma of a CUT
from nodes, in plain numpy, against the sum over every grid point.  The node
counts come from the header itself (shipped_counts)."""
import ctypes
import functools
import math
import os
import subprocess

import numpy as np

from paper_2401_18022_gb300 import build

MENU = (2, 3, 4, 5, 6, 7, 8, 10, 12, 14, 16, 18, 20, 24, 28, 32, 40, 48)
MAX_N = 256
BLOCK_PHI, LOW_PHI = 6.0, 0.15

SRC = """
#include "quad_nodes.cuh"
extern "C" int run_need(float A, float D) { return isrs::gauss_need(A, D); }
extern "C" int block_need(float A, float D, int part) { return isrs::block_need(A, D, part != 0); }
extern "C" int picked(int n) { return isrs::gauss_nodes(isrs::gauss_pick(n)); }
"""


def shipped_counts(folder):
    """gauss_need, block_need and the menu of the header, compiled for the host."""
    src, lib = os.path.join(folder, "counts.cu"), os.path.join(folder, "counts.so")
    with open(src, "w") as f:
        f.write(SRC)
    subprocess.check_call([build.nvcc(), *build.ARCH, *build.FLAGS, "-shared", "-o", lib, src])
    so = ctypes.CDLL(lib)
    so.run_need.argtypes = [ctypes.c_float, ctypes.c_float]
    so.block_need.argtypes = [ctypes.c_float, ctypes.c_float, ctypes.c_int]
    assert [so.picked(n) for n in range(1, 49)] == [next(m for m in MENU if m >= n) for n in range(1, 49)]
    return so.run_need, so.block_need


@functools.lru_cache(None)
def rule(N, n):
    """n-node Gauss rule of the uniform measure on N points (Golub-Welsch)."""
    i = np.arange(1, n)
    J = np.diag(np.sqrt(i * i * (N * N - i * i) / (N * N * (4.0 * i * i - 1.0))), 1)
    t, V = np.linalg.eigh(J + J.T)
    return t, N * V[0] ** 2


def nodes(N, need):
    """Positions (from the centre, in points) and weights for N points."""
    m = next(m for m in MENU if m >= need) if need <= MENU[-1] else N
    if m >= N:
        return np.arange(N) - 0.5 * (N - 1), np.ones(N)
    t, w = rule(N, m)
    return 0.5 * N * t, w


class Fibre:
    def __init__(self, wl):
        self.wl, self.spans, self.L = wl, wl.n_spans, wl.L_km
        lam, w = 299792.458 / wl.f_ref_THz, 2 * math.pi * 299792.458
        self.b2 = -wl.D_ref * lam ** 2 / w
        self.c3 = math.pi * lam ** 3 / w ** 2 * (2 * wl.D_ref + wl.S_ref * lam)
        self.c4 = -2 * math.pi ** 2 / 3 * lam ** 4 / w ** 3 * (6 * wl.D_ref + 6 * wl.S_ref * lam + wl.Sdot_ref * lam ** 2)
        M, a = wl.n_edges - 1, wl.alpha_R_per_km
        ze = -np.log(1 - np.arange(M + 1) / M * (1 - math.exp(-a * wl.L_km))) / a
        self.z, self.dz = 0.5 * (ze[1:] + ze[:-1]), np.diff(ze)
        self.f, self.B = wl.f_THz - wl.f_ref_THz, wl.B_THz

    def s2(self, phi, at):
        """|S|^2 of all spans, p = e^{-at z}."""
        out = []
        for p, a in zip(np.array_split(phi, 1 + len(phi) // 50000), np.array_split(at, 1 + len(phi) // 50000)):
            amp = np.exp(-a[:, None] * self.z) * self.dz * np.sinc(p[:, None] * self.dz / (2 * math.pi))
            v = np.abs((amp * np.exp(1j * p[:, None] * self.z)).sum(1)) ** 2
            out.append(v * np.abs(np.exp(1j * p[:, None] * self.L * np.arange(self.spans)).sum(1)) ** 2)
        return np.concatenate(out)

    def pieces(self, i):
        def split(c):
            lo, hi = self.f[c] - 0.5 * self.B[c] - self.f[i], self.f[c] + 0.5 * self.B[c] - self.f[i]
            return ([(1.0, max(lo, 0.0), hi)] if hi > 0 else []) + ([(-1.0, max(-hi, 0.0), -lo)] if lo < 0 else [])

        n = len(self.f)
        for a in range(n):
            for b in range(a, n):
                if self.wl.cell_set == 0 and i not in (a, b):
                    continue
                for s1, xl, xh in split(a):
                    for s2, yl, yh in split(b):
                        if a == b and s1 < 0 < s2:
                            continue
                        mult = 2.0 if a != b or s1 != s2 else 1.0
                        axes = ((a, s1, xl, xh), (b, s2, yl, yh))
                        yield Piece(self, i, *(axes if xh >= yh else axes[::-1]), mult)


class Piece:
    def __init__(self, fib, i, first, second, mult):
        (a, self.s1, xl, self.xhi), (b, self.s2, yl, self.yhi) = first, second
        self.fib, self.mult, self.G = fib, mult, fib.wl.G
        self.R = math.log(self.xhi / xl) if xl > 0 else 1e30
        self.Rb = math.log(self.yhi / yl) if yl > 0 else 1e30
        self.ds = min(self.R + self.Rb, -math.log(fib.wl.eps_v1)) / self.G
        fi, U = fib.f[i], self.s1 * self.xhi + self.s2 * self.yhi
        b1 = fib.c3 + 3 * fib.c4 * fi
        self.br0, self.br1 = fib.b2 + fi * (fib.c3 + b1) + U * (fib.c4 * U + b1), 2 * fib.c4 * U + b1
        e = fib.f - fi - U
        self.lo, self.hi = e - 0.5 * fib.B, e + 0.5 * fib.B
        al, P = fib.wl.alpha_per_km, fib.wl.P_W / fib.B
        self.at, self.pd = 0.5 * (al[a] + al[b] + al - al[i]), P * P[a] * P[b] * mult
        self.band = fib.L * fib.spans

    def rows(self, k):
        """Rows k pitches below the corner (k real-valued)."""
        l, R, Rb = -np.asarray(k, float) * self.ds, self.R, self.Rb
        a, b = l > -Rb, l + R < 0
        D = np.where(a, np.where(b, R, -l), np.where(b, l + R + Rb, Rb))
        gx = np.where(a, np.where(b, -0.5 * R, 0.5 * l), np.where(b, 0.5 * (l + Rb - R), l + 0.5 * Rb))
        u1, D = self.xhi * self.yhi * np.exp(l), np.maximum(D, 0.0)
        return [dict(zip(("u1", "D", "w", "lim", "xc", "yc", "u0"), v)) for v in zip(
            u1, D, u1 * self.ds * D / self.G, np.where(D > 0, a + 2 * b, -1), self.xhi * np.exp(gx),
            self.yhi * np.exp(l - gx), self.s1 * self.xhi * np.expm1(gx) + self.s2 * self.yhi * np.expm1(l - gx))]

    def u(self, r, pos):
        d = pos * r["D"] / self.G                       # pos: columns from the row's centre
        return r["u0"] + self.s1 * r["xc"] * np.expm1(d) + self.s2 * r["yc"] * np.expm1(-d)

    def phi(self, r, u):
        ss, c4 = self.s1 * self.s2, self.fib.c4
        return -4 * math.pi ** 2 * ss * r["u1"] * (self.br0 + u * (self.br1 + c4 * u) - 0.5 * c4 * ss * r["u1"])

    def slopes(self, r):
        c = 4 * math.pi ** 2 * r["u1"]
        return c * abs(2 * self.fib.c4 * r["u0"] + self.br1), c * abs(self.fib.c4)

    def turn(self, r):
        if self.s1 != self.s2:
            return 0
        return int(min(max(math.ceil(0.5 * math.log(r["yc"] / r["xc"]) / r["D"] * self.G + 0.5 * self.G - 0.5), 0), self.G))

    def test(self, r):
        """(candidate and limits of a row that lies in one channel, |phi| band)."""
        if r["lim"] < 0:
            return -1, 0.0
        us = [self.u(r, 0.5 - 0.5 * self.G), self.u(r, 0.5 * self.G - 0.5)]
        jm = self.turn(r)
        if 0 < jm < self.G:
            us += [self.u(r, jm - q - 0.5 * (self.G - 1)) for q in (0, 1)]
        p1, p2 = self.slopes(r)
        sw = max(us) - min(us)
        c = [q for q in range(len(self.lo)) if min(us) >= self.lo[q] and max(us) < self.hi[q]]
        return (4 * c[0] + r["lim"] if c else -1), self.band * (abs(self.phi(r, r["u0"])) + sw * (p1 + p2 * sw))

    def units(self, block_need):
        """(k, weight, whether it is a block's, so in one channel) of the rows that stand for all G."""
        G = self.G
        tests = [self.test(r) for r in self.rows(G - np.arange(G) - 0.5)]
        key0, R1 = tests[0][0], 0
        while R1 < G and key0 >= 0 and tests[R1][0] == key0 and tests[R1][1] <= BLOCK_PHI:
            R1 += 1
        out = [(G - r - 0.5, 1.0, False) for r in range(R1, G)]
        if R1 == 0:
            return out
        q = max(t[1] * math.exp((R1 - 1 - r) * self.ds) for r, t in enumerate(tests[:R1]))
        top = min(R1, math.ceil(math.log(q / LOW_PHI) / self.ds)) if q > LOW_PHI else 0
        for r0, n, cap, part in ((0, R1 - top, min(q, LOW_PHI), top > 0), (R1 - top, top, q, False)):
            parts = -(-n // MAX_N)
            for s in range(parts):
                a, N = n * s // parts, n * (s + 1) // parts - n * s // parts
                D = 0.5 * N * self.ds
                pos, w = nodes(N, block_need(cap * D, D, part))
                out += [(G - (r0 + a + 0.5 * N + p), v, True) for p, v in zip(pos, w)]
        return out

    def sigma(self, run_need, block_need):
        phi, at, wt = [], [], []
        units = self.units(block_need)
        for r, (_, wr, whole) in zip(self.rows([k for k, _, _ in units]), units):
            if r["w"] == 0:
                continue
            G = self.G
            u = self.u(r, np.arange(G) + 0.5 - 0.5 * G)
            p1, p2 = self.slopes(r)
            E, hd = math.exp(0.5 * r["D"]), 0.5 * r["D"] / G
            x, y = self.s1 * r["xc"], self.s2 * r["yc"]
            e = max(abs(x * E - y / E), abs(x / E - y * E)) * hd
            per, jm = e * self.band * (p1 + 2 * p2 * e * G), 0 if whole else self.turn(r)
            for ja, jb in ((0, jm), (jm, G)):
                for c in range(len(self.lo)):
                    j = np.flatnonzero((u[ja:jb] >= self.lo[c]) & (u[ja:jb] < self.hi[c])) + ja
                    if not len(j):
                        continue
                    N, parts = len(j), 1
                    n = run_need(per * N, hd * N)
                    if N > MENU[-1] and (n > MENU[-1] or N > MAX_N):
                        parts = min(max(-(-N // MAX_N), (n + 23) // 24), -(-N // MENU[-1]))
                    for s in range(parts):
                        a, b = N * s // parts, N * (s + 1) // parts
                        pos, w = nodes(b - a, run_need(per * (b - a), hd * (b - a)))
                        v = self.u(r, j[0] + 0.5 * (a + b) + pos - 0.5 * G)
                        phi.append(self.phi(r, v))
                        at.append(np.full(len(v), self.at[c]))
                        wt.append(w * (r["w"] * wr * self.pd[c]))
        self.nodes = sum(len(v) for v in phi)
        return float(np.sum(np.concatenate(wt) * self.fib.s2(np.concatenate(phi), np.concatenate(at)))) if wt else 0.0

    def points(self):
        """|phi| of every grid point whose F_c lies in a channel."""
        out = []
        for r in self.rows(self.G - np.arange(self.G) - 0.5):
            if r["w"] > 0:
                u = self.u(r, np.arange(self.G) + 0.5 - 0.5 * self.G)
                ok = ((u[:, None] >= self.lo) & (u[:, None] < self.hi)).any(1)
                out.append(np.abs(self.phi(r, u[ok])))
        return np.concatenate(out) if out else np.zeros(0)

    def full(self):
        """Every grid point."""
        return self.sigma(lambda A, D: 1 << 20, lambda A, D, part: 1 << 20)
