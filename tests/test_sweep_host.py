"""The fixed-point sweeps (csrc/amrfd_sweep.cuh) on the CPU, against rational arithmetic.

The header compiles with a host compiler as a one-lane sweep. Reference: MP5 (Suresh & Huynh
1997) and LIMO3 (Cada & Torrilhon 2009) evaluated in exact fractions on the same doubles. The
sweeps are exact up to one conversion to double wherever a cell's seven-cell window spans at
most 110 bits, so there the results are required to be the correctly rounded ones; beyond,
the cells are rounded to a unit of at most 2^-108 of the window's largest value and the
difference, a sum of magnitudes below 520 of them, is off by less than 2^-98 of it besides
its own rounding. Parts of any length give the same bits and the same recorded pieces.
"""
import ctypes
import math
import os
import shutil
import subprocess
from fractions import Fraction

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1407_2052_gb300", "csrc")

HARNESS = """
#include "amrfd_sweep.cuh"
extern "C" void sweep(int limo, const double* gp, const double* gm, int plen, double thr, double* out,
                      unsigned short* tp, unsigned short* tm, int f0, int fend) {
  using namespace amrfd;
  if (limo) fixed_sweep<true, true>(gp, gm, plen, thr, out, 1, ~0ull, tp, tm, f0, fend, 1 << 30, 1);
  else fixed_sweep<false, true>(gp, gm, plen, 0.0, out, 1, ~0ull, tp, tm, f0, fend, 1 << 30, 1);
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no g++")
    d = tmp_path_factory.mktemp("sweep")
    src, so = d / "h.cpp", d / "h.so"
    src.write_text(HARNESS)
    subprocess.run([gxx, "-O1", "-std=gnu++17", "-ffp-contract=off", "-w", "-shared", "-fPIC", "-I", CSRC, str(src),
                    "-o", str(so)], check=True)
    L = ctypes.CDLL(str(so))
    L.sweep.argtypes = [ctypes.c_int] + [ctypes.c_void_p] * 2 + [ctypes.c_int, ctypes.c_double] + \
        [ctypes.c_void_p] * 3 + [ctypes.c_int] * 2
    return L


def _run(lib, limo, g, h, thr, cuts):
    n = len(g) - 6
    out = np.full(n, np.nan)
    tp, tm = np.full(n + 1, 999, np.uint16), np.full(n + 1, 999, np.uint16)
    for a, b in zip(cuts[:-1], cuts[1:]):
        lib.sweep(limo, g[a:].ctypes.data, h[a:].ctypes.data, b - a, thr, out[a:].ctypes.data, tp.ctypes.data,
                  tm.ctypes.data, a, b + 1)
    return out, tp, tm


def _minmod(a, b):
    return Fraction(0) if a * b <= 0 else (a if abs(a) < abs(b) else b)


def _mp5(a, b, c, d, e):  # G = 2 F: the acceptance threshold 1e-10 on F
    v = (2 * a - 13 * b + 47 * c + 27 * d - 3 * e) / 60
    if (v - c) * (v - c - _minmod(d - c, 4 * (c - b))) <= Fraction(4, 10 ** 10):
        return v

    def m4(p, q):
        return _minmod(_minmod(4 * p - q, 4 * q - p), _minmod(p, q))
    km, k0, kp = a - 2 * b + c, b - 2 * c + d, c - 2 * d + e
    ul, lc, md = c + 4 * (c - b), c + (c - b) / 2 + Fraction(4, 3) * m4(km, k0), (c + d) / 2 - m4(k0, kp) / 2
    lo, hi = max(min(c, d, md), min(c, ul, lc)), min(max(c, d, md), max(c, ul, lc))
    return max(min(v, lo), min(max(v, lo), hi))


def _limo3(b, c, d, thr):
    dm, dp = c - b, d - c
    y3 = (2 * dp + dm) / 3
    s = 1 if dp >= 0 else -1
    yl = s * max(Fraction(0), min(s * y3, max(-s * dm / 2, min(2 * s * dm, s * y3, Fraction(8, 5) * s * dp))))
    z = ((dm * dm + dp * dp) / thr - 1) * 10 ** 12 if thr else Fraction(1)  # the blend band |z| < 1
    z = max(Fraction(-1), min(Fraction(1), z))
    return c + ((1 - z) * y3 + (1 + z) * yl) / 4


def _reference(limo, g, h, thr):
    g, h = [Fraction(float(x)) for x in g], [Fraction(float(x)) for x in h]
    F = []
    for k in range(3, len(g) - 2):
        if limo:
            F.append(_limo3(*g[k - 2:k + 1], Fraction(thr)) + _limo3(h[k + 1], h[k], h[k - 1], Fraction(thr)))
        else:
            F.append(_mp5(*g[k - 3:k + 2]) + _mp5(*h[k + 2:k - 3 if k > 3 else None:-1][:5]))
    return [60 * (a - b) for a, b in zip(F[:-1], F[1:])]


def _line(kind, rng, n):
    j, u = np.arange(n), lambda: rng.uniform(-1, 1, n)
    amp, k, ph = 10.0 ** rng.uniform(-3, 3), rng.uniform(-0.4, 0.4), rng.uniform(0, 6)
    if kind == "smooth":
        return amp * (2 + np.sin(k * j + ph)), -amp * (1.5 + 0.3 * np.cos(k * j))
    if kind == "noise":
        return amp * u(), amp * u()
    if kind == "small_noise":
        return 1 + 1e-3 * u(), -1 + 1e-3 * u()
    if kind == "jump":
        s = j < n // 2
        return np.where(s, 10, 0.03) * (1 + 1e-3 * u()), np.where(s, 8.0, 0.01)
    if kind == "zero_crossing":
        return amp * np.sin(k * j + ph), 0.7 * amp * np.sin(k * j + ph + 0.05)
    if kind == "front":  # into an exactly uniform, and into a vanishing state
        return np.where(j < n // 3, 1 + 1e-2 * u(), 1.0), np.where(j < n // 2, 1e-2 * u(), 0.0)
    if kind == "decay":
        return amp * 10.0 ** (-1.3 * j) * u(), amp * 10.0 ** (-0.9 * j) * u()
    if kind == "wide":
        return amp * 10.0 ** (60 * u()), np.where(rng.random(n) < 0.5, 0.0, amp * 10.0 ** (60 * u()))
    raise ValueError(kind)


KINDS = ("smooth", "noise", "small_noise", "jump", "zero_crossing", "front", "decay", "wide")


@pytest.mark.parametrize("limo", [0, 1], ids=["mp5", "limo3"])
@pytest.mark.parametrize("kind", KINDS)
def test_sweeps_are_correctly_rounded_and_independent_of_their_parts(lib, kind, limo):
    rng = np.random.default_rng(14072052 + KINDS.index(kind))
    for length in (1, 2, 4, 15, 16, 17, 33, 64):
        for _ in range(6):
            g, h = (np.ascontiguousarray(x, dtype=np.float64) for x in _line(kind, rng, length + 6))
            # a switch between the faces' a^2 + b^2 (at it the value jumps), on both sides of them
            thr = 1.37 * float(np.median(np.abs(np.diff(g)))) ** 2 if limo else 0.0
            out, tp, tm = _run(lib, limo, g, h, thr, [0, length])
            cuts = sorted({0, length, *rng.integers(0, length + 1, 3).tolist()})
            again, up, um = _run(lib, limo, g, h, thr, cuts)
            assert out.tobytes() == again.tobytes()
            assert np.array_equal(tp, up) and np.array_equal(tm, um)
            for i, want in enumerate(_reference(limo, g, h, thr)):
                win = [abs(x) for x in (*g[i:i + 7], *h[i:i + 7]) if x]
                top = max(math.frexp(x)[1] for x in win) if win else 0
                low = min(math.frexp(x)[1] for x in win) - 53 if win else 0
                if top - low <= 110:
                    assert out[i] == float(want), (kind, length, i)
                else:
                    tol = Fraction(2) ** (top - 98) + abs(want) * Fraction(2) ** -53
                    assert abs(Fraction(float(out[i])) - want) <= tol, (kind, length, i)


def test_sweeps_mark_windows_that_are_not_finite(lib):
    g, h = np.linspace(1.0, 2.0, 38), np.linspace(-1.0, 1.0, 38)
    for bad in (np.nan, np.inf, -np.inf):
        g2 = g.copy()
        g2[20] = bad
        out, _, _ = _run(lib, 0, g2, h, 0.0, [0, 32])
        want, _, _ = _run(lib, 0, g, h, 0.0, [0, 32])
        hit = np.array([i <= 20 <= i + 6 for i in range(32)])
        assert np.isnan(out[hit]).all() and np.array_equal(out[~hit], want[~hit])
