"""The transposed fixed-point sweep (csrc/amrfd_sweep.cuh) on the CPU, against fractions.

With the limiters' pieces fixed, 60 times a face's flux is a whole combination of the cells;
the reference sums the transposed combinations in exact fractions from the formulas of the
pieces. The sweep is exact up to one conversion to double wherever the seven gradients that
reach a cell span at most 106 bits, so there the correctly rounded gradient is required;
beyond, the gradients are rounded to a unit of 2^-106 of the largest and a cell's sum takes
less than 2^13 of them (2^-92 of it).
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
extern "C" void adjoint(int limo, const double* g, int slen, const unsigned short* tp, const unsigned short* tm,
                        int fofs, int n, int wrap, int kb, int ke, int lo, int hi, double* gp, double* gm) {
  using namespace amrfd;
  const TapeLine t = {tp, tm, fofs, n, wrap != 0};
  if (limo) adjoint_sweep<true>(g, slen, t, kb, ke, lo, hi, gp, gm, 1);
  else adjoint_sweep<false>(g, slen, t, kb, ke, lo, hi, gp, gm, 1);
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no g++")
    d = tmp_path_factory.mktemp("adjoint")
    src, so = d / "h.cpp", d / "h.so"
    src.write_text(HARNESS)
    subprocess.run([gxx, "-O1", "-std=gnu++17", "-ffp-contract=off", "-w", "-shared", "-fPIC", "-I", CSRC, str(src),
                    "-o", str(so)], check=True)
    L = ctypes.CDLL(str(so))
    L.adjoint.argtypes = [ctypes.c_int, ctypes.c_void_p, ctypes.c_int, ctypes.c_void_p, ctypes.c_void_p] + \
        [ctypes.c_int] * 7 + [ctypes.c_void_p] * 2
    return L


def _dm4(piece):  # of (ka, kb)
    return [(0, 0), (1, 0), (0, 1), (4, -1), (-1, 4)][piece]


def _weights(limo, code):
    """60 times a face value in its stencil's cells, upwind cell 2 (MP5) or 1 (LIMO3)."""
    if limo:
        mode, piece = (code >> 3) & 3, code & 7
        a, b = [(0, 0), (Fraction(1, 3), Fraction(2, 3)), (Fraction(-1, 2), 0), (2, 0), (0, Fraction(8, 5))][
            1 if mode in (0, 2) else piece]
        return [-30 * a, 60 + 30 * a - 30 * b, 30 * b]
    sel, mp, mm = code & 7, _dm4((code >> 3) & 7), _dm4((code >> 6) & 7)
    if sel == 0:
        return [2, -13, 47, 27, -3]
    w = [Fraction(0)] * 5
    w[2] += 60

    def add(c, i, j):  # c (f_j - f_i)
        w[j] += 60 * Fraction(c)
        w[i] -= 60 * Fraction(c)

    def curv(c, i):  # c (f_{i-1} - 2 f_i + f_{i+1})
        add(c, i, i + 1)
        add(-c, i - 1, i)
    if sel == 2:
        add(1, 2, 3)
    elif sel == 3:
        add(Fraction(1, 2), 2, 3)
        curv(Fraction(-mp[0], 2), 2)
        curv(Fraction(-mp[1], 2), 3)
    elif sel == 4:
        add(4, 1, 2)
    elif sel == 5:
        add(Fraction(1, 2), 1, 2)
        curv(Fraction(4 * mm[0], 3), 1)
        curv(Fraction(4 * mm[1], 3), 2)
    return w


def _codes(limo, rng, n, share):
    if limo:
        c = (rng.integers(0, 3, n) << 3) | rng.integers(0, 5, n)
    else:
        sel = rng.integers(1, 6, n)
        c = sel | np.where(sel == 3, rng.integers(0, 5, n) << 3, 0) | np.where(sel == 5, rng.integers(0, 5, n) << 6, 0)
    return np.where(rng.random(n) < share, c, 0).astype(np.uint16)


@pytest.mark.parametrize("limo", [0, 1], ids=["mp5", "limo3"])
@pytest.mark.parametrize("spread", [0, 12, 40, 300], ids=lambda b: "spread%d" % b)
@pytest.mark.parametrize("ends", ["inside", "low", "high", "both"])
def test_transposed_sweep_is_correctly_rounded(lib, ends, spread, limo):
    rng = np.random.default_rng(1407 + spread)
    for slen in (1, 3, 4, 16, 17):
        for share in (0.0, 0.3, 1.0):
            n = slen + 20
            low, high = ends in ("low", "both"), ends in ("high", "both")
            if ends == "both":
                n = slen
            fofs = 0 if low else (n - slen if high else 1)  # "inside" wraps round a periodic line
            kb, ke = (0 if low else -2), (slen if high else slen + 2)
            lo, hi = (-3 if low else 0), (slen + 2 if high else slen - 1)
            g = rng.uniform(-1, 1, slen + 6) * 2.0 ** rng.uniform(-spread, 0, slen + 6)
            if low:
                g[:3] = 0.0
            if high:
                g[slen + 3:] = 0.0
            tp, tm = _codes(limo, rng, n + 1, share), _codes(limo, rng, n + 1, share)
            gp, gm = np.full(slen + 10, np.nan), np.full(slen + 10, np.nan)
            wrap = not low and not high
            lib.adjoint(limo, g.ctypes.data, slen, tp.ctypes.data, tm.ctypes.data, fofs, n, wrap, kb, ke, lo, hi,
                        gp.ctypes.data, gm.ctypes.data)
            G = [Fraction(float(x)) for x in g]
            wantp, wantm = {}, {}
            for k in range(kb, ke + 1):
                d = G[k + 3] - G[k + 2]
                f = (k + fofs) % n if wrap else k + fofs
                wp, wm = _weights(limo, int(tp[f])), _weights(limo, int(tm[f]))[::-1]
                for q, w in enumerate(wp):
                    c = k - (2 if limo else 3) + q
                    wantp[c] = wantp.get(c, 0) + w * d
                for q, w in enumerate(wm):
                    c = k - (1 if limo else 2) + q
                    wantm[c] = wantm.get(c, 0) + w * d
            for c in range(lo, hi + 1):
                win = [abs(x) for x in g[max(c, 0):c + 7] if x]
                top = max(math.frexp(x)[1] for x in win) if win else 0
                span = top - (min(math.frexp(x)[1] for x in win) - 53) if win else 0
                for got, want in ((gp[c + 5], wantp.get(c, Fraction(0))), (gm[c + 5], wantm.get(c, Fraction(0)))):
                    if span <= 106:
                        assert got == float(want), (slen, share, c)
                    else:
                        tol = Fraction(2) ** (top - 92) + abs(want) * Fraction(2) ** -53
                        assert abs(Fraction(float(got)) - want) <= tol, (slen, share, c)
