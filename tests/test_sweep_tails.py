"""Tails ahead of a front, which fall off by binades per cell, in the fixed-point sweeps
(csrc/amrfd_sweep.cuh) on the CPU: their parts are swept as a fixed filter, in halves or
quarters where they span more than 110 bits."""
import ctypes
import shutil
import subprocess
from fractions import Fraction

import numpy as np
import pytest

from test_sweep_host import _reference
from test_sweep_range import CSRC

HARNESS = """
#include "amrfd_sweep.cuh"
using namespace amrfd;
template <bool L> int wide(const double* gp, const double* gm, int plen, double thr, double* out, unsigned short* tp,
                           unsigned short* tm) {
  const Wide5 w = wide_sweep<L, true>(gp, gm, plen, thr, out, 1, ~0ull, tp, tm, 0, plen + 1, 1 << 30,
                                      window_span<false>(gp, gm, L ? 1 : 0, plen + (L ? 4 : 6)), 1);
  return __builtin_popcountll(w.todo & (plen < 64 ? (1ull << plen) - 1ull : ~0ull));
}
extern "C" int left(int limo, const double* gp, const double* gm, int plen, double thr, double* out,
                    unsigned short* tp, unsigned short* tm) {
  return limo ? wide<true>(gp, gm, plen, thr, out, tp, tm) : wide<false>(gp, gm, plen, thr, out, tp, tm);
}
extern "C" int sweep(int limo, const double* gp, const double* gm, int plen, double thr, double* out,
                     unsigned short* tp, unsigned short* tm) {
  return limo ? fixed_sweep<true, true>(gp, gm, plen, thr, out, 1, ~0ull, tp, tm, 0, plen + 1, 1 << 30, 1)
              : fixed_sweep<false, true>(gp, gm, plen, thr, out, 1, ~0ull, tp, tm, 0, plen + 1, 1 << 30, 1);
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no g++")
    d = tmp_path_factory.mktemp("tails")
    src, so = d / "h.cpp", d / "h.so"
    src.write_text(HARNESS)
    subprocess.run([gxx, "-O1", "-std=gnu++17", "-ffp-contract=off", "-w", "-shared", "-fPIC", "-I", CSRC, str(src),
                    "-o", str(so)], check=True)
    L = ctypes.CDLL(str(so))
    for f in (L.left, L.sweep):
        f.argtypes = ([ctypes.c_int] + [ctypes.c_void_p] * 2 + [ctypes.c_int, ctypes.c_double] +
                      [ctypes.c_void_p] * 3)
    return L


def _tail(rng, n, binades, top, end=-900):
    """Full mantissas of any sign, falling off by `binades` a cell from 2^top, to the left or
    to the right, down to 2^end (near underflow the sweeps keep FP64's own precision: see
    test_weak_cells_beside_strong_ones_keep_their_precision)."""
    e = top - np.floor(binades * np.arange(n)).astype(int)
    g, h = (np.where(e < end, 0.0, np.ldexp(rng.uniform(1, 2, n) * rng.choice((-1, 1), n), e)) for _ in range(2))
    return (g[::-1].copy(), h[::-1].copy()) if rng.random() < 0.5 else (g, h)


def _call(f, limo, g, h, thr):
    n = len(g) - 6
    out, tp, tm = np.full(n, np.nan), np.full(n + 1, 77, np.uint16), np.full(n + 1, 77, np.uint16)
    left = f(limo, g.ctypes.data, h.ctypes.data, n, thr, out.ctypes.data, tp.ctypes.data, tm.ctypes.data)
    return left, out, tp, tm


@pytest.mark.parametrize("limo", [0, 1], ids=["mp5", "limo3"])
@pytest.mark.parametrize("binades, cells", [(1, 64), (2, 21), (3, 16), (3, 20), (5, 16), (5, 19), (9, 1), (8, 2)])
def test_tails_are_swept_without_a_cell_by_itself(lib, binades, cells, limo):
    """Windows of 4 cells more than a quarter of a part (6 with MP5) hold up to 57 binades; a
    part below 16 cells is cut in halves only, one below 8 not at all."""
    rng = np.random.default_rng(binades)
    for _ in range(10):
        g, h = _tail(rng, cells + 6, binades, -30)
        left, out, tp, tm = _call(lib.left, limo, g, h, 1.0)
        assert left == 0 and not tp.any() and not tm.any()
        assert out.tolist() == [float(x) for x in _reference(limo, g, h, 1.0)]


@pytest.mark.parametrize("limo", [0, 1], ids=["mp5", "limo3"])
@pytest.mark.parametrize("top", [-18, 2, 40])
@pytest.mark.parametrize("binades", [0.5, 2.5, 4, 8, 20, 90])
def test_tails_round_once_from_any_height(lib, binades, top, limo):
    """From surely unlimited faces (below 2^-17) to limited ones; windows over 110 bits keep
    what FP64 keeps: half a unit of the result and 2^-100 of the window's largest value."""
    rng, thr = np.random.default_rng(top + 100), 1e-3
    for cells in (1, 7, 8, 15, 16, 33, 64):
        g, h = _tail(rng, cells + 6, binades, top)
        g[rng.random(len(g)) < 0.05] = 0.0
        _, out, _, _ = _call(lib.sweep, limo, g, h, thr)
        for i, want in enumerate(_reference(limo, g, h, thr)):
            w = np.abs(np.concatenate((g[i:i + 7], h[i:i + 7])))
            w = w[w > 0]
            if not len(w):
                assert out[i] == 0.0
            elif w.max() / w.min() < 2.0 ** 57:
                assert out[i] == float(want), (cells, i)
            else:
                near = abs(want) * Fraction(2) ** -52 + Fraction(float(w.max())) * Fraction(2) ** -100
                assert abs(Fraction(float(out[i])) - want) <= near, (cells, i)


@pytest.mark.parametrize("limo", [0, 1], ids=["mp5", "limo3"])
@pytest.mark.parametrize("binades, cells", [(1, 64), (2, 21), (3, 16), (5, 19), (8, 2), (12, 16)])
def test_tails_down_to_underflow_are_swept_too(lib, binades, cells, limo):
    """From 2^-960 or less into the subnormals and zero: whole multiples of 2^-1074, hence exact.
    Values below 2^-1042 count as zero."""
    rng = np.random.default_rng(binades)
    for top in (-960, -1000, -1015, -1025, -1035):
        g, h = (np.where(np.abs(x) < 2.0 ** -1042, 0.0, x) for x in _tail(rng, cells + 6, binades, top, -1080))
        left, out, tp, tm = _call(lib.left, limo, g, h, 1.0)
        assert not tp.any() and not tm.any() and (left == 0 or binades > 5 or top > -1015)
        full = _call(lib.sweep, limo, g, h, 1.0)[1]
        for i, want in enumerate(_reference(limo, g, h, 1.0)):
            w = np.abs(np.concatenate((g[i:i + 7], h[i:i + 7])))
            if w.max() < 2.0 ** -967:  # its unit of 2^-110 is the subnormals' or below
                assert full[i] == float(want), (top, i)
