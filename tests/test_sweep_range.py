"""The fixed-point sweeps (csrc/amrfd_sweep.cuh) at the ends of their range, on the CPU: wide
sums, windows of far more than 110 bits, cells that are exactly equal."""
import ctypes
import os
import shutil
import subprocess
from fractions import Fraction

import numpy as np
import pytest

from test_sweep_host import _reference

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1407_2052_gb300", "csrc")

HARNESS = """
#include "amrfd_sweep.cuh"
using namespace amrfd;
extern "C" double wide(long long hi, unsigned long long lo) {
  return wide_double((__int128)(((unsigned __int128)(unsigned long long)hi << 64) | lo));
}
extern "C" void sweep(int limo, const double* gp, const double* gm, int plen, double thr, double* out,
                      unsigned short* tp, unsigned short* tm) {
  if (limo) fixed_sweep<true, true>(gp, gm, plen, thr, out, 1, ~0ull, tp, tm, 0, plen + 1, 1 << 30, 1);
  else fixed_sweep<false, true>(gp, gm, plen, 0.0, out, 1, ~0ull, tp, tm, 0, plen + 1, 1 << 30, 1);
}
extern "C" void adjoint(int limo, const double* g, int slen, const unsigned short* codes, double* gp, double* gm) {
  const TapeLine t = {codes, codes, 1, slen + 20, true};
  if (limo) adjoint_sweep<true>(g, slen, t, -2, slen + 2, 0, slen - 1, gp, gm, 1);
  else adjoint_sweep<false>(g, slen, t, -2, slen + 2, 0, slen - 1, gp, gm, 1);
}
// The cells a three-limb sweep leaves to the exact arithmetic.
extern "C" int left(int limo, const double* gp, const double* gm, int plen, double thr) {
  double out[64];
  int lob, limited = 0;
  bool bad;
  if (!window_scale<3, false>(gp, gm, 0, plen + 6, lob, bad)) return -1;
  const unsigned long long todo =
      limo ? sweep_part<true, false, 3>(gp, gm, plen, thr, out, 1, ~0ull, 0, 0, 0, 0, 0, lob, limited)
           : sweep_part<false, false, 3>(gp, gm, plen, 0.0, out, 1, ~0ull, 0, 0, 0, 0, 0, lob, limited);
  return __builtin_popcountll(todo & ((1ull << plen) - 1ull));
}
extern "C" double weight(double dtb, double dx) { return stage_weight(dtb, dx); }
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no g++")
    d = tmp_path_factory.mktemp("range")
    src, so = d / "h.cpp", d / "h.so"
    src.write_text(HARNESS)
    subprocess.run([gxx, "-O1", "-std=gnu++17", "-ffp-contract=off", "-w", "-shared", "-fPIC", "-I", CSRC, str(src),
                    "-o", str(so)], check=True)
    L = ctypes.CDLL(str(so))
    L.wide.restype, L.wide.argtypes = ctypes.c_double, [ctypes.c_longlong, ctypes.c_ulonglong]
    L.left.argtypes = [ctypes.c_int] + [ctypes.c_void_p] * 2 + [ctypes.c_int, ctypes.c_double]
    L.weight.restype, L.weight.argtypes = ctypes.c_double, [ctypes.c_double] * 2
    L.sweep.argtypes = [ctypes.c_int] + [ctypes.c_void_p] * 2 + [ctypes.c_int, ctypes.c_double] + [ctypes.c_void_p] * 3
    L.adjoint.argtypes = [ctypes.c_int, ctypes.c_void_p, ctypes.c_int] + [ctypes.c_void_p] * 3
    return L


def _sweep(lib, limo, g, h, thr=0.0):
    n = len(g) - 6
    out, tp, tm = np.full(n, np.nan), np.zeros(n + 1, np.uint16), np.zeros(n + 1, np.uint16)
    lib.sweep(limo, g.ctypes.data, h.ctypes.data, n, thr, out.ctypes.data, tp.ctypes.data, tm.ctypes.data)
    return out, tp, tm


@pytest.mark.parametrize("bits", [53, 54, 95, 96, 97, 120, 121, 122, 123, 124, 125])
def test_wide_sums_round_once(lib, bits):
    """Whole numbers of `bits` bits, near ties of the conversion among them."""
    rng = np.random.default_rng(bits)
    for _ in range(2000):
        a = (1 << (bits - 1)) | int(rng.integers(0, 1 << 52)) << max(0, bits - 53)
        a += (1 << max(0, bits - 54)) + int(rng.integers(-2, 3))  # half a unit in the last place, about
        a = min(a, (1 << bits) - 1) * int(rng.choice((-1, 1)))
        assert lib.wide(a >> 64, a & (2 ** 64 - 1)) == float(Fraction(a)), a


@pytest.mark.parametrize("limo", [0, 1], ids=["mp5", "limo3"])
@pytest.mark.parametrize("weak", [1e-20, 1e-34, 1e-60, 1e-200, 1e-300])
def test_weak_cells_beside_strong_ones_keep_their_precision(lib, weak, limo):
    """Where the limiter drops the strong cells of a window, the difference is one of the weak
    cells alone, and off by no more than FP64 sums of them are: fewer than 40 roundings of
    terms below 2000 weak cells."""
    rng, dropped = np.random.default_rng(7), 0
    for _ in range(60):
        n = 24
        s = rng.integers(3, 12)
        g = np.where(np.arange(n) < s, 1 + 0.1 * rng.random(n), weak * rng.uniform(0.5, 2.0, n))
        h = np.where(np.arange(n) >= n - s, 1 + 0.1 * rng.random(n), weak * rng.uniform(-1, 1, n))
        out, _, _ = _sweep(lib, limo, g, h, 1e-30)
        for i, want in enumerate(_reference(limo, g, h, 1e-30)):
            strong = any(abs(x) > 0.5 for x in (*g[i:i + 7], *h[i:i + 7]))
            if abs(want) < 2000 * 2 * weak:
                dropped += strong
                err = abs(Fraction(float(out[i])) - want)
                assert err <= Fraction(40 * 2000 * 2 * weak) * Fraction(2) ** -53 + Fraction(2) ** -1060, i
    assert dropped > 50


@pytest.mark.parametrize("limo", [0, 1], ids=["mp5", "limo3"])
def test_finite_values_of_any_size_give_the_rounded_difference(lib, limo):
    rng = np.random.default_rng(8)
    for top in (1005, 1012, 1018, 1023):
        g, h = (np.ldexp(rng.uniform(-1, 1, 30), top) for _ in range(2))
        out, _, _ = _sweep(lib, limo, g, h, 1e-30)
        for i, want in enumerate(_reference(limo, g, h, 1e-30)):
            try:
                w = float(want)
            except OverflowError:
                w = np.inf if want > 0 else -np.inf
            assert out[i] == w, (top, i)


@pytest.mark.parametrize("limo", [0, 1], ids=["mp5", "limo3"])
@pytest.mark.parametrize("binades", [12, 13, 14, 34, 35, 36, 56, 57])
def test_every_width_of_the_sums_rounds_correctly(lib, binades, limo):
    """One limb more or less: the cells' exponents span exactly `binades`, full mantissas."""
    rng = np.random.default_rng(binades)
    for _ in range(20):
        e = rng.integers(-binades, 1, (2, 38))
        e[0, 5], e[1, 6] = 0, -binades
        g, h = (np.ldexp(rng.uniform(1, 2, 38) * rng.choice((-1, 1), 38), x) for x in e)
        out, _, _ = _sweep(lib, limo, g, h, 0.1)
        assert out.tolist() == [float(x) for x in _reference(limo, g, h, 0.1)]


@pytest.mark.parametrize("limo", [0, 1], ids=["mp5", "limo3"])
@pytest.mark.parametrize("weak", [1e-20, 1e-40, 1e-290])
def test_weak_gradients_beside_strong_ones_keep_their_precision(lib, weak, limo):
    """With every face on the piece "zero" a cell's gradient is 60 times one difference of the
    upstream gradient: of two weak ones wherever it is, whatever else lies within reach."""
    rng, n = np.random.default_rng(11), 16
    codes = np.full(n + 21, 8 if limo else 1, np.uint16)
    for _ in range(20):
        g = np.where(rng.random(n + 6) < 0.3, 1.0, weak) * rng.uniform(0.5, 2.0, n + 6)
        gp, gm = np.zeros(n + 10), np.zeros(n + 10)
        lib.adjoint(limo, g.ctypes.data, n, codes.ctypes.data, gp.ctypes.data, gm.ctypes.data)
        G = [Fraction(float(x)) for x in g]
        for c in range(n):  # G+ of cell c is the centre of face c + 1, G- of face c
            for got, want in ((gp[c + 5], 60 * (G[c + 4] - G[c + 3])), (gm[c + 5], 60 * (G[c + 3] - G[c + 2]))):
                assert abs(Fraction(float(got)) - want) <= abs(want) * Fraction(2) ** -51, c


def test_stage_weight_rounds_once_on_power_of_two_grids(lib):
    rng = np.random.default_rng(5)
    for _ in range(3000):
        dtb, k = float(rng.uniform(1e-6, 1.0)), int(rng.integers(0, 14))
        assert lib.weight(dtb, 2.0 ** -k) == float(Fraction(dtb) * 2 ** k / 120)


@pytest.mark.parametrize("limo", [0, 1], ids=["mp5", "limo3"])
@pytest.mark.parametrize("size", [1.0, 1e20, 1e25, 1e30, 1e100, 1e290])
def test_uniform_lines_in_any_units_leave_no_cell(lib, size, limo):
    g, h = np.full(38, size), np.full(38, -0.3 * size)
    assert lib.left(limo, g.ctypes.data, h.ctypes.data, 32, 1e-4) == 0
    g[:10] *= 1.5  # and the cells whose stencils are uniform, beside a jump
    assert lib.left(limo, g.ctypes.data, h.ctypes.data, 32, 1e-4) <= 10


@pytest.mark.parametrize("step", [1, 2, 3, 5, 9])
def test_steps_between_flat_states_leave_no_cell_with_limo3(lib, step):
    """A difference of exactly zero beside another one gives a face value of zero by several of
    LIMO3's pieces; FP32 and the exact selection give it the same name."""
    rng, thr = np.random.default_rng(step), 1e-14
    for _ in range(20):
        g, h = (np.repeat(rng.uniform(0.5, 1.5, 60 // step + 1), step)[:60] for _ in range(2))
        left = lib.left(1, g.ctypes.data, h.ctypes.data, 54, thr)
        assert left == 0 if step > 1 else left <= 2
        out, tp, tm = _sweep(lib, 1, g, h, thr)
        assert out.tolist() == [float(x) for x in _reference(1, g, h, thr)]
        for k in range(3, 58):
            a, b = g[k - 1] - g[k - 2], g[k] - g[k - 1]
            assert a * b != 0 or tp[k - 3] == (0 if a == b else 8)
