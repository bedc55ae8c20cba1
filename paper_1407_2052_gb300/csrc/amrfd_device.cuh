// amrfd_device.cuh -- device-side building blocks of the FD-MP5 update.
//
// FP64 issue rate on GB300 is 1/64 of FP32, so everything that can be done exactly
// without the FP64 pipe is: the reconstruction sweeps run in exact fixed point
// (amrfd_sweep.cuh), comparisons and sign logic on the integer pipe over the IEEE bit
// patterns, and the FP64 operations that remain are issued in the pipe's fastest form,
// DFMAs whose operands are all registers (see "FP64 operations as register FMAs").
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "amrfd_internal.h"

namespace amrfd {

enum { PH_EULER = 0, PH_MHD = 1 };

// Descriptor checks of the checked builds: a flux item lies inside its domain and its
// tile fits the shared memory (P lines of SS doubles); a cell item lies
// inside its block.
__device__ __forceinline__ bool flux_item_ok(const DomDev* doms, int ndom, int ndim, int P, int SS,
                                             const FluxItem& it) {
  if (it.dom < 0 || it.dom >= ndom) return false;
  const DomDev& dm = doms[it.dom];
  const int d = it.d;
  if (d >= ndim || it.blk < 0 || it.blk >= dm.nb[0] * dm.nb[1] * dm.nb[2]) return false;
  const int od1 = d == 0 ? 1 : 0, od2 = d == 2 ? 1 : 2;
  const int bd = (d == 0 ? it.blk % dm.nb[0] : (d == 1 ? (it.blk / dm.nb[0]) % dm.nb[1] : it.blk / (dm.nb[0] * dm.nb[1])));
  return it.nl >= 1 && it.nl * tile_stride(it.slen) <= P * SS && it.l0 >= 0 &&
         it.l0 + it.nl <= dm.be[od1] * dm.be[od2] && it.s0 >= 0 && it.slen >= 1 &&
         bd * dm.be[d] + it.s0 + it.slen <= dm.n[d];
}

__device__ __forceinline__ bool cell_item_ok(const DomDev* doms, int ndom, const CellItem& ci) {
  if (ci.dom < 0 || ci.dom >= ndom) return false;
  const DomDev& dm = doms[ci.dom];
  return ci.blk >= 0 && ci.blk < dm.nb[0] * dm.nb[1] * dm.nb[2] && ci.c0 >= 0 && ci.cnt >= 0 &&
         ci.c0 + ci.cnt <= dm.be[0] * dm.be[1] * dm.be[2];
}

// ---------------------------------------------------------------- exact helpers
// Bit pattern of x through an opaque PTX move, so that integer tests on it stay on the
// integer pipe (from a plain reinterpretation the compiler rebuilds FP64 compares,
// absolute values and negations).
__device__ __forceinline__ long long dbits(double x) {
  long long r;
  asm("mov.b64 %0, %1;" : "=l"(r) : "d"(x));
  return r;
}
__device__ __forceinline__ double bitsd(long long b) { return __longlong_as_double(b); }

// The helpers below are written in inline PTX so that they stay on the integer
// pipe: left to itself the compiler turns some of these bit manipulations of
// doubles back into FP64 compares, negations or multiplies.

// Monotone signed-integer key of a double (total order; -0 sorts before +0).
// Bit pattern of |x| (in PTX: masking the sign of a double's bits in C++ is turned by
// the compiler into an FP64 add with an absolute-value operand).
__device__ __forceinline__ long long abits(double x) {
  long long r;
  asm("{\n\t.reg .b64 t;\n\tmov.b64 t, %1;\n\tand.b64 %0, t, 0x7fffffffffffffff;\n\t}" : "=l"(r) : "d"(x));
  return r;
}

__device__ __forceinline__ long long okey(double x) {
  long long b = dbits(x);
  return b ^ ((b >> 63) & 0x7fffffffffffffffLL);
}

#define AMRFD_OKEY(dst, src) \
  "shr.s64 " dst ", " src ", 63;\n\t" "and.b64 " dst ", " dst ", 0x7fffffffffffffff;\n\t" \
  "xor.b64 " dst ", " src ", " dst ";\n\t"

__device__ __forceinline__ double imin(double a, double b) {
  double r;
  asm("{\n\t.reg .b64 xa, xb, ka, kb;\n\t.reg .pred p;\n\t"
      "mov.b64 xa, %1;\n\tmov.b64 xb, %2;\n\t" AMRFD_OKEY("ka", "xa") AMRFD_OKEY("kb", "xb")
      "setp.lt.s64 p, ka, kb;\n\tselp.b64 xa, xa, xb, p;\n\tmov.b64 %0, xa;\n\t}"
      : "=d"(r) : "d"(a), "d"(b));
  return r;
}
__device__ __forceinline__ double imax(double a, double b) {
  double r;
  asm("{\n\t.reg .b64 xa, xb, ka, kb;\n\t.reg .pred p;\n\t"
      "mov.b64 xa, %1;\n\tmov.b64 xb, %2;\n\t" AMRFD_OKEY("ka", "xa") AMRFD_OKEY("kb", "xb")
      "setp.lt.s64 p, ka, kb;\n\tselp.b64 xa, xb, xa, p;\n\tmov.b64 %0, xa;\n\t}"
      : "=d"(r) : "d"(a), "d"(b));
  return r;
}

// -x by flipping the sign bit (in PTX: the compiler would otherwise emit an FP64 add)
__device__ __forceinline__ double dneg(double x) {
  double r;
  asm("{\n\t.reg .b64 t;\n\tmov.b64 t, %1;\n\txor.b64 t, t, 0x8000000000000000;\n\tmov.b64 %0, t;\n\t}"
      : "=d"(r) : "d"(x));
  return r;
}

// |x| rounded toward zero to FP32, from the bits of |x| whose exponent lies in
// [2^-60, 2^61) (caller checks): the mantissa's top 23 bits and a rebiased exponent.
__device__ __forceinline__ float f32_trunc_abs(long long ax) {
  float r;
  asm("{\n\t.reg .b64 t;\n\t.reg .b32 u;\n\t"
      "shr.u64 t, %1, 29;\n\tsub.u64 t, t, 7516192768;\n\tcvt.u32.u64 u, t;\n\tmov.b32 %0, u;\n\t}"
      : "=f"(r) : "l"(ax));
  return r;
}

// ------------------------------------------------ FP64 operations as register FMAs
// GB300 issues a DFMA whose three operands are registers at 19.6 G warp instructions/s,
// and a DADD, a DMUL or a DFMA with an immediate or constant-bank operand at 16.5 G/s
// (independent chains on every SM, whatever the operand values). The hot loops therefore
// form sums, differences and products as register DFMAs, bit for bit the plain
// operations: x + y = fma(x, 1, y) and x - y = fma(x, 1, -y) (the exact sum, rounded
// once), c x = fma(c, x, -0) (adding -0 changes no product, zeros included). The
// constants are read from a mutable device array through an opaque load, so the
// compiler can neither fold them back into immediates nor read them from the constant
// bank.
enum { K_ONE, K_MZ, K_HALF, K_ZERO, K_COUNT };
static __device__ double g_regk[K_COUNT] = {1.0, -0.0, 0.5, 0.0};

// Constant K_* as a register value (an opaque load at this point of the code).
__device__ __forceinline__ double ldk(int i) {
  double x;
  asm volatile("ld.f64 %0, [%1];" : "=d"(x) : "l"(g_regk + i));
  return x;
}

__device__ __forceinline__ double radd(double x, double y, double one) { return fma(x, one, y); }
__device__ __forceinline__ double rsub(double x, double y, double one) { return fma(x, one, -y); }
__device__ __forceinline__ double rmul(double c, double x, double mz) { return fma(c, x, mz); }

// Reciprocal of a positive normal double: FP32 seed from the leading bits (integer
// conversion, MUFU reciprocal) and two Newton steps y <- y + y (1 - x y) in FP64.
__device__ __forceinline__ double frcp(double x) {
  const long long b = dbits(x);
  const int e = (int)((b >> 52) & 0x7ff);
  if (e < 1023 - 120 || e > 1023 + 120) return 1.0 / x;
  const unsigned fb = ((unsigned)((unsigned long long)b >> 32) & 0x80000000u) | ((unsigned)(e - 1023 + 127) << 23) |
                      (unsigned)((b >> 29) & 0x7fffff);
  const unsigned yb = __float_as_uint(__frcp_rn(__uint_as_float(fb)));
  const long long db = ((long long)(yb & 0x80000000u) << 32) | ((long long)(((yb >> 23) & 0xff) - 127 + 1023) << 52) |
                       ((long long)(yb & 0x7fffff) << 29);
  double y = bitsd(db);
  const double one = ldk(K_ONE);
  double r = fma(-x, y, one);
  y = fma(y, r, y);
  r = fma(-x, y, one);
  return fma(y, r, y);
}

// ------------------------------------------------- exact characteristic speeds
// Same operation order as the CPU definition (no contraction), so that splitting
// speeds and time steps of a given state agree bit for bit.
struct Prim {
  double rho, v[3], p, B[3], psi;
};

template <int PHYS, int NV>
__device__ __forceinline__ bool cons2prim_exact(const double* u, double gamma, int ndim, Prim& w) {
  w.rho = u[0];
  const int nm = PHYS == PH_EULER ? NV - 2 : 3;
#pragma unroll
  for (int k = 0; k < 3; k++) w.v[k] = (k < nm) ? __ddiv_rn(u[1 + k], w.rho) : 0.0;
  double vv = __dadd_rn(__dadd_rn(__dmul_rn(w.v[0], w.v[0]), __dmul_rn(w.v[1], w.v[1])), __dmul_rn(w.v[2], w.v[2]));
  double ekin = __dmul_rn(__dmul_rn(0.5, w.rho), vv);
  double emag = 0.0, E;
  if (PHYS == PH_MHD) {
    w.B[0] = u[5]; w.B[1] = u[6]; w.B[2] = u[7]; w.psi = u[8];
    emag = __dmul_rn(0.5, __dadd_rn(__dadd_rn(__dmul_rn(w.B[0], w.B[0]), __dmul_rn(w.B[1], w.B[1])),
                                    __dmul_rn(w.B[2], w.B[2])));
    E = u[4];
  } else {
    w.B[0] = w.B[1] = w.B[2] = 0.0; w.psi = 0.0;
    E = u[NV - 1];
  }
  w.p = __dmul_rn(__dsub_rn(gamma, 1.0), __dsub_rn(__dsub_rn(E, ekin), emag));
  return (w.rho > 0.0) && (w.p > 0.0) && isfinite(w.rho) && isfinite(w.p) && isfinite(w.psi);
}

template <int PHYS>
__device__ __forceinline__ double char_speed_exact(const Prim& w, double gamma, int d) {
  if (PHYS == PH_EULER) return __dadd_rn(fabs(w.v[d]), __dsqrt_rn(__ddiv_rn(__dmul_rn(gamma, w.p), w.rho)));
  double a2 = __ddiv_rn(__dmul_rn(gamma, w.p), w.rho);
  double b2 = __ddiv_rn(__dadd_rn(__dadd_rn(__dmul_rn(w.B[0], w.B[0]), __dmul_rn(w.B[1], w.B[1])),
                                  __dmul_rn(w.B[2], w.B[2])), w.rho);
  double s = __dadd_rn(a2, b2);
  double bd = w.B[d];
  double disc = __dsub_rn(__dmul_rn(s, s), __ddiv_rn(__dmul_rn(__dmul_rn(4.0, a2), __dmul_rn(bd, bd)), w.rho));
  if (disc < 0.0) disc = 0.0;
  double cf = __dsqrt_rn(__dmul_rn(0.5, __dadd_rn(s, __dsqrt_rn(disc))));
  return __dadd_rn(fabs(w.v[d]), cf);
}

// --------------------------------------- bounded FP32 estimate of the speeds
// FP32 conversion of x (truncation, relative error < 2^-23) when |x| lies in
// [2^-100, 2^100] or x is zero; ok = false otherwise.
__device__ __forceinline__ float f32_of(double x, bool& ok) {
  const long long ax = abits(x);
  if (ax == 0) return 0.0f;
  const int e = (int)(ax >> 52);
  if (e < 923 || e > 1123) { ok = false; return 0.0f; }
  const float f = f32_trunc_abs(ax);
  return ax != dbits(x) ? -f : f;
}

// As f32_of for a momentum or field component, except that a nonzero |x| < 2^-100
// gives 0 and sets flushed (the caller bounds the effect of the change).
__device__ __forceinline__ float f32_of_flush(double x, bool& ok, bool& flushed) {
  const long long ax = abits(x);
  if (ax == 0) return 0.0f;
  const int e = (int)(ax >> 52);
  if (e < 923) { flushed = true; return 0.0f; }
  if (e > 1123) { ok = false; return 0.0f; }
  const float f = f32_trunc_abs(ax);
  return ax != dbits(x) ? -f : f;
}

// Bounds lo <= c_d <= up of the exact characteristic speeds of a cell (d < ndim), and
// of its CFL rate sum_d c_d/dx_d (index 3), from an FP32 evaluation. The relative
// error of every FP32 quantity is bounded by the input truncation (2^-23 each), the
// FP32 roundings (2^-24 each) and the cancellation in p = (gamma-1)(E - rho v^2/2 -
// B^2/2), which scales them by T/S with T = E + rho v^2/2 + B^2/2, S = p/(gamma-1);
// the discriminant of the fast speed is formed as (a^2 - b_d^2)^2 + b_t^2 (b_t^2 +
// 2 (a^2 + b_d^2)) (b_t the transverse Alfven speed), a sum of non-negative terms,
// so the square roots do not amplify it. The bound used, 2^-17 (T/S + 1), holds with
// a margin of four. Momentum and field components below 2^-100 in magnitude (the
// exactly-zero components of a uniform state pick up such values ahead of a wave)
// enter as 0. Each such change moves c_d = |v_d| + c_f by at most 2^-100 (1.5 +
// gamma) (1/rho + 1/sqrt(rho)): c_f is 1-Lipschitz in the sound speed a and in
// b_d = |B_d|/sqrt(rho), 1.5-Lipschitz in the transverse b_t, and a moves by at most
// the square root of the change of a^2. With at most six such components, with
// T/S < 2^10 (FP32 a^2 then within 2^-10 of its value) and with
// (1.5 + gamma)(1/rho + 1/sqrt(rho))/a <= 2^76, the total is below 2^-21 c_d, and
// the bounds widen by 2^-20 relative; otherwise the cell is evaluated exactly.
// force = true when no bound is claimed (non-physical or out of FP32 range): the
// caller then evaluates the cell exactly.
template <int PHYS, int NV>
__device__ __forceinline__ void speed_bounds(const double* u, float gam, int ndim, const float* rdx, bool want_rate,
                                             float up[4], float lo[4], bool& force) {
  bool ok = true, fl = false;
  const float rho = f32_of(u[0], ok);
  constexpr int nm = PHYS == PH_EULER ? NV - 2 : 3;
  float m[3] = {0.f, 0.f, 0.f}, B[3] = {0.f, 0.f, 0.f};
#pragma unroll
  for (int k = 0; k < nm; k++) m[k] = f32_of_flush(u[1 + k], ok, fl);
  const float E = f32_of(u[PHYS == PH_EULER ? NV - 1 : 4], ok);
  if (PHYS == PH_MHD) {
#pragma unroll
    for (int k = 0; k < 3; k++) B[k] = f32_of_flush(u[5 + k], ok, fl);
  }
  if (PHYS == PH_MHD && ((dbits(u[8]) >> 52) & 0x7ff) == 0x7ff) ok = false;  // psi not finite
  force = !ok || !(rho > 0.0f) || !(E > 0.0f);
  if (force) return;
  const float ir = __frcp_rn(rho);
  const float v[3] = {m[0] * ir, m[1] * ir, m[2] * ir};
  const float ke2 = fmaf(m[2], v[2], fmaf(m[1], v[1], m[0] * v[0]));
  const float sq[3] = {B[0] * B[0], B[1] * B[1], B[2] * B[2]};
  const float b2 = sq[0] + sq[1] + sq[2];
  const float half = 0.5f * (ke2 + b2);
  const float T = E + half, S = E - half;
  if (!(S > 1.9073486e-6f * T)) { force = true; return; }  // S <= 2^-19 T: too uncertain
  float rel = 7.6293945e-6f * fmaf(T, __frcp_rn(S), 1.0f);  // 2^-17 (T/S + 1)
  const float a2 = gam * (gam - 1.0f) * S * ir;             // gamma p / rho
  if (fl) {
    const float q = (1.5f + gam) * (ir + sqrtf(ir)) / sqrtf(a2);
    if (!(S > 9.765625e-4f * T) || !(q <= 7.5557864e22f)) { force = true; return; }  // 2^-10, 2^76
    rel += 9.5367431640625e-07f;                                                   // 2^-20
  }
  float rate_up = 0.0f, rate_lo = 0.0f;
#pragma unroll
  for (int d = 0; d < 3; d++) {
    if (d >= ndim) { up[d] = 0.0f; lo[d] = 0.0f; continue; }
    float cf;
    if (PHYS == PH_EULER) {
      cf = sqrtf(a2);
    } else {
      const float bd2 = sq[d] * ir;
      const float bt2 = (sq[(d + 1) % 3] + sq[(d + 2) % 3]) * ir;
      const float x = a2 - bd2;
      const float disc = fmaf(x, x, bt2 * (bt2 + 2.0f * (a2 + bd2)));
      cf = sqrtf(0.5f * (a2 + bd2 + bt2 + sqrtf(disc)));
    }
    const float c = fabsf(v[d]) + cf;
    up[d] = c * (1.0f + rel);
    lo[d] = c * (1.0f - rel);
    if (want_rate) {
      rate_up = fmaf(up[d], rdx[d], rate_up);
      rate_lo = fmaf(lo[d], rdx[d], rate_lo);
    }
  }
  up[3] = rate_up * 1.0000153f;  // (1 + 2^-16): rounding of the rate sums and 1/dx
  lo[3] = rate_lo * 0.9999847f;
}

// ------------------------------------------------------ fast flux + LF split
// G^{+-} = F_d +- alpha_d U = 2 F^{+-}: the factor 1/2 of the splitting is
// applied once to the final flux difference (MP5 commutes with scaling by 2
// when its acceptance threshold is scaled by 4).
// Number of per-cell derived quantities the flux needs besides U: MHD v_x, v_y, v_z,
// p_tot = p + B^2/2, v.B; Euler v_1..v_ndim, p.
template <int PHYS, int NV>
struct NumW { static constexpr int value = PHYS == PH_EULER ? NV - 1 : 5; };

// The derived quantities of one cell (the FP64 part of cons -> prim the flux needs).
template <int PHYS, int NV>
__device__ __forceinline__ void prim_w(const double* u, double gm1, double* w) {
  const double ir = frcp(u[0]);
  const double one = ldk(K_ONE), mz = ldk(K_MZ), half = ldk(K_HALF);
  if (PHYS == PH_EULER) {
    constexpr int nm = NV - 2;
    double mv = ldk(K_ZERO);
#pragma unroll
    for (int k = 0; k < nm; k++) { w[k] = rmul(u[1 + k], ir, mz); mv = fma(u[1 + k], w[k], mv); }
    w[nm] = gm1 * fma(-half, mv, u[NV - 1]);
  } else {
    const double v[3] = {rmul(u[1], ir, mz), rmul(u[2], ir, mz), rmul(u[3], ir, mz)};
    const double b2 = fma(u[7], u[7], fma(u[6], u[6], rmul(u[5], u[5], mz)));
    const double mv = fma(u[3], v[2], fma(u[2], v[1], rmul(u[1], v[0], mz)));
    const double p = gm1 * fma(-half, radd(mv, b2, one), u[4]);
    w[0] = v[0]; w[1] = v[1]; w[2] = v[2];
    w[3] = fma(half, b2, p);
    w[4] = fma(v[2], u[7], fma(v[1], u[6], rmul(v[0], u[5], mz)));
  }
}

// Physical flux along D from U and its derived quantities, then the Lax-Friedrichs
// split in doubled form G^{+-} = F +- alpha U (= 2 F^{+-}); psi's flux is c_h^2 B_D.
// one, mz: 1 and -0 in registers.
template <int PHYS, int NV, int D>
__device__ __forceinline__ void split_flux_w(const double* u, const double* w, double alpha, double ch2,
                                             double one, double mz, double* gp, double* gm) {
  double f[NV];
  if (PHYS == PH_EULER) {
    constexpr int nm = NV - 2;
    const double p = w[nm], vd = w[D];
    f[0] = u[1 + D];
#pragma unroll
    for (int k = 0; k < nm; k++) f[1 + k] = (k == D) ? fma(vd, u[1 + k], p) : rmul(vd, u[1 + k], mz);
    f[NV - 1] = rmul(vd, radd(u[NV - 1], p, one), mz);
  } else {
    const double ptot = w[3], vb = w[4];
    const double vd = w[D], bd = u[5 + D];
    f[0] = u[1 + D];
#pragma unroll
    for (int k = 0; k < 3; k++) {
      f[1 + k] = fma(vd, u[1 + k], rmul(-bd, u[5 + k], mz));
      if (k == D) f[1 + k] = radd(f[1 + k], ptot, one);
      f[5 + k] = (k == D) ? u[8] : fma(vd, u[5 + k], rmul(-bd, w[k], mz));
    }
    f[4] = fma(vd, radd(u[4], ptot, one), rmul(-bd, vb, mz));
    f[8] = rmul(ch2, bd, mz);
  }
#pragma unroll
  for (int v = 0; v < NV; v++) {
    gp[v] = fma(alpha, u[v], f[v]);
    gm[v] = fma(-alpha, u[v], f[v]);
  }
}

// ------------------------------------------------------------- block reductions
__device__ __forceinline__ unsigned long long warp_max_u64(unsigned long long x) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    unsigned long long y = __shfl_xor_sync(0xffffffffu, x, o);
    x = y > x ? y : x;
  }
  return x;
}

}  // namespace amrfd
