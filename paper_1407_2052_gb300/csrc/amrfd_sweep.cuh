// amrfd_sweep.cuh -- reconstruction sweeps of the flux pass in exact fixed point.
//
// GB300 issues one FP64 warp instruction (an FMA, or a conversion to or from a 64-bit
// type) per 64 cycles and SM sub-partition, an integer one per 1-2 cycles. The sweeps
// therefore hold G^{+-} of the line as fixed-point numbers of three signed 22-bit limbs in
// 32-bit registers: MP5 and LIMO3 are linear in the cells once the limiter's piece is
// known, with whole coefficients after scaling by 60, so a face flux is a short integer dot
// product without rounding, and the flux difference of a cell is exact until its one
// conversion to double. What is decided by comparing (the acceptance test, min, max,
// median, minmod) is decided in FP32 on differences rounded from the exact ones, with a
// rigorous error bound; a comparison that FP32 cannot settle is made in exact 128-bit
// arithmetic.
//
// Measured, the whole flux launch (FP64 sweeps before, these after): 1024^2 MHD vortex 768
// and 352 us, 256^3 MHD blast in noise 16.1 and 10.2 ms (it limits at half its faces; 10.7 in
// later steps, up to 12.7 while tails run through the box, see wide_sweep), 128^3 MHD blast
// with LIMO3 2.12 and 0.97 ms. What bounds them now: integer issue (50 to 60 % of the slots,
// about 490 instructions a face and warp where the limiter runs, 230 where not) and, at 35 %,
// the FP64 pipe (phase A and one conversion a cell).
//
// Scale. A sweep works at one power-of-two scale at which every cell of its part is a whole
// number: of 66 bits (three limbs) where the cells' exponents span at most 13 binades, of 88
// (four limbs, 35 binades) or of 110 bits (five limbs). A sine that crosses zero is past 13
// binades in most warps, hence the four: 75x62x96 MHD waves 2.40 ms a step without them and
// 2.15 with, 42x36x42 0.87 and 0.80. Nothing is rounded then, so the results do not depend on
// the scale, hence not on where a sweep starts. Where a part spans more than 110 bits it is cut
// (wide_sweep), and the cells whose window still holds a value that is no whole number are left
// to exact_cell, which takes each by itself at its own window's scale; where a seven-cell
// window spans more, it carries what the units of 2^-110 of the largest value leave over as
// doubles besides (Wide), so that a component that is weak next to a strong one keeps its
// FP64 precision where the limiter drops the strong one. Values below 2^-1042 count as zero,
// and a window holding a value that is not finite gives NaN.
#pragma once
#include <math.h>
#include <stdint.h>

#ifdef __CUDACC__
#include <cuda_runtime.h>
#define AMRFD_HD __device__ __forceinline__
#define AMRFD_HD_CALL static __device__ __noinline__
#define AMRFD_TABLE static __device__ const
#define AMRFD_ANY(lanes, p) __any_sync((lanes), (p))
typedef unsigned line_t;  // shared-memory address of a line of doubles
#else  // a host compiler: one lane, for the tests of the arithmetic
#define AMRFD_HD static inline
#define AMRFD_HD_CALL static inline
#define AMRFD_TABLE static const
#define AMRFD_ANY(lanes, p) (p)
typedef const double* line_t;
struct float4 { float x, y, z, w; };
static inline float4 make_float4(float x, float y, float z, float w) { return {x, y, z, w}; }
#endif

namespace amrfd {

constexpr int kLimb = 22;                    // bits per limb
constexpr int kLimbMask = (1 << kLimb) - 1;
constexpr int kExpMax = 2030;                // largest biased exponent of a sweep's top
constexpr int kExpUnit = 87;                 // smallest biased exponent of a scale's lob

constexpr float kTiny = 1e-27f;

template <int N>
struct Limbs {  // a fixed-point number: sum of v[l] 2^(22 l) units
  int v[N];
};
// binades below the top exponent whose 53-bit values are whole numbers of N limbs
constexpr int room(int n) { return n * kLimb - 53; }
// floats of differences are in units of 2^float_shift(N) fixed-point units (a top limb has
// the same weight for every N)
constexpr int float_shift(int n) { return n * kLimb - 46; }

AMRFD_HD unsigned shf_l(unsigned lo, unsigned hi, int s) {  // high word of (hi:lo) << (s & 31)
#ifdef __CUDACC__
  return __funnelshift_l(lo, hi, s);
#else
  s &= 31;
  return s ? (hi << s) | (lo >> (32 - s)) : hi;
#endif
}
AMRFD_HD unsigned shf_r(unsigned lo, unsigned hi, int s) {  // low word of (hi:lo) >> (s & 31)
#ifdef __CUDACC__
  return __funnelshift_r(lo, hi, s);
#else
  s &= 31;
  return s ? (lo >> s) | (hi << (32 - s)) : lo;
#endif
}
AMRFD_HD void words(double x, int& hi, unsigned& lo) {
#ifdef __CUDACC__
  asm("mov.b64 {%0, %1}, %2;" : "=r"(lo), "=r"(hi) : "d"(x));
#else
  union { double d; unsigned long long u; } c;
  c.d = x;
  hi = (int)(unsigned)(c.u >> 32);
  lo = (unsigned)c.u;
#endif
}
// The words of element j of a line.
AMRFD_HD void cell_words(line_t l, int j, int& hi, unsigned& lo) {
#ifdef __CUDACC__
  asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(lo), "=r"(hi) : "r"(l + 8u * (unsigned)j));
#else
  words(l[j], hi, lo);
#endif
}
AMRFD_HD line_t line_at(line_t l, int j) {
#ifdef __CUDACC__
  return l + 8u * (unsigned)j;
#else
  return l + j;
#endif
}
AMRFD_HD int cell_hi(line_t l, int j) {
#ifdef __CUDACC__
  int hi;
  asm volatile("ld.shared.u32 %0, [%1];" : "=r"(hi) : "r"(l + 8u * (unsigned)j + 4u));
  return hi;
#else
  int hi;
  unsigned lo;
  words(l[j], hi, lo);
  return hi;
#endif
}
AMRFD_HD double from_words(int hi, unsigned lo) {
#ifdef __CUDACC__
  double x;
  asm("mov.b64 %0, {%1, %2};" : "=d"(x) : "r"(lo), "r"(hi));
  return x;
#else
  union { double d; unsigned long long u; } c;
  c.u = ((unsigned long long)(unsigned)hi << 32) | lo;
  return c.d;
#endif
}
// 2^e as a double, 0 or infinity beyond the normal range
AMRFD_HD double pow2d(int e) {
  const int b = e + 1023;
  return from_words(b < 1 ? 0 : (b > 2046 ? 0x7ff00000 : b << 20), 0u);
}

// The limbs of a value whose exponent lies in [lob >> 20, (lob >> 20) + 13] (or zero): the
// mantissa shifted left. lob = (exponent whose mantissa's last bit is the unit) << 20.
AMRFD_HD Limbs<3> limbs(int hi, unsigned lo, int lob) {
  const int x = hi & 0x7fffffff;
  const int L = (x - lob) >> 20;
  const unsigned m = ((unsigned)hi & 0xfffffu) | 0x100000u;
  const int sg = x ? ((hi >> 31) | 1) : 0;
  const unsigned w0 = shf_l(0u, lo, L), w1 = shf_l(lo, m, L), w2 = shf_l(m, 0u, L);
  Limbs<3> r;
  r.v[0] = (int)(w0 & (unsigned)kLimbMask) * sg;
  r.v[1] = (int)(shf_r(w0, w1, 22) & (unsigned)kLimbMask) * sg;
  r.v[2] = (int)shf_r(w1, w2, 12) * sg;
  return r;
}

// The limbs of a mantissa m shifted left by L <= 57, of sign sg.
AMRFD_HD Limbs<5> limbs5(unsigned mh, unsigned ml, int L, int sg) {
  const unsigned a0 = shf_l(0u, ml, L), a1 = shf_l(ml, mh, L), a2 = shf_l(mh, 0u, L);  // by L & 31
  const bool up = L >= 32;
  const unsigned w0 = up ? 0u : a0, w1 = up ? a0 : a1, w2 = up ? a1 : a2, w3 = up ? a2 : 0u;
  Limbs<5> r;
  r.v[0] = (int)(w0 & (unsigned)kLimbMask) * sg;
  r.v[1] = (int)(shf_r(w0, w1, 22) & (unsigned)kLimbMask) * sg;
  r.v[2] = (int)(shf_r(w1, w2, 12) & (unsigned)kLimbMask) * sg;
  r.v[3] = (int)((w2 >> 2) & (unsigned)kLimbMask) * sg;
  r.v[4] = (int)shf_r(w2, w3, 24) * sg;
  return r;
}
// The limbs of any value below the top, rounded to the unit (half away from zero; exact for
// whole multiples of it); FIT: of one whose exponent lies in [lob >> 20, (lob >> 20) + 57].
template <bool FIT = false>
AMRFD_HD Limbs<5> limbs_wide(int hi, unsigned lo, int lob) {
  const int x = hi & 0x7fffffff;
  int L = (x - lob) >> 20;
  unsigned mh = ((unsigned)hi & 0xfffffu) | 0x100000u;
  if (!FIT && L < 0) {
    const unsigned long long m = ((unsigned long long)mh << 32) | lo;
    const unsigned long long r = L < -54 ? 0ull : (m + (1ull << (-L - 1))) >> -L;
    mh = (unsigned)(r >> 32);
    lo = (unsigned)r;
    L = 0;
  }
  return limbs5(mh, lo, L, x ? ((hi >> 31) | 1) : 0);
}
// The same at scales down to the last bit of the subnormals, which have no leading one. What
// lies below 2^-1042 (no bit in the high word) counts as zero, as in every sweep.
AMRFD_HD Limbs<5> limbs_low(int hi, unsigned lo, int lob) {
  const int x = hi & 0x7fffffff;
  const bool sub = x < 0x100000;
  unsigned mh = sub ? (unsigned)x : ((unsigned)hi & 0xfffffu) | 0x100000u;
  int L = (sub ? 1 : x >> 20) - (lob >> 20);
  if (L < 0) {
    const unsigned long long m = ((unsigned long long)mh << 32) | lo;
    const unsigned long long r = L < -54 ? 0ull : (m + (1ull << (-L - 1))) >> -L;
    mh = (unsigned)(r >> 32);
    lo = (unsigned)r;
    L = 0;
  }
  return limbs5(mh, lo, L, x ? ((hi >> 31) | 1) : 0);
}
// The same as limbs with four limbs: exponents in [lob >> 20, (lob >> 20) + 35].
AMRFD_HD Limbs<4> limbs4(int hi, unsigned lo, int lob) {
  const int x = hi & 0x7fffffff;
  const int L = (x - lob) >> 20;
  const unsigned m = ((unsigned)hi & 0xfffffu) | 0x100000u;
  const int sg = x ? ((hi >> 31) | 1) : 0;
  const unsigned a0 = shf_l(0u, lo, L), a1 = shf_l(lo, m, L), a2 = shf_l(m, 0u, L);  // by L & 31
  const bool up = L >= 32;
  const unsigned w0 = up ? 0u : a0, w1 = up ? a0 : a1, w2 = up ? a1 : a2;
  Limbs<4> r;
  r.v[0] = (int)(w0 & (unsigned)kLimbMask) * sg;
  r.v[1] = (int)(shf_r(w0, w1, 22) & (unsigned)kLimbMask) * sg;
  r.v[2] = (int)(shf_r(w1, w2, 12) & (unsigned)kLimbMask) * sg;
  r.v[3] = (int)(w2 >> 2) * sg;
  return r;
}
template <int N>
AMRFD_HD Limbs<N> to_limbs(int hi, unsigned lo, int lob) {
  if constexpr (N == 3) return limbs(hi, lo, lob);
  else if constexpr (N == 4) return limbs4(hi, lo, lob);
  else return limbs_wide(hi, lo, lob);
}

// A difference of two limb numbers (limbs below 2^24, exact in FP32) as a float in units of
// 2^float_shift(N): relative error <= 2^-23 (a prefix that cancels leaves an exact sum).
template <int N>
AMRFD_HD float to_float(const Limbs<N>& d) {
  float f = (float)d.v[N - 1] * 16777216.0f;  // 2^24
  float w = 4.0f;
#pragma unroll
  for (int l = N - 2; l >= 0; l--) {
    f = fmaf((float)d.v[l], w, f);
    w *= 2.384185791015625e-07f;  // 2^-22
  }
  return f;
}

template <int N>
AMRFD_HD __int128 to_wide(const Limbs<N>& d) {
  __int128 r = d.v[N - 1];
#pragma unroll
  for (int l = N - 2; l >= 0; l--) r = r * (1 << kLimb) + d.v[l];
  return r;
}

// The double nearest to a, |a| < 2^125.
AMRFD_HD double wide_double(__int128 a) {
  double f = 1.0;
  const __int128 h = a >> 96;
  if (h != 0 && h != -1) {  // 64 to 93 bits remain, the rest in a sticky one: a >> 44 is exact
    a = (a >> 32) | (__int128)((a & 0xffffffffll) != 0);
    f = 4294967296.0;
  }
  return f * fma((double)(long long)(a >> 44), 17592186044416.0, (double)((long long)a & ((1ll << 44) - 1)));
}

AMRFD_HD double scaled(double x, int adj) {  // x 2^(adj >> 20); normal results
  int hi;
  unsigned lo;
  words(x, hi, lo);
  return from_words(hi ? hi + adj : 0, lo);
}

// The double nearest to A - B (ties to even), units of 2^((lob >> 20) - 1075); limbs of the
// difference below 2^31, the whole below 2^(22 N + 9).
AMRFD_HD double to_double(const Limbs<3>& A, const Limbs<3>& B, int lob) {
  const int d0 = A.v[0] - B.v[0], d1 = A.v[1] - B.v[1], d2 = A.v[2] - B.v[2];
  const long long W = (long long)d1 * (1 << 22) + d0;
  const int H = d2 + ((int)(W >> 32) >> 12);  // the sum >> 44
  long long V = (long long)((unsigned long long)W + ((unsigned long long)(unsigned)d2 << 44));
  int adj = lob - (1075 << 20);
  if ((unsigned)(H + (1 << 18)) >= (1u << 19)) {
    // over 62 bits: drop 6 or 13 into a sticky one; 55 or more remain
    const long long r = W & ((1ll << 44) - 1);
    const int sh = (unsigned)(H + (1 << 24)) < (1u << 25) ? 6 : 13;
    V = (long long)((unsigned long long)(long long)H << (44 - sh)) + (r >> sh);
    V |= (r & ((1ll << sh) - 1)) != 0;
    adj += sh << 20;
  }
#ifdef __CUDACC__
  const double x = __ll2double_rn(V);
#else
  const double x = (double)V;
#endif
  return scaled(x, adj);
}
// The double nearest to X 2^44 + r, 0 <= r < 2^44, in units of 2^(adj >> 20).
AMRFD_HD double round_sum(long long X, unsigned long long r, int adj) {
  const long long a = X ^ (X >> 63);
#ifdef __CUDACC__
  const int nb = 64 - __clzll(a);
#else
  const int nb = a ? 64 - __builtin_clzll((unsigned long long)a) : 0;
#endif
  const int sh = nb > 18 ? nb - 18 : 0;  // over 62 bits: the rest into a sticky one
  long long V = (long long)((unsigned long long)X << (44 - sh)) + (long long)(r >> sh);
  V |= (r & ((1ull << sh) - 1)) != 0;
#ifdef __CUDACC__
  const double x = __ll2double_rn(V);
#else
  const double x = (double)V;
#endif
  return scaled(x, adj + (sh << 20));
}
// The same for one number of four limbs, each below 2^31.
AMRFD_HD double to_double(const Limbs<4>& d, int lob) {
  const long long W = (long long)d.v[1] * (1 << 22) + d.v[0];
  const long long X = (long long)d.v[3] * (1 << 22) + d.v[2] + (W >> 44);  // the sum >> 44
  return round_sum(X, (unsigned long long)W & ((1ull << 44) - 1), lob - (1075 << 20));
}
AMRFD_HD double to_double(const Limbs<4>& A, const Limbs<4>& B, int lob) {
  return to_double(Limbs<4>{{A.v[0] - B.v[0], A.v[1] - B.v[1], A.v[2] - B.v[2], A.v[3] - B.v[3]}}, lob);
}
// Five: one conversion too (two and two more FP64 operations through 128 bits cost a sweep
// 256 cycles a cell).
AMRFD_HD double to_double(const Limbs<5>& d, int lob) {
  constexpr unsigned long long low = (1ull << 44) - 1;
  const long long W = (long long)d.v[1] * (1 << 22) + d.v[0];
  const long long X = (long long)d.v[3] * (1 << 22) + d.v[2] + (W >> 44);
  long long Z = d.v[4] + (X >> 44);  // the sum >> 88, below 2^32
  unsigned long long x = (unsigned long long)X & low, r = (unsigned long long)W & low;
  const bool large = (unsigned long long)(Z + (1 << 18)) >= (1ull << 19);  // then the lowest 44 bits into a sticky one
  int adj = lob - (1075 << 20);
  if (large) {
    x |= r != 0;
    r = x;
    adj += 44 << 20;
  } else {
    Z = (long long)((unsigned long long)Z << 44) + (long long)x;
  }
  return round_sum(Z, r, adj);
}
AMRFD_HD double to_double(const Limbs<5>& A, const Limbs<5>& B, int lob) {
  Limbs<5> d;
#pragma unroll
  for (int l = 0; l < 5; l++) d.v[l] = A.v[l] - B.v[l];
  return to_double(d, lob);
}

// ----------------------------------------------------------------------- MP5
// MP5 (Suresh & Huynh 1997) at face i+1/2 from (f_{i-2}, ..., f_{i+2}), in the differences
// dm = f_{i-1}-f_{i-2}, d0 = f_i-f_{i-1}, d1 = f_{i+1}-f_i, dp = f_{i+2}-f_{i+1} and the
// curvature-limited second differences Mp (at i+1/2) and Mm (at i-1/2):
//   f_or - f_i = (11 d0 - 2 dm + 24 d1 - 3 dp)/60,  f_mp - f_i = minmod(d1, 4 d0),
//   f_ul - f_i = 4 d0,  f_md - f_i = d1/2 - Mp/2,  f_lc - f_i = d0/2 + 4 Mm/3,
// with the acceptance test (f_or - f_i)(f_or - f_mp) <= 1e-10 (on F^{+-} = G^{+-}/2) and
// otherwise median(f_or, f_min, f_max).
// Per face and bias, with the differences of the five stencil cells (the right-biased
// stencil reversed), every candidate of the limiter is a whole combination of
// them after scaling by 30: 30 times the doubled value relative to the centre cell,
//   X = -2 dm + 11 d0 + 24 d1 - 3 dp (unlimited),  0,  60 d1,  30 md = 30 (d1 - Mp),
//   30 ul = 240 d0,  30 lc = 30 d0 + 80 Mm,
// Mp, Mm one of 0, ka, kb, 4 ka - kb, 4 kb - ka of two neighbouring curvatures. The rows
// give each combination less the unlimited one as coefficients of the five cells; a row is
// the piece of the value and of Mp or Mm, as recorded for the adjoint: 0 X,
// 1 zero, 2 d1, 3 md, 4 ul, 5 lc, and 0 zero, 1 ka, 2 kb, 3 4 ka - kb, 4 4 kb - ka.
struct alignas(16) CoefRow { short v[8]; };
AMRFD_TABLE CoefRow g_mp5_coef[14] = {
    {{0, 0, 0, 0, 0, 0, 0, 0}},  // 0  unlimited: no correction
    {{-2, 13, 13, -27, 3, 0, 0, 0}},  // 1  zero
    {{-2, 13, -47, 33, 3, 0, 0, 0}},  // 2  2 d1
    {{-2, 13, -17, 3, 3, 0, 0, 0}},  // 3  md, Mp = 0
    {{-2, -17, 43, -27, 3, 0, 0, 0}},  // 4  md, Mp = kC = d1 - d0
    {{-2, 13, -47, 63, -27, 0, 0, 0}},  // 5  md, Mp = kR = dp - d1
    {{-2, -107, 253, -177, 33, 0, 0, 0}},  // 6  md, Mp = 4 kC - kR
    {{-2, 43, -197, 273, -117, 0, 0, 0}},  // 7  md, Mp = 4 kR - kC
    {{-2, -227, 253, -27, 3, 0, 0, 0}},  // 8  ul = 8 d0
    {{-2, -17, 43, -27, 3, 0, 0, 0}},  // 9  lc, Mm = 0
    {{78, -177, 123, -27, 3, 0, 0, 0}},  // 10  lc, Mm = kL = d0 - dm
    {{-2, 63, -117, 53, 3, 0, 0, 0}},  // 11  lc, Mm = kC
    {{318, -737, 523, -107, 3, 0, 0, 0}},  // 12  lc, Mm = 4 kL - kC
    {{-82, 463, -677, 293, 3, 0, 0, 0}},  // 13  lc, Mm = 4 kC - kL
};
constexpr int kD0Code = 3 | (1 << 3);
// Row of a recorded code (piece | Mp's piece << 3 | Mm's piece << 6).
AMRFD_HD int mp5_row(int code) {
  const int s = code & 7;
  if (s == 3) return 3 + ((code >> 3) & 7);
  if (s == 5) return 9 + ((code >> 6) & 7);
  return s == 4 ? 8 : s;
}

// 30 X, the bound's sum 24|d1| + 11|d0| + 2|dm| + 3|dp|, and t = 30X (30X - 30mp) with a
// bound B of its error: |t - exact| <= B. Inputs carry a relative error of 2^-23, so 30X
// is off by at most 2^-21 S, 30 mp by 2^-22 |30 mp|, and t by less than 2^-19 S (S + |30 mp|).
AMRFD_HD void mp5_test(float dm, float d0, float d1, float dp, float& X, float& t, float& B) {
  X = fmaf(-3.0f, dp, fmaf(24.0f, d1, fmaf(11.0f, d0, -2.0f * dm)));
  const float S = fmaf(3.0f, fabsf(dp), fmaf(24.0f, fabsf(d1), fmaf(11.0f, fabsf(d0), 2.0f * fabsf(dm))));
  const float a = 4.0f * d0;
  // minmod(d1, 4 d0) = median(0, d1, 4 d0)
  const float m = fmaxf(fminf(a, 0.0f), fminf(fmaxf(a, 0.0f), d1));
  t = X * fmaf(-60.0f, m, X);
  B = (1.9073486328125e-06f * S) * fmaf(60.0f, fabsf(m), S);
}
// Floats of differences are zero exactly where the differences are.
AMRFD_HD bool equal_cells(float dm, float d0, float d1, float dp) {
  return fmaxf(fmaxf(fabsf(dm), fabsf(d0)), fmaxf(fabsf(d1), fabsf(dp))) == 0.0f;
}
// Whether the acceptance test surely holds, cheaper: with m between 0 and each of d1, 4 d0
// or outside, t is at most the larger of 30X (30X - 60 d1) and 30X (30X - 240 d0), whose
// FP32 error is below 0.0091 max|d|^2 (|30X| <= 40 max|d|). Equal cells need no threshold: in
// large units it is below what FP32's products can tell from zero (thr_lo is -kTiny then), and
// uniform lines of 1e25 or more would all be limited and taken cell by cell.
AMRFD_HD bool mp5_accepts(float dm, float d0, float d1, float dp, float thr_lo) {
  const float X = fmaf(-3.0f, dp, fmaf(24.0f, d1, fmaf(11.0f, d0, -2.0f * dm)));
  const float q = fmaxf(X * fmaf(-60.0f, d1, X), X * fmaf(-240.0f, d0, X));
  const float mx = fmaxf(fmaxf(fabsf(dm), fabsf(d0)), fmaxf(fabsf(d1), fabsf(dp)));
  return fmaf(0.01171875f * mx, mx, q) < thr_lo || mx == 0.0f;
}

// minmod4(4 ka - kb, 4 kb - ka, ka, kb) in FP32 and its piece (0 zero, 1 ka, 2 kb,
// 3 4 ka - kb, 4 4 kb - ka); piece -1 when two candidates lie within tau of the value.
AMRFD_HD float m4_float(float ka, float kb, float tau, int& piece) {
  const float c3 = fmaf(4.0f, ka, -kb), c4 = fmaf(4.0f, kb, -ka);
  float v = 0.0f;
  if (ka > 0.0f && kb > 0.0f) v = fmaxf(0.0f, fminf(fminf(ka, kb), fminf(c3, c4)));
  if (ka < 0.0f && kb < 0.0f) v = fminf(0.0f, fmaxf(fmaxf(ka, kb), fmaxf(c3, c4)));
  const bool n0 = fabsf(v) <= tau, n1 = fabsf(v - ka) <= tau, n2 = fabsf(v - kb) <= tau, n3 = fabsf(v - c3) <= tau,
             n4 = fabsf(v - c4) <= tau;
  const int n = n0 + n1 + n2 + n3 + n4;
  piece = n != 1 ? -1 : (n0 ? 0 : (n1 ? 1 : (n2 ? 2 : (n3 ? 3 : 4))));
  return v;
}

// The code of a face that mp5_accepts did not pass, from FP32; -1 when FP32 cannot tell.
// With s = |dm| + |d0| + |d1| + |dp| every candidate's error is below 2^-18 s (curvatures
// 2^-22.4 s, 4 ka - kb 2^-20.1 s, 8/3 of that 2^-18.7 s), and min, max and median are
// 1-Lipschitz, so a piece whose value is the only one within 2^-17 s of the result is the
// exact selection. Candidates that vanish exactly (equal cells: fronts into a uniform
// state) count as one.
AMRFD_HD int mp5_code_float(float dm, float d0, float d1, float dp, float thr_lo) {
  float X, t, B;
  mp5_test(dm, d0, d1, dp, X, t, B);
  if (t + B < thr_lo || equal_cells(dm, d0, d1, dp)) return 0;
  // thr_lo lies below the threshold by 2^-20: its upper side is 2^-19 above that
  if (!(t - B > fmaxf(thr_lo * 1.0000020f, kTiny))) return -1;
  const float tau = 7.62939453125e-06f * (fabsf(dm) + fabsf(d0) + fabsf(d1) + fabsf(dp));
  const float kL = d0 - dm, kC = d1 - d0, kR = dp - d1;
  int cp, cm;
  const float Mp = m4_float(kC, kR, tau, cp), Mm = m4_float(kL, kC, tau, cm);
  const float x = X * (1.0f / 30.0f), c1 = 2.0f * d1, c2 = d1 - Mp, c3 = 8.0f * d0, c4 = fmaf(8.0f / 3.0f, Mm, d0);
  const float lo = fmaxf(fminf(fminf(0.0f, c1), c2), fminf(fminf(0.0f, c3), c4));
  const float hi = fminf(fmaxf(fmaxf(0.0f, c1), c2), fmaxf(fmaxf(0.0f, c3), c4));
  const float r = fmaxf(fminf(x, lo), fminf(fmaxf(x, lo), hi));
  // exact zeros: d1, and md where besides kC or kR vanishes; d0, and lc where kL or kC does
  const bool z1 = d1 == 0.0f, z0 = d0 == 0.0f, z2 = z1 && (z0 || dp == 0.0f), z4 = z0 && (z1 || dm == 0.0f);
  const bool nx = fabsf(x - r) <= tau, n0 = fabsf(r) <= tau, n1 = fabsf(c1 - r) <= tau && !z1,
             n2 = fabsf(c2 - r) <= tau && !z2, n3 = fabsf(c3 - r) <= tau && !z0, n4 = fabsf(c4 - r) <= tau && !z4;
  // md with Mp = kC and lc with Mm = 0 are the same combination, d0: recorded as the former
  const bool same = n2 && n4 && cp == 1 && cm == 0;
  if (nx + n0 + n1 + n2 + n3 + n4 - same != 1) return -1;
  if (nx) return 0;
  if (n0) return 1;
  if (n1) return 2;
  if (n3) return 4;
  if (n2) return cp < 0 ? -1 : 3 | (cp << 3);
  return cm < 0 ? -1 : (cm == 0 ? kD0Code : 5 | (cm << 6));
}

// minmod4 in FP32 from curvatures known to ea, eb, and its piece as m4_float's; e: the
// value's error.
AMRFD_HD float m4_bounded(float ka, float ea, float kb, float eb, int& piece, float& e) {
  const float sg = ka < 0.0f ? -1.0f : 1.0f, a = ka * sg, b = kb * sg;
  piece = 0;
  e = 0.0f;
  if (b < -eb || (ea == 0.0f && a == 0.0f) || (eb == 0.0f && b == 0.0f)) return 0.0f;
  const float c3 = fmaf(4.0f, a, -b), c4 = fmaf(4.0f, b, -a), e3 = fmaf(4.0f, ea, eb), e4 = fmaf(4.0f, eb, ea);
  if (a > ea && b > eb && (c3 < -1.01f * e3 || c4 < -1.01f * e4)) return 0.0f;
  const float v = fmaxf(0.0f, fminf(fminf(a, b), fminf(c3, c4)));
  // the candidate that gave v, if no other one's interval meets its own
  const bool i1 = v == a, i2 = !i1 && v == b, i3 = !i1 && !i2 && v == c3, i4 = !i1 && !i2 && !i3 && v == c4;
  const float es = i1 ? ea : (i2 ? eb : (i3 ? e3 : e4));
  const bool clear = v > es && (i1 || a - v > 1.01f * (ea + es)) && (i2 || b - v > 1.01f * (eb + es)) &&
                     (i3 || c3 - v > 1.01f * (e3 + es)) && (i4 || c4 - v > 1.01f * (e4 + es));
  e = 1.01f * (clear ? es : fmaxf(e3, e4));
  piece = clear ? (i1 ? 1 : (i2 ? 2 : (i3 ? 3 : 4))) : -1;
  return v * sg;
}

// A second look at a face mp5_code_float could not settle, with an error for every candidate
// (differences far smaller than the stencil's largest, as ahead of a front, keep their own
// precision): the selection is exact when no other candidate's interval meets the selected
// one's, for which candidates lie above and below it then does not depend on the errors.
AMRFD_HD int mp5_code_bounded(float dm, float d0, float d1, float dp, float thr_lo) {
  constexpr float u = 1.1920929e-07f;  // 2^-23, the differences' relative error
  float X, t, B;
  mp5_test(dm, d0, d1, dp, X, t, B);
  if (t + B < thr_lo || equal_cells(dm, d0, d1, dp)) return 0;
  if (!(t - B > fmaxf(thr_lo * 1.0000020f, kTiny))) return -1;
  const float am = fabsf(dm), a0 = fabsf(d0), a1 = fabsf(d1), ap = fabsf(dp);
  const float kL = d0 - dm, kC = d1 - d0, kR = dp - d1;
  int cp, cm;
  float eP, eM;
  const float Mp = m4_bounded(kC, 2.0f * u * (a1 + a0), kR, 2.0f * u * (ap + a1), cp, eP);
  const float Mm = m4_bounded(kL, 2.0f * u * (a0 + am), kC, 2.0f * u * (a1 + a0), cm, eM);
  float c[6], e[6];
  c[0] = X * (1.0f / 30.0f);
  e[0] = 0.15f * u * fmaf(3.0f, ap, fmaf(24.0f, a1, fmaf(11.0f, a0, 2.0f * am)));  // 4 u S / 30
  c[1] = 0.0f;
  e[1] = 0.0f;
  c[2] = 2.0f * d1;
  e[2] = 2.0f * u * a1;
  c[3] = d1 - Mp;
  e[3] = fmaf(2.0f * u, a1 + fabsf(Mp), eP);
  c[4] = 8.0f * d0;
  e[4] = 8.0f * u * a0;
  c[5] = fmaf(8.0f / 3.0f, Mm, d0);
  e[5] = fmaf(2.0f * u, fmaf(3.0f, fabsf(Mm), a0), 2.7f * eM);
  const float lo = fmaxf(fminf(fminf(0.0f, c[2]), c[3]), fminf(fminf(0.0f, c[4]), c[5]));
  const float hi = fminf(fmaxf(fmaxf(0.0f, c[2]), c[3]), fmaxf(fmaxf(0.0f, c[4]), c[5]));
  const float r = fmaxf(fminf(c[0], lo), fminf(fmaxf(c[0], lo), hi));
  int s = -1;
  float es = 0.0f;
#pragma unroll
  for (int q = 5; q >= 0; q--)
    if (c[q] == r) { s = q; es = e[q]; }  // an exact zero by its own name
  if (r == 0.0f) { s = 1; es = 0.0f; }
  // md with Mp = kC and lc with Mm = 0 are the same combination, d0
  const bool same = cp == 1 && cm == 0 && (s == 3 || s == 5);
  bool clear = s >= 0;
#pragma unroll
  for (int q = 0; q < 6; q++) {
    const bool zero = s == 1 && c[q] == 0.0f && e[q] == 0.0f;  // also exactly zero
    if (q != s && !zero && !(same && (q == 3 || q == 5))) clear = clear && fabsf(c[q] - r) > 1.01f * (e[q] + es);
  }
  if (!clear) return -1;
  if (s == 3) return cp < 0 ? -1 : 3 | (cp << 3);
  if (s == 5) return cm < 0 ? -1 : (cm == 0 ? kD0Code : 5 | (cm << 6));
  return s;
}

// ------------------------------------------------------------- wide numbers
// h units + r. With RES (a window that spans more than the units reach) r carries what the
// whole units of each cell left over, as a double of its own: a value far below the unit is
// then all remainder and keeps its FP64 precision where the limiter drops the large ones.
// Without RES every cell is a whole number of units and r is not used.
template <bool RES>
struct Wide {
  __int128 h;
  double r;
};
struct Unit {  // of a scale lob: the unit as a double, its reciprocal
  double u, inv;
};
AMRFD_HD Unit unit_of(int lob) { return {pow2d((lob >> 20) - 1075), pow2d(1075 - (lob >> 20))}; }

AMRFD_HD bool any_bits(double x) {  // not +-0, without an FP64 comparison
  int hi;
  unsigned lo;
  words(x, hi, lo);
  return ((hi << 1) | (int)lo) != 0;
}
// |r| <= unit/2 (or a little more) again, so that h and then r order the numbers.
template <bool RES>
AMRFD_HD void carry_units(Wide<RES>& c, const Unit& un) {
  int hr, hu;
  unsigned lr, lu;
  words(c.r, hr, lr);
  words(un.u, hu, lu);
  if ((hr & 0x7fffffff) < hu - (1 << 20)) return;
  const double q = rint(c.r * un.inv);
  c.h += (long long)q;
  c.r = fma(-q, un.u, c.r);
}
// ca a + cb b
template <bool RES>
AMRFD_HD Wide<RES> lin(int ca, const Wide<RES>& a, int cb, const Wide<RES>& b, const Unit& un) {
  Wide<RES> c;
  c.h = a.h * ca + b.h * cb;
  c.r = 0.0;
  if (RES && (any_bits(a.r) || any_bits(b.r))) {
    c.r = fma((double)ca, a.r, (double)cb * b.r);
    carry_units(c, un);
  }
  return c;
}
template <bool RES>
AMRFD_HD bool less(const Wide<RES>& a, const Wide<RES>& b) {
  return a.h < b.h || (RES && a.h == b.h && a.r < b.r);
}
template <bool RES>
AMRFD_HD int sign(const Wide<RES>& a) {
  if (a.h != 0) return a.h < 0 ? -1 : 1;
  return RES ? (a.r > 0.0) - (a.r < 0.0) : 0;
}
template <bool RES>
AMRFD_HD Wide<RES> absw(const Wide<RES>& a) {
  return sign(a) < 0 ? Wide<RES>{-a.h, RES ? -a.r : 0.0} : a;
}
// The number as a float in units of 2^float_shift(5): relative error <= 2^-23. small: not zero,
// but too small for FP32's comparisons.
template <bool RES>
AMRFD_HD float wide_float(const Wide<RES>& a, const Unit& un, bool& small) {
  const __int128 m = a.h < 0 ? -a.h : a.h;
  float f;
  if (RES && any_bits(a.r) && m < (1 << 26)) {
    const double x = (double)(int)m + (a.h < 0 ? -a.r : a.r) * un.inv;
    f = (float)(x * 0x1p-64);
    small |= fabsf(f) < 1e-30f;
  } else {
    f = (float)(int)(m >> 96) * 0x1p32f;
    f = fmaf((float)(int)((m >> 72) & 0xffffff), 0x1p8f, f);
    f = fmaf((float)(int)((m >> 48) & 0xffffff), 0x1p-16f, f);
    f = fmaf((float)(int)((m >> 24) & 0xffffff), 0x1p-40f, f);
    f = fmaf((float)(int)(m & 0xffffff), 0x1p-64f, f);
  }
  return a.h < 0 ? -f : f;
}
template <bool RES>  // in units
AMRFD_HD double in_units(const Wide<RES>& a, const Unit& un) {
  return RES ? fma(a.r, un.inv, wide_double(a.h)) : wide_double(a.h);
}
// The double nearest to the number, |h| < 2^122; infinity beyond the largest.
template <bool RES>
AMRFD_HD double nearest(const Wide<RES>& a, const Unit& un, int lob) {
  const int e = (lob >> 20) - 1075;
  if (RES && a.r != 0.0) {
    if (absw(Wide<false>{a.h, 0.0}).h < (1ll << 53)) return fma((double)(long long)a.h, un.u, a.r);
    return ldexp(wide_double(4 * a.h + (a.r > 0.0 ? 1 : -1)), e - 2);  // r decides a tie
  }
  return ldexp(wide_double(a.h), e);
}
// Element j of a line. Cells whose units round: half away from zero.
template <bool RES>
AMRFD_HD Wide<RES> wide_cell(line_t l, int j, int lob, const Unit& un) {
  int hi;
  unsigned lo;
  cell_words(l, j, hi, lo);
  const int L = ((hi & 0x7fffffff) - lob) >> 20;
  const unsigned long long m = ((unsigned long long)(((unsigned)hi & 0xfffffu) | 0x100000u) << 32) | lo;
  Wide<RES> a = {0, 0.0};
  if (L >= 0) a.h = (__int128)m << L;
  else if (L >= -54) a.h = (__int128)((m + (1ull << (-L - 1))) >> -L);
  if (hi < 0) a.h = -a.h;
  if (RES && L < 0) a.r = a.h == 0 ? from_words(hi, lo) : fma(-(double)(long long)a.h, un.u, from_words(hi, lo));
  return a;
}

// minmod4 and its piece, exactly.
template <bool RES>
AMRFD_HD Wide<RES> m4_exact(const Wide<RES>& ka, const Wide<RES>& kb, const Unit& un, int& piece) {
  const Wide<RES> zero = {0, 0.0};
  piece = 0;
  const int sg = sign(ka);
  if (sg == 0 || sg != sign(kb)) return zero;
  const bool as = less(absw(ka), absw(kb));
  const Wide<RES> s = as ? ka : kb, t = lin(4, s, -1, as ? kb : ka, un);
  if (sign(t) != sg) return zero;
  const bool four = less(absw(t), absw(s));
  piece = four ? (as ? 3 : 4) : (as ? 1 : 2);
  return four ? t : s;
}
template <bool RES>
AMRFD_HD void minw(const Wide<RES>& a, int ca, const Wide<RES>& b, int cb, Wide<RES>& r, int& cr) {
  const bool t = less(a, b);
  r = t ? a : b;
  cr = t ? ca : cb;
}
template <bool RES>
AMRFD_HD void maxw(const Wide<RES>& a, int ca, const Wide<RES>& b, int cb, Wide<RES>& r, int& cr) {
  const bool t = less(a, b);
  r = t ? b : a;
  cr = t ? cb : ca;
}

// The code of a face and 30 times its doubled value y relative to the centre cell, in exact
// arithmetic. thr: the acceptance threshold on 30X (30X - 30mp) in squared units; the
// product of the two exact factors, each rounded to FP64, is compared with it.
template <bool RES>
AMRFD_HD int mp5_exact(const Wide<RES>& dm, const Wide<RES>& d0, const Wide<RES>& d1, const Wide<RES>& dp, double thr,
                       const Unit& un, Wide<RES>& y) {
  const Wide<RES> zero = {0, 0.0};
  const Wide<RES> X = lin(1, lin(24, d1, 11, d0, un), -1, lin(2, dm, 3, dp, un), un);
  Wide<RES> mp = zero;
  const Wide<RES> d04 = lin(4, d0, 0, zero, un);
  if (sign(d1) == sign(d0)) mp = less(absw(d1), absw(d04)) ? d1 : d04;
  const Wide<RES> Z = lin(1, X, -60, mp, un);
  y = X;
  if (sign(X) * sign(Z) <= 0) return 0;
  if (in_units(absw(X), un) * in_units(absw(Z), un) <= thr) return 0;
  const Wide<RES> kL = lin(1, d0, -1, dm, un), kC = lin(1, d1, -1, d0, un), kR = lin(1, dp, -1, d1, un);
  int cp, cm;
  const Wide<RES> Mp = m4_exact(kC, kR, un, cp), Mm = m4_exact(kL, kC, un, cm);
  const Wide<RES> md = lin(30, d1, -30, Mp, un), lc = lin(30, d0, 80, Mm, un), d12 = lin(60, d1, 0, zero, un),
                  ul = lin(60, d04, 0, zero, un);
  Wide<RES> a, b, lo, hi, t1, t2, t3;
  int ca, cb, cl, ch, c1, c2, c3, code;
  minw(zero, 1, d12, 2, a, ca);
  minw(a, ca, md, 3, a, ca);
  minw(zero, 1, ul, 4, b, cb);
  minw(b, cb, lc, 5, b, cb);
  maxw(a, ca, b, cb, lo, cl);
  maxw(zero, 1, d12, 2, a, ca);
  maxw(a, ca, md, 3, a, ca);
  maxw(zero, 1, ul, 4, b, cb);
  maxw(b, cb, lc, 5, b, cb);
  minw(a, ca, b, cb, hi, ch);
  minw(X, 0, lo, cl, t1, c1);
  maxw(X, 0, lo, cl, t2, c2);
  minw(t2, c2, hi, ch, t3, c3);
  maxw(t1, c1, t3, c3, y, code);
  if (sign(y) == 0) return 1;  // as the FP32 selection names an exact zero
  if (code == 3) return 3 | (cp << 3);
  if (code == 5) return cm == 0 ? kD0Code : 5 | (cm << 6);
  return code;
}

// --------------------------------------------------------------------- LIMO3
// With a, b the differences left and right of the centre cell, 30 times the value:
// y3 10 a + 20 b, -a/2 -15 a, 2a 60 a, 1.6 b 48 b. Codes, as recorded for the adjoint:
// piece (0 zero, 1 y3, 2 -a/2, 3 2a, 4 1.6 b) | mode << 3 (0 unlimited, 1 limited, 2 / 3 in
// the blend band). From FP32, -1 when it cannot tell; thr = 4 (r dx)^2 in squared units.
AMRFD_HD int limo3_code_float(float a, float b, float thr) {
  const float s2 = fmaf(a, a, b * b);
  if (s2 < thr * 0.99999809f || (a == 0.0f && b == 0.0f)) return 0;
  if (!(s2 > fmaxf(thr * 1.00000191f, kTiny))) return -1;
  if (a == 0.0f || b == 0.0f) return 1 << 3;  // exactly zero, as the exact selection names it
  const float sg = b < 0.0f ? -1.0f : 1.0f;
  const float ap = a * sg, bp = b * sg, y3 = fmaf(2.0f, bp, ap) * (1.0f / 3.0f);
  const float c2 = -0.5f * ap, c3 = 2.0f * ap, c4 = 1.6f * bp;
  const float r = fmaxf(0.0f, fminf(y3, fmaxf(c2, fminf(fminf(c3, y3), c4))));
  const float tau = 3.814697265625e-06f * (fabsf(a) + fabsf(b));  // 2^-18; candidate errors < 2^-20
  const bool n0 = r <= tau, n1 = fabsf(y3 - r) <= tau, n2 = fabsf(c2 - r) <= tau, n3 = fabsf(c3 - r) <= tau,
             n4 = fabsf(c4 - r) <= tau;
  if (n0 + n1 + n2 + n3 + n4 != 1) return -1;
  return (n0 ? 0 : (n1 ? 1 : (n2 ? 2 : (n3 ? 3 : 4)))) | (1 << 3);
}

// The code and 30 times the value in exact arithmetic; inside the blend band the value's
// difference from y3 is formed in FP64. thr as above.
template <bool RES>
AMRFD_HD int limo3_exact(const Wide<RES>& a, const Wide<RES>& b, double thr, const Unit& un, Wide<RES>& y) {
  const Wide<RES> zero = {0, 0.0};
  const double fa = in_units(a, un), fb = in_units(b, un), s2 = fma(fa, fa, fb * fb);
  const Wide<RES> y3 = lin(10, a, 20, b, un);
  y = y3;
  if (s2 <= thr * (1.0 - 1e-12)) return 0;
  const int sg = sign(b) < 0 ? -1 : 1;
  const Wide<RES> yp = lin(sg, y3, 0, zero, un);
  Wide<RES> t;
  int c;
  minw(lin(60 * sg, a, 0, zero, un), 3, yp, 1, t, c);
  minw(t, c, lin(48 * sg, b, 0, zero, un), 4, t, c);
  maxw(lin(-15 * sg, a, 0, zero, un), 2, t, c, t, c);
  minw(yp, 1, t, c, t, c);
  maxw(zero, 0, t, c, t, c);
  if (s2 >= thr * (1.0 + 1e-12)) {
    y = lin(sg, t, 0, zero, un);
    return c | (1 << 3);
  }
  const double z = (s2 / thr - 1.0) * 1e12;
  const double x = in_units(lin(sg, t, -1, y3, un), un) * (0.5 * (1.0 + z));
  const long long xh = (long long)(x * 8.470329472543003e-22);  // 2^-70
  const double xl = x - (double)xh * 1.1805916207174113e+21;
  const long long xm = (long long)(xl * 5.820766091346741e-11);  // 2^-34
  const double xr = xl - (double)xm * 17179869184.0;
  const Wide<RES> d = {((__int128)xh << 70) + ((__int128)xm << 34) + (long long)xr,
                       RES ? (xr - (double)(long long)xr) * un.u : 0.0};
  y = lin(1, y3, 1, d, un);
  return c | ((z < 0.0 ? 2 : 3) << 3);
}

// ------------------------------------------------------------------- sweeps
// A cell's exponent word, with FINE raised by its mantissa's trailing zeros (that of a value
// with the same last bit and a full mantissa); 0 for a zero.
template <bool FINE>
AMRFD_HD unsigned cell_key(line_t l, int j, unsigned& a) {
  int hi;
  unsigned lo = 0u;
  if (FINE) cell_words(l, j, hi, lo);
  else hi = cell_hi(l, j);
  a = (unsigned)hi & 0x7fffffffu;
  unsigned k = a;
  if (FINE && a) {
    const unsigned m = lo ? lo : ((a & 0xfffffu) | 0x100000u);
#ifdef __CUDACC__
    const int z = __ffs((int)m) - 1;
#else
    const int z = __builtin_ctz(m);
#endif
    k += (unsigned)(z + (lo ? 0 : 32)) << 20;
  }
  return k;
}

// Largest exponent word and smallest key, less one (a zero wraps), of nc cells of both lines
// from j on.
struct Span { unsigned mx, mn; };
template <bool FINE>
AMRFD_HD Span window_span(line_t gp, line_t gm, int j, int nc) {
  Span w = {0u, 0xffffffffu};
  for (int q = 0; q < nc; q++) {
#pragma unroll
    for (int s = 0; s < 2; s++) {
      unsigned a;
      const unsigned k = cell_key<FINE>(s ? gm : gp, j + q, a);
      w.mx = a > w.mx ? a : w.mx;
      w.mn = k - 1u < w.mn ? k - 1u : w.mn;
    }
  }
  return w;
}
// The scale (lob) for N limbs; false when some cell is not a whole multiple of its unit or is
// 2^1008 or more. bad: a value that is not finite. HEAD: bits left free above the largest.
template <int N, int HEAD = 0, int LOW = kExpUnit>
AMRFD_HD bool span_scale(const Span& w, int& lob, bool& bad) {
  int top = (int)(w.mx >> 20);
  bad = top == 2047;
  top = bad ? 2046 : top;
  constexpr int span = room(N) - HEAD;
  lob = (top - span < LOW ? LOW : top - span) << 20;
  const unsigned low = w.mn == 0xffffffffu ? w.mn : (w.mn + 1u) >> 20;
  return (low >= (unsigned)(lob >> 20) || lob == 1 << 20) && top <= kExpMax;  // 1: the subnormals' own unit
}
// Both. FINE looks at the mantissas' trailing zeros, else every mantissa counts as 53 bits.
template <int N, bool FINE, int HEAD = 0>
AMRFD_HD bool window_scale(line_t gp, line_t gm, int j, int nc, int& lob, bool& bad) {
  return span_scale<N, HEAD>(window_span<FINE>(gp, gm, j, nc), lob, bad);
}

// The thresholds of the FP32 decisions in squared floats' units: MP5's acceptance threshold
// on 30X (30X - 30mp), 2^-20 below; LIMO3's switch. Below kTiny, where products could meet
// FP32's denormals, -kTiny: FP32 then settles only what lies farther from zero.
template <bool LIMO, int N>
AMRFD_HD float float_threshold(int lob, double limo_thr) {
  const int e = -((lob >> 20) - 1075) - float_shift(N);
  const float t = (float)(LIMO ? limo_thr * pow2d(e) * pow2d(e) : 1.43999863e-6 * pow2d(2 * e));  // 1.44e-6 (1 - 2^-20)
  return t < kTiny ? -kTiny : t;
}

template <bool REC>
AMRFD_HD void record(unsigned short* tp, unsigned short* tm, int f, int fend, int fmod, int cp, int cm) {
  if (REC && f < fend) {
    const int fi = f >= fmod ? f - fmod : f;
    tp[fi] = (unsigned short)cp;
    tm[fi] = (unsigned short)cm;
  }
}

// The limiter's correction of one stencil as coefficients of its cells (5 with MP5, 3 with
// LIMO3), from the left (G+) or from the right (G-): the selected combination less the
// unlimited one.
template <bool LIMO>
AMRFD_HD void limited_coefs(int code, int e[5]) {
  if constexpr (LIMO) {
    const int piece = code & 7;
    int ca = 0, cb = 0;  // of a and b
    if (((code >> 3) & 3) == 1) {
      ca = piece == 0 || piece == 4 ? -10 : (piece == 2 ? -25 : (piece == 3 ? 50 : 0));
      cb = piece == 1 ? 0 : (piece == 4 ? 28 : -20);
    }
    e[0] = -ca; e[1] = ca - cb; e[2] = cb;
  } else {
#ifdef __CUDACC__
    const uint4 t = *reinterpret_cast<const uint4*>(g_mp5_coef + mp5_row(code));
    e[0] = (int)(short)t.x; e[1] = (int)t.x >> 16; e[2] = (int)(short)t.y; e[3] = (int)t.y >> 16; e[4] = (int)(short)t.z;
#else
    for (int q = 0; q < 5; q++) e[q] = g_mp5_coef[mp5_row(code)].v[q];
#endif
  }
}

// Adds a whole number given limb by limb to F.
template <int N>
AMRFD_HD void add_carried(Limbs<N>& F, const long long* s) {
  long long carry = 0;
#pragma unroll
  for (int l = 0; l < N - 1; l++) {
    const long long t = s[l] + carry;
    F.v[l] += (int)t & kLimbMask;
    carry = t >> kLimb;
  }
  F.v[N - 1] += (int)(s[N - 1] + carry);
}

// A face's code from its differences in FP32, -1 when that cannot tell: numbers with
// remainders are costly to compare (28x78x45 MHD step: 733 us without, 663 with), whole ones
// cheaper exactly.
template <bool LIMO, bool RES>
AMRFD_HD int float_code(const Wide<RES>* D, float thr_lo, const Unit& un) {
  bool small = false;
  float f[4];
#pragma unroll
  for (int q = 0; q < (LIMO ? 2 : 4); q++) f[q] = wide_float(D[q], un, small);
  if (small) return -1;
  if constexpr (LIMO) return limo3_code_float(f[0], f[1], thr_lo);
  const int c = mp5_code_float(f[0], f[1], f[2], f[3], thr_lo);
  return c < 0 ? mp5_code_bounded(f[0], f[1], f[2], f[3], thr_lo) : c;
}

// One cell by itself, its comparisons exact: the cells a sweep could not finish (a
// comparison FP32 could not settle, a window over more than 110 bits, values of 2^1008 or
// more). i: the cell; its window starts at extended cell i + C0. RES: some value is no whole
// number of units.
template <bool LIMO, bool REC, bool RES>
AMRFD_HD double exact_value(line_t gp, line_t gm, int i, double limo_thr, int lob, unsigned short* tp,
                            unsigned short* tm, int f0, int fend, int fmod) {
  constexpr int NC = LIMO ? 4 : 6;
  constexpr int C0 = LIMO ? 1 : 0;
  constexpr int ND = LIMO ? 2 : 4;
  const Unit un = unit_of(lob);
  const int qe = (lob >> 20) - 1075;
  const double thr = (LIMO ? limo_thr : 1.44e-6) * pow2d(-qe) * pow2d(-qe);
  const float thr_lo = float_threshold<LIMO, 5>(lob, limo_thr);
  // 60 (Fsum_{k-1} - Fsum_k) as 30 times the doubled values and 60 times the differences of the
  // two faces' centre cells
  Wide<RES> F = {0, 0.0};
#pragma unroll 1
  for (int face = 0; face < 2; face++) {
    const int c0 = i + C0 + face;  // first cell of the face's window
    int code[2];
#pragma unroll 1
    for (int s = 0; s < 2; s++) {
      // the stencil from the left (G+) or from the right (G-), as differences
      Wide<RES> D[ND], last;
#pragma unroll
      for (int q = 0; q <= ND; q++) {
        const Wide<RES> u = wide_cell<RES>(s ? gm : gp, s ? c0 + NC - 1 - q : c0 + q, lob, un);
        if (q) D[q - 1] = lin(1, u, -1, last, un);
        last = u;
      }
      Wide<RES> y;
      code[s] = RES ? float_code<LIMO>(D, thr_lo, un) : -1;
      if (code[s] >= 0) {
        y = {0, 0.0};
        int e[5], sum = 0;
        limited_coefs<LIMO>(code[s], e);
#pragma unroll
        for (int q = 0; q < ND; q++) {  // the cells' coefficients add up to zero
          sum += e[q];
          y = lin(1, y, (LIMO ? (q == 0 ? 10 : 20) : (q == 0 ? -2 : (q == 1 ? 11 : (q == 2 ? 24 : -3)))) - sum, D[q], un);
        }
      } else if constexpr (LIMO) {
        code[s] = limo3_exact(D[0], D[1], thr, un, y);
      } else {
        code[s] = mp5_exact(D[0], D[1], D[2], D[3], thr, un, y);
      }
      F = lin(1, F, face ? -1 : 1, y, un);
      if (face) F = lin(1, F, s ? 60 : -60, D[LIMO ? s : 1 + s], un);
    }
    record<REC>(tp, tm, f0 + i + face, fend, fmod, code[0], code[1]);
  }
  return nearest(F, un, lob);
}

// to_double at a unit below 2^-988: results may be subnormal, and are then whole multiples of
// the last bit.
AMRFD_HD double low_double(const Limbs<5>& F, int lob) {
  if (lob >= kExpUnit << 20) return to_double(F, lob);
  return to_double(F, 1075 << 20) * 0x1p-537 * pow2d((lob >> 20) - 538);
}

// A cell both of whose faces are surely unlimited: a fixed filter of its cells, their largest
// value (with a weight of at least 2) at 110 bits. What rounds, below 2^-110 of that, is far
// below the rounding of any sum the large values are in. The tails ahead of a front, which
// fall off by binades per cell down to underflow, go this way.
template <bool LIMO>
AMRFD_HD double linear_value(line_t gp, line_t gm, int j, int top) {
  constexpr int NC = LIMO ? 4 : 6;
  const int lob = (top - room(5) < 1 ? 1 : top - room(5)) << 20;
  Limbs<5> F = {};
#pragma unroll
  for (int q = 0; q < NC; q++) {
    const int w = LIMO ? (q == 0 ? -10 : (q == 1 ? 60 : (q == 2 ? -30 : -20)))
                       : (q == 0 ? 2 : (q == 1 ? -15 : (q == 2 ? 60 : (q == 3 ? -20 : (q == 4 ? -30 : 3)))));
    int ah, bh;
    unsigned al, bl;
    cell_words(gp, j + q, ah, al);
    cell_words(gm, j + NC - q, bh, bl);
    const Limbs<5> a = limbs_low(ah, al, lob), b = limbs_low(bh, bl, lob);
#pragma unroll
    for (int l = 0; l < 5; l++) F.v[l] += w * (a.v[l] - b.v[l]);
  }
  return low_double(F, lob);
}

// Whether no face can be limited whose cells' exponents are most at most: differences lie below
// 2 x, 30X (30X - 30mp) below 16000 x^2, LIMO3's a^2 + b^2 below 8 x^2.
template <bool LIMO>
AMRFD_HD bool surely_unlimited(int most, double limo_thr) {
  if (!LIMO) return most - 1022 < -17;
  const double x = pow2d(most - 1022);
  return 8.01 * x * x < limo_thr;
}

// Out of line: its registers stay out of the sweeps'.
template <bool LIMO, bool REC>
AMRFD_HD_CALL void exact_cell(line_t gp, line_t gm, int i, double limo_thr, double* out, bool write, unsigned short* tp,
                              unsigned short* tm, int f0, int fend, int fmod) {
  constexpr int NC = LIMO ? 4 : 6;
  const int j = i + (LIMO ? 1 : 0);
  // largest exponents of the window and of the cells in it that the faces' stencils hold
  int most = 0, top = 0;
#pragma unroll
  for (int q = 0; q <= NC; q++) {
    const int a = (cell_hi(gp, j + q) >> 20) & 0x7ff, b = (cell_hi(gm, j + NC - q) >> 20) & 0x7ff, m = a > b ? a : b;
    most = m > most ? m : most;
    if (q < NC) top = m > top ? m : top;
  }
  double r;
  if (surely_unlimited<LIMO>(most, limo_thr)) {
    r = linear_value<LIMO>(gp, gm, j, top);
    record<REC>(tp, tm, f0 + i, fend, fmod, 0, 0);
    record<REC>(tp, tm, f0 + i + 1, fend, fmod, 0, 0);
  } else {
    int lob;
    bool bad;
    const bool whole = window_scale<5, true>(gp, gm, j, NC + 1, lob, bad);
    r = whole ? exact_value<LIMO, REC, false>(gp, gm, i, limo_thr, lob, tp, tm, f0, fend, fmod)
              : exact_value<LIMO, REC, true>(gp, gm, i, limo_thr, lob, tp, tm, f0, fend, fmod);
    if (bad) r = from_words(0x7ff80000, 0u);
  }
  if (write) *out = r;
}

// The cells of a part whose window holds a value that is no whole number of units at the
// scale lob, or is beyond a sweep's range.
template <bool LIMO>
AMRFD_HD unsigned long long partial_cells(line_t gp, line_t gm, int nc, int lob) {
  constexpr int NC = LIMO ? 4 : 6;
  constexpr unsigned long long hit = (2ull << NC) - 1ull;  // the cells i with q in [i, i + NC]
  unsigned long long m = 0ull;
  for (int q = 0; q < nc; q++) {
    bool part = false;
#pragma unroll
    for (int s = 0; s < 2; s++) {
      unsigned a;
      const unsigned k = cell_key<true>(s ? gm : gp, q + (LIMO ? 1 : 0), a);
      part |= (k && k < (unsigned)lob) || (int)(a >> 20) > kExpMax;
    }
    if (part) m |= q < NC ? hit >> (NC - q) : hit << (q - NC);
  }
  return m;
}

// The faces k = 3..plen+3 of one (line, variable) at the scale lob of N limbs, and the
// differences of its cells: see fixed_sweep. Returns the cells left to exact_cell; faces:
// counts those at which the limiter was needed.
template <bool LIMO, bool REC, int N>
AMRFD_HD unsigned long long sweep_part(line_t gp, line_t gm, int plen, double limo_thr, double* out, int ostr,
                                       unsigned long long wmask, unsigned short* tp, unsigned short* tm, int f0,
                                       int fend, int fmod, int lob, int& limited) {
  constexpr int NC = LIMO ? 4 : 6;        // cells of a face's window
  constexpr int C0 = LIMO ? 1 : 0;        // first cell of face 3
  constexpr int NA = NC - 1;
  constexpr int ND = LIMO ? 2 : 4;        // differences of a stencil
  Limbs<N> A[NA];                         // A[n]: the face that lacks n + 1 more cells
  Limbs<N> gl, hl, Fp;                    // last cell's G+, G-; last face
  float P[5], M[5];                       // differences of G+, G-, newest last
  unsigned long long todo = 0ull;
  const int cend = plen + 6 - C0;
  const float thr_lo = float_threshold<LIMO, N>(lob, limo_thr);
#pragma unroll
  for (int l = 0; l < N; l++) {
#pragma unroll
    for (int q = 0; q < NA; q++) A[q].v[l] = 0;
    gl.v[l] = hl.v[l] = Fp.v[l] = 0;
  }
#pragma unroll
  for (int q = 0; q < 5; q++) P[q] = M[q] = 0.0f;
#pragma unroll 1
  for (int c = C0; c < cend; c++) {
    int ph, mh;
    unsigned pl, ml;
    cell_words(gp, c, ph, pl);
    cell_words(gm, c, mh, ml);
    const Limbs<N> x = to_limbs<N>(ph, pl, lob), y = to_limbs<N>(mh, ml, lob);
    Limbs<N> F, dg, dh;
#pragma unroll
    for (int l = 0; l < N; l++) {
      const int g = x.v[l], h = y.v[l];
      dg.v[l] = g - gl.v[l];
      dh.v[l] = h - hl.v[l];
      if constexpr (LIMO) {  // -10 g0 + 50 g1 + 20 g2 + 20 h1 + 50 h2 - 10 h3
        F.v[l] = A[0].v[l] - 10 * h;
        A[0].v[l] = A[1].v[l] + 20 * g + 50 * h;
        A[1].v[l] = A[2].v[l] + 50 * g + 20 * h;
        A[2].v[l] = -10 * g;
      } else {  // 2 g0 - 13 g1 + 47 g2 + 27 g3 - 3 g4 - 3 h1 + 27 h2 + 47 h3 - 13 h4 + 2 h5
        F.v[l] = A[0].v[l] + 2 * h;
        A[0].v[l] = A[1].v[l] - 3 * g - 13 * h;
        A[1].v[l] = A[2].v[l] + 27 * g + 47 * h;
        A[2].v[l] = A[3].v[l] + 47 * g + 27 * h;
        A[3].v[l] = A[4].v[l] - 13 * g - 3 * h;
        A[4].v[l] = 2 * g;
      }
    }
    gl = x;
    hl = y;
    P[0] = P[1]; P[1] = P[2]; P[2] = P[3]; P[3] = P[4]; P[4] = to_float(dg);
    M[0] = M[1]; M[1] = M[2]; M[2] = M[3]; M[3] = M[4]; M[4] = to_float(dh);
    const int i = c - NC - C0;  // the cell left of the face whose last cell is c
    if (i < -1) continue;
    // left-biased value of G+, right-biased of G-
    int cp = 0, cm = 0;
    bool np, nm;
    if constexpr (LIMO) {
      cp = limo3_code_float(P[2], P[3], thr_lo);
      cm = limo3_code_float(M[4], M[3], thr_lo);
      np = cp != 0 && cp != 9;  // not the unlimited value
      nm = cm != 0 && cm != 9;
    } else {
      np = !mp5_accepts(P[0], P[1], P[2], P[3], thr_lo);
      nm = !mp5_accepts(M[4], M[3], M[2], M[1], thr_lo);
    }
    if (np || nm) {
      limited++;
      // both biases together: the two chains of dependent operations overlap
      if constexpr (!LIMO) {
        cp = mp5_code_float(P[0], P[1], P[2], P[3], thr_lo);
        cm = mp5_code_float(M[4], M[3], M[2], M[1], thr_lo);
        if (cp < 0 || cm < 0) {
#pragma unroll 1
          for (int s = 0; s < 2; s++) {
            if ((s ? cm : cp) >= 0) continue;
            const int cd = mp5_code_bounded(s ? M[4] : P[0], s ? M[3] : P[1], s ? M[2] : P[2], s ? M[1] : P[3], thr_lo);
            if (s) cm = cd;
            else cp = cd;
          }
        }
      }
      if (cp < 0 || cm < 0) todo |= i < 0 ? 1ull : 3ull << i;
      // the stencils again, from the left (G+) and from the right (G-)
      int e[5], k[5];
      limited_coefs<LIMO>(cp < 0 ? 0 : cp, e);
      limited_coefs<LIMO>(cm < 0 ? 0 : cm, k);
      long long a[N];
#pragma unroll
      for (int l = 0; l < N; l++) a[l] = 0;
#pragma unroll
      for (int q = 0; q <= ND; q++) {
        int hi;
        unsigned lo;
        cell_words(gp, c - NC + 1 + q, hi, lo);
        const Limbs<N> u = to_limbs<N>(hi, lo, lob);
        cell_words(gm, c - q, hi, lo);
        const Limbs<N> v = to_limbs<N>(hi, lo, lob);
#pragma unroll
        for (int l = 0; l < N; l++) a[l] += (long long)e[q] * u.v[l] + (long long)k[q] * v.v[l];
      }
      add_carried(F, a);
    }
    record<REC>(tp, tm, f0 + i + 1, fend, fmod, cp, cm);
    if (i >= 0) {
      if (wmask & 1ull) *out = to_double(Fp, F, lob);
      out += ostr;
      wmask >>= 1;
    }
    Fp = F;
  }
  return todo;
}

// The cells of a part whose faces are all surely unlimited (FIT: and whose exponents span
// at most 57 binades, at a scale of 2^-988 or more): their differences as a fixed filter (linear_value) by transposed sums, without the face fluxes and FP32 differences of
// sweep_part.
template <bool LIMO, bool REC, bool FIT>
AMRFD_HD void linear_part(line_t gp, line_t gm, int plen, double* out, int ostr, unsigned long long wmask,
                          unsigned short* tp, unsigned short* tm, int f0, int fend, int fmod, int lob) {
  constexpr int NC = LIMO ? 4 : 6;
  constexpr int C0 = LIMO ? 1 : 0;
  Limbs<5> A[NC];  // A[n]: the cell that lacks n + 1 more
#pragma unroll
  for (int q = 0; q < NC; q++) A[q] = Limbs<5>{};
#pragma unroll 1
  for (int i = -NC; i < plen; i++) {  // the cell whose last one this is
    int ph, mh;
    unsigned pl, ml;
    cell_words(gp, i + NC + C0, ph, pl);
    cell_words(gm, i + NC + C0, mh, ml);
    const Limbs<5> x = FIT ? limbs_wide<true>(ph, pl, lob) : limbs_low(ph, pl, lob);
    const Limbs<5> y = FIT ? limbs_wide<true>(mh, ml, lob) : limbs_low(mh, ml, lob);
    Limbs<5> F;
#pragma unroll
    for (int l = 0; l < 5; l++) {
      const int g = x.v[l], h = y.v[l];
      if constexpr (LIMO) {  // -10 g0 + 60 g1 - 30 g2 - 20 g3 + 20 h1 + 30 h2 - 60 h3 + 10 h4
        F.v[l] = A[0].v[l] + 10 * h;
        A[0].v[l] = A[1].v[l] - 20 * g - 60 * h;
        A[1].v[l] = A[2].v[l] - 30 * g + 30 * h;
        A[2].v[l] = A[3].v[l] + 60 * g + 20 * h;
        A[3].v[l] = -10 * g;
      } else {  // 2 g0 - 15 g1 + 60 g2 - 20 g3 - 30 g4 + 3 g5 - 3 h1 + 30 h2 + 20 h3 - 60 h4 + 15 h5 - 2 h6
        F.v[l] = A[0].v[l] - 2 * h;
        A[0].v[l] = A[1].v[l] + 3 * g + 15 * h;
        A[1].v[l] = A[2].v[l] - 30 * g - 60 * h;
        A[2].v[l] = A[3].v[l] - 20 * g + 20 * h;
        A[3].v[l] = A[4].v[l] + 60 * g + 30 * h;
        A[4].v[l] = A[5].v[l] - 15 * g - 3 * h;
        A[5].v[l] = 2 * g;
      }
    }
    if (i < -1) continue;
    record<REC>(tp, tm, f0 + i + 1, fend, fmod, 0, 0);
    if (i < 0) continue;
    if (wmask & 1ull) *out = FIT ? to_double(F, lob) : low_double(F, lob);
    out += ostr;
    wmask >>= 1;
  }
}

// fixed_sweep of a part with five limbs: the cells left to exact_cell, and the faces limited.
// Out of line: most warps hold none, and its registers stay out of the other sweeps'.
// What comes here is mostly tails ahead of a front: in the MHD blast eight of 27 (variable,
// direction) pairs, through the whole box. Hence the filter where no face can be limited, and
// the cuts that keep cells out of exact_cell: a part over 57 binades goes in halves, one of
// which, if it does not fit, in quarters (at once from 88 binades on: level with 76 and 110).
// 256^3 flux launch in steps 1, 10, 24 and 80: 10.3, 13.0, 19.8 and 14.2 ms with plain five-limb
// sweeps and each cell over 110 bits by itself, 10.2, 10.8, 12.7 and 10.7 with both; halves
// only 12.6 at step 13, halves or quarters for the whole part 11.5, this 11.2.
struct Wide5 {
  unsigned long long todo;
  int limited;
};
template <bool LIMO, bool REC>
AMRFD_HD_CALL Wide5 wide_sweep(line_t gp, line_t gm, int plen, double limo_thr, double* out, int ostr,
                               unsigned long long wmask, unsigned short* tp, unsigned short* tm, int f0, int fend,
                               int fmod, Span span, unsigned lanes) {
  constexpr int C0 = LIMO ? 1 : 0;
  constexpr int NC = LIMO ? 4 : 6;
  unsigned long long todo = 0ull;
  int lob, limited = 0;
  // ahead of a front a component falls off by about three binades a cell: 66 over the cells of
  // a part of 16, 42 over its half's
  const int range = span.mn + 1u ? (int)(span.mx >> 20) - (int)((span.mn + 1u) >> 20) : 0;
  const int least = AMRFD_ANY(lanes, plen < 8) ? 4 : (AMRFD_ANY(lanes, plen < 16) ? 2 : 1);
  int most = 4, size;
  if (AMRFD_ANY(lanes, range > 57)) most = AMRFD_ANY(lanes, range > 88) ? 1 : 2;
  most = most < least ? least : most;
#pragma unroll 1
  for (int q = 0; q < 4; q += size) {  // size quarters from the q-th on
    size = q & 1 ? 1 : most;
    int p0, len;
    line_t p, m;
    bool bad, fits, weak;
    for (;;) {
      p0 = q * plen / 4;
      len = (q + size) * plen / 4 - p0;
      p = line_at(gp, p0);
      m = line_at(gm, p0);
      if (size < 4) span = window_span<false>(p, m, C0, len + NC);
      weak = surely_unlimited<LIMO>((int)(span.mx >> 20), limo_thr);
      fits = weak ? span_scale<5, 0, 1>(span, lob, bad) : span_scale<5>(span, lob, bad);
      if (size == least || !AMRFD_ANY(lanes, !fits)) break;
      size >>= 1;
    }
    double* o = out + (long long)p0 * ostr;
    const int fe = q + size < 4 && f0 + p0 + len + 1 < fend ? f0 + p0 + len + 1 : fend;
    const bool linear = !AMRFD_ANY(lanes, !weak);
    const bool low = linear && lob < kExpUnit << 20 && span.mx;  // (zeros fit any scale)
    if (linear && !AMRFD_ANY(lanes, !fits || low)) {
      linear_part<LIMO, REC, true>(p, m, len, o, ostr, wmask >> p0, tp, tm, f0 + p0, fe, fmod, lob);
      continue;
    }
    if (!linear) fits = span_scale<5>(span, lob, bad);
    const unsigned long long cells = len < 64 ? (1ull << len) - 1ull : ~0ull;
    unsigned long long part = 0ull;
    if (!fits && (low || !window_scale<5, true>(p, m, C0, len + NC, lob, bad)))
      part = partial_cells<LIMO>(p, m, len + NC, lob) & cells;
    if (linear)
      linear_part<LIMO, REC, false>(p, m, len, o, ostr, wmask >> p0, tp, tm, f0 + p0, fe, fmod, lob);
    else if (AMRFD_ANY(lanes, part != cells))
      part |= sweep_part<LIMO, REC, 5>(p, m, len, limo_thr, o, ostr, wmask >> p0, tp, tm, f0 + p0, fe, fmod, lob,
                                       limited) & cells;
    todo |= part << p0;
  }
  return {todo, limited};
}

// One (line, variable): the faces k = 3..plen+3 of the line's extended index (cell j = k-1
// left of face k) and 60 (Fsum_{k-1} - Fsum_k) of its plen <= 64 cells, Fsum = G+_{k-1} +
// G-_k + (Y+_k + Y-_k)/2, stored to out[i ostr] where wmask has its bit (the factor
// 1/(120 dx) is applied by the stage combination). Every lane in `lanes` must call this: the
// votes on the number of limbs, before any loop over faces, wait for all of them (parts may
// differ in length). REC records per face and bias the code of the piece the limiter took:
// face k at index f0 + k - 3 if below fend (face fmod as face 0). Returns the number of
// faces at which the lane's limiter was needed.
// A cell enters the partial sums of the faces it belongs to when it is read (a transposed
// filter), so that only those sums and the last cell stay in registers; the limiter's
// correction of a face reads its stencil again. What FP32 cannot decide is left to
// exact_cell after the loop, which keeps that code's registers out of it.
template <bool LIMO, bool REC>
AMRFD_HD int fixed_sweep(line_t gp, line_t gm, int plen, double limo_thr, double* out, int ostr,
                         unsigned long long wmask, unsigned short* tp, unsigned short* tm, int f0, int fend, int fmod,
                         unsigned lanes) {
  constexpr int C0 = LIMO ? 1 : 0;
  constexpr int NC = LIMO ? 4 : 6;
  const int nc = plen + NC;
  int lob, limited = 0;
  bool bad;
  const Span span = window_span<false>(gp, gm, C0, nc);
  const unsigned long long all = plen < 64 ? (1ull << plen) - 1ull : ~0ull;
  unsigned long long todo;
  if (!AMRFD_ANY(lanes, !span_scale<3>(span, lob, bad))) {
    todo = sweep_part<LIMO, REC, 3>(gp, gm, plen, limo_thr, out, ostr, wmask, tp, tm, f0, fend, fmod, lob, limited);
  } else if (!AMRFD_ANY(lanes, !span_scale<4>(span, lob, bad))) {
    todo = sweep_part<LIMO, REC, 4>(gp, gm, plen, limo_thr, out, ostr, wmask, tp, tm, f0, fend, fmod, lob, limited);
  } else {
    const Wide5 w = wide_sweep<LIMO, REC>(gp, gm, plen, limo_thr, out, ostr, wmask, tp, tm, f0, fend, fmod, span, lanes);
    todo = w.todo;
    limited = w.limited;
  }
  todo &= all;
  while (todo) {
#ifdef __CUDACC__
    const int i = __ffsll((long long)todo) - 1;
#else
    const int i = __builtin_ctzll(todo);
#endif
    todo &= todo - 1ull;
    exact_cell<LIMO, REC>(gp, gm, i, limo_thr, out + (long long)i * ostr, (wmask >> i) & 1ull, tp, tm, f0, fend, fmod);
  }
  return limited;
}

// The stage combination's weight of a sweep's differences, b dt / (120 dx): one rounding where
// dx is a power of two. Its error against the extended-precision step drowns in the state's
// own rounding (512-cell Sod step: 1.38e-18 of the state with three roundings, 1.41e-18 with
// this, 1.42e-18 with the weight in two terms, which costs 6 % of a step).
AMRFD_HD double stage_weight(double dtb, double dx) { return dtb / (120.0 * dx); }

// ------------------------------------------------------------------- adjoint
// Transposed sweep of one (line, variable), in the same arithmetic: with the pieces of the
// forward pass fixed, 60 Fsum_k is a whole combination of the G+- cells, so 60 times the
// gradient with respect to a cell is a whole combination of the differences gF_k of the
// upstream gradient over the faces within reach. g: the upstream gradient, g[r] at cell
// s0 - 3 + r for r = 0..slen+5; faces kb..ke (relative to s0, -2 <= kb, ke <= slen + 2);
// tp, tm: the recorded codes of face k at index k + fofs, wrapped into [0, n) on a periodic
// line (wrap). The gradients of cells lo..hi (relative to s0) go to gp, gm[cell + 5], those
// that no face reaches as zeros.
// LIMO3's codes inside the blend band stand for the nearer half.
// A cell's gradient sums up to five faces' differences (twice the largest value) with
// coefficients of magnitude 2140 together (the largest of each stencil cell over the
// limiter's pieces: 320, 750, 630, 320, 120), less than 2^13 times the largest value.
constexpr int kAdjHead = 4;

template <bool LIMO>
AMRFD_HD int adjoint_code(int code) {
  if (!LIMO) return code;
  const int mode = (code >> 3) & 3;
  return mode == 0 || mode == 2 ? 0 : (code & 7) | (1 << 3);
}

struct TapeLine {
  const unsigned short *tp, *tm;
  int fofs, n;
  bool wrap;
};
AMRFD_HD int tape_index(const TapeLine& t, int k) {
  const int f = k + t.fofs;
  return t.wrap ? (f < 0 ? f + t.n : (f >= t.n ? f - t.n : f)) : f;
}

// One cell by itself (relative to s0), at the scale of the seven values that reach it; what
// its units leave over (RES) is carried as in exact_value.
template <bool LIMO, bool RES>
AMRFD_HD void adjoint_values(line_t g, const TapeLine& t, int kb, int ke, int cell, int lob, double v[2]) {
  constexpr int NS = LIMO ? 3 : 5;         // cells of a stencil
  constexpr int off = LIMO ? 2 : 3;        // G+ stencil of face k: cells k - off ..
  const Unit un = unit_of(lob);
  const int k0 = cell - off + 1 > kb ? cell - off + 1 : kb, k1 = cell + off < ke ? cell + off : ke;
  Wide<RES> F[2] = {{0, 0.0}, {0, 0.0}}, b = wide_cell<RES>(g, k0 + 2, lob, un);
#pragma unroll 1
  for (int k = k0; k <= k1; k++) {
    const Wide<RES> a = wide_cell<RES>(g, k + 3, lob, un);
    const __int128 h = a.h - b.h;
    const double r = RES && (any_bits(a.r) || any_bits(b.r)) ? a.r - b.r : 0.0;
    b = a;
    if (h == 0 && !any_bits(r)) continue;  // no code where the gradient does not reach
    const int f = tape_index(t, k);
#pragma unroll
    for (int s = 0; s < 2; s++) {
      // the face's stencil cell this one is: G+ cells k - off .., G- counted from the right
      const int q = s ? k + off - 1 - cell : cell + off - k;
      if (q < 0 || q >= NS) continue;
      int e[5];
      limited_coefs<LIMO>(adjoint_code<LIMO>(s ? t.tm[f] : t.tp[f]), e);
      const int w = LIMO ? (q == 0 ? -10 : (q == 1 ? 50 : 20))
                         : (q == 0 ? 2 : (q == 1 ? -13 : (q == 2 ? 47 : (q == 3 ? 27 : -3))));
      const int c = w + (q == 0 ? e[0] : (q == 1 ? e[1] : (q == 2 ? e[2] : (q == 3 ? e[3] : e[4]))));
      F[s].h += h * c;
      if (RES && any_bits(r)) F[s].r = fma((double)c, r, F[s].r);
    }
  }
#pragma unroll
  for (int s = 0; s < 2; s++) {
    if (RES) carry_units(F[s], un);
    v[s] = nearest(F[s], un, lob);
  }
}
template <bool LIMO>
AMRFD_HD_CALL void adjoint_cell(line_t g, TapeLine t, int kb, int ke, int cell, double* gp, double* gm) {
  int lob;
  bool bad;
  const int r0 = cell < 0 ? 0 : cell, r1 = cell + 6;  // g[r] of cells cell-3 .. cell+3, those there are
  const int last = ke + 3;
  double v[2];
  if (window_scale<5, true, kAdjHead>(g, g, r0, (r1 < last ? r1 : last) - r0 + 1, lob, bad))
    adjoint_values<LIMO, false>(g, t, kb, ke, cell, lob, v);
  else adjoint_values<LIMO, true>(g, t, kb, ke, cell, lob, v);
  const double nan = from_words(0x7ff80000, 0u);
  gp[cell + 5] = bad ? nan : v[0];
  gm[cell + 5] = bad ? nan : v[1];
}

template <int N>
AMRFD_HD double gradient(const Limbs<N>& d, int lob) {
  if constexpr (N >= 4) return to_double(d, lob);
  else return to_double(d, Limbs<N>{}, lob);
}

template <bool LIMO, int N>
AMRFD_HD void adjoint_part(line_t g, const TapeLine& t, int kb, int ke, int lo, int hi, int lob, double* gp,
                           double* gm) {
  constexpr int NS = LIMO ? 3 : 5;
  constexpr int off = LIMO ? 2 : 3;
  Limbs<N> P[NS], M[NS], last;             // partial sums of the stencils' cells, leftmost first
  const Limbs<N> zero = {};
#pragma unroll
  for (int q = 0; q < NS; q++) P[q] = M[q] = zero;
  int h;
  unsigned w;
  cell_words(g, kb + 2, h, w);
  last = to_limbs<N>(h, w, lob);
  for (int c = lo; c <= kb - off; c++) {   // ghosts that no face reaches
    gm[c + 5] = 0.0;
    if (c < kb - off) gp[c + 5] = 0.0;
  }
  const int kend = hi + off;               // the face that completes cell hi's G+
#pragma unroll 1
  for (int k = kb; k <= kend; k++) {
    if (k <= ke) {
      cell_words(g, k + 3, h, w);
      const Limbs<N> x = to_limbs<N>(h, w, lob);
      Limbs<N> d;
#pragma unroll
      for (int l = 0; l < N; l++) d.v[l] = x.v[l] - last.v[l];
      last = x;
      int any = 0;
#pragma unroll
      for (int l = 0; l < N; l++) any |= d.v[l];
      int cp = 0, cm = 0;
      if (any) {  // a face the gradient does not reach may hold no code (passive blocks)
        const int f = tape_index(t, k);
        cp = adjoint_code<LIMO>(t.tp[f]);
        cm = adjoint_code<LIMO>(t.tm[f]);
      }
#pragma unroll
      for (int l = 0; l < N; l++) {
        const int x0 = d.v[l];
        if constexpr (LIMO) {
          P[0].v[l] -= 10 * x0; P[1].v[l] += 50 * x0; P[2].v[l] += 20 * x0;
          M[0].v[l] += 20 * x0; M[1].v[l] += 50 * x0; M[2].v[l] -= 10 * x0;
        } else {
          P[0].v[l] += 2 * x0; P[1].v[l] -= 13 * x0; P[2].v[l] += 47 * x0; P[3].v[l] += 27 * x0; P[4].v[l] -= 3 * x0;
          M[0].v[l] -= 3 * x0; M[1].v[l] += 27 * x0; M[2].v[l] += 47 * x0; M[3].v[l] -= 13 * x0; M[4].v[l] += 2 * x0;
        }
      }
      if ((cp | cm) > 0) {
        int e[5], m[5];
        limited_coefs<LIMO>(cp, e);
        limited_coefs<LIMO>(cm, m);
#pragma unroll
        for (int q = 0; q < NS; q++) {
          long long x0[N], x1[N];
#pragma unroll
          for (int l = 0; l < N; l++) {
            x0[l] = (long long)e[q] * d.v[l];
            x1[l] = (long long)m[NS - 1 - q] * d.v[l];
          }
          add_carried(P[q], x0);
          add_carried(M[q], x1);
        }
      }
    }
    // G+ of cell k - off and G- of the cell after it are complete
    const int c = k - off;
    if (c >= lo) gp[c + 5] = gradient(P[0], lob);
    if (c + 1 >= lo && c + 1 <= hi) gm[c + 6] = gradient(M[0], lob);
#pragma unroll
    for (int q = 0; q < NS - 1; q++) {
      P[q] = P[q + 1];
      M[q] = M[q + 1];
    }
    P[NS - 1] = M[NS - 1] = zero;
  }
}

// Four limbs first (31 binades): an upstream gradient of random numbers spans more than the 9
// that three would leave in nearly every warp, and the fallback's five limbs and two
// conversions of 128 bits a cell then cost what the integers save (512^2 MHD, adjoint of one
// step: 1.68 ms with three limbs, 1.48 with four, about 1.75 with the FP64 transposition).
template <bool LIMO>
AMRFD_HD void adjoint_sweep(line_t g, int slen, const TapeLine& t, int kb, int ke, int lo, int hi, double* gp,
                            double* gm, unsigned lanes) {
  int lob;
  bool bad;
  const bool narrow = window_scale<4, false, kAdjHead>(g, g, 0, slen + 6, lob, bad);
  if (!AMRFD_ANY(lanes, !narrow)) {
    adjoint_part<LIMO, 4>(g, t, kb, ke, lo, hi, lob, gp, gm);
    return;
  }
  if (window_scale<5, true, kAdjHead>(g, g, 0, slen + 6, lob, bad)) {
    adjoint_part<LIMO, 5>(g, t, kb, ke, lo, hi, lob, gp, gm);
  } else {
    for (int c = lo; c <= hi; c++) adjoint_cell<LIMO>(g, t, kb, ke, c, gp, gm);
  }
}

}  // namespace amrfd
