// tde_fx.cuh -- 64-bit fixed-point arithmetic for the tabulated EOS: log2, exp2,
// interpolation and the cell solve on the integer pipe.
//
// Why: the inversion is arithmetic on logarithms, whose absolute precision is
// what counts, and sm_103a issues one FP64 warp instruction per 16 cycles and SM
// against about 32 integer ones.  In FP64 an inversion takes about 100 such
// slots (1600 cycles per warp); here it is a few hundred integer instructions
// and no FP64 at all: 2^24 inversions of (T, P, cs^2) with densities and energies
// scattered over the 256 x 256 table went from 3.10 ms to 0.63 ms (1.06 TB/s of
// input and output), the learned-guess form on 6 million from 1.86 to 0.78 ms (0.72 since), a
// step of the 8.4 M-cell star mesh from 25.6 to 21.4 ms.  A fixed-point logarithm of 55 fraction bits resolves
// 2.8e-17 in log2, an FP64 one of size 40 (log10 of size 12) only 7e-15, so the
// results are nearer to the exact ones than the FP64 form's.
//
// Format: Q55 in a signed 64-bit integer, in log2 units (values in (-128, 128));
// weights and fractions are unsigned Q64.  Every step is a fixed sequence of
// integer operations, so all kernels (and the host) get the same bits.
//
// Methods: log2 by a table of reciprocals c_j ~ 1/m of 10 bits (the product of
// the 53-bit significand with c_j is exact in 64 bits) and the series of
// ln(1 + r), |r| < 2^-8.4; exp2 by a table of 2^((j + 1/2)/256) and the series
// of 2^g, |g| <= 2^-9 (both after the table-driven scheme of P. T. Tang, ACM
// TOMS 15 and 16); the quotient from the FP32 reciprocal refined to second
// order.
#pragma once
#include <stdint.h>
#include <string.h>

#ifdef __CUDACC__
#define FX_HD __host__ __device__ __forceinline__
#else
#define FX_HD inline
#endif

namespace tde {

typedef long long fx;              // Q55, log2 units
typedef unsigned long long ufx;    // fractions, Q64

constexpr int FX_Q = 55;
constexpr fx FX_ONE = 1LL << FX_Q;
constexpr fx FX_BAD = (fx)0x8000000000000000ull;   // a value outside the format
constexpr fx FX_SAT = 128 * (FX_ONE - 1);          // |log2| of what lies beyond every table
constexpr double FX_MAX_LOG10 = 38.0;              // |log10| of a table entry the format takes
constexpr unsigned long long FX_LOG2_10 = 0xD49A784BCD1B8AFEull;   // log2(10), Q62

struct FxMath {
  fx lg[256];                    // -log2(c_j / 1024), Q55
  unsigned long long ex[256];    // 2^((j + 1/2) / 256), Q62
  unsigned c[256];               // 1024 / (1 + (j + 1/2) / 256), rounded
};

FX_HD fx fx_bits(double x) {
  fx b;
#ifdef __CUDA_ARCH__
  // opaque: a sign or magnitude mask of it must not become an FP64 instruction
  asm("mov.b64 %0, %1;" : "=l"(b) : "d"(x));
#else
  memcpy(&b, &x, 8);
#endif
  return b;
}
FX_HD double fx_double(fx b) {
#ifdef __CUDA_ARCH__
  return __longlong_as_double(b);
#else
  double x;
  memcpy(&x, &b, 8);
  return x;
#endif
}
FX_HD ufx fx_umulhi(ufx a, ufx b) {
#ifdef __CUDA_ARCH__
  return __umul64hi(a, b);
#else
  return (ufx)(((unsigned __int128)a * b) >> 64);
#endif
}
FX_HD fx fx_mulhi(fx a, fx b) {
#ifdef __CUDA_ARCH__
  return __mul64hi(a, b);
#else
  return (fx)(((__int128)a * b) >> 64);
#endif
}
FX_HD int fx_mulhi32(int a, int b) {
#ifdef __CUDA_ARCH__
  return __mulhi(a, b);
#else
  return (int)(((fx)a * b) >> 32);
#endif
}
FX_HD int fx_clz(ufx a) {
#ifdef __CUDA_ARCH__
  return __clzll((fx)a);
#else
  return __builtin_clzll(a);
#endif
}

// log10 value v (a table entry, FP64, below FX_MAX_LOG10 in magnitude) in Q55 log2 units,
// rounded to nearest
FX_HD fx fx_of_log10_in(double v) {
  const fx b = fx_bits(v), a = b & 0x7fffffffffffffffLL;
  const int e = (int)(a >> 52);   // 2^(e - 1023) <= |v|; subnormals round to 0 below
  const ufx m = ((ufx)(a & 0xfffffffffffffLL) | 0x10000000000000ull) << 11;
  // |v| log2(10) = m 2^(e - 1086) LOG2_10 2^-62 = h 2^(e - 1084), wanted times 2^55
  const ufx h = fx_umulhi(m, FX_LOG2_10);
  const int s = 1029 - e;         // >= 1 for |v| < 64
  const fx q = s < 64 ? (fx)((h >> (s & 63)) + ((h >> ((s - 1) & 63)) & 1)) : 0;
  return b < 0 ? -q : q;
}
// FX_BAD if it is not (or not a number)
FX_HD fx fx_of_log10(double v) {
  return (fx_bits(v) & 0x7fffffffffffffffLL) >= fx_bits(FX_MAX_LOG10) ? FX_BAD : fx_of_log10_in(v);
}

// likewise, but the end of the range on its side
FX_HD fx fx_of_log10_sat(double v) {
  const fx b = fx_bits(v);
  return (b & 0x7fffffffffffffffLL) >= fx_bits(FX_MAX_LOG10) ? (b < 0 ? -FX_SAT : FX_SAT) : fx_of_log10_in(v);
}

// log2 of x > 0 in Q55.  x above 2^127 (or infinite, or a positive NaN)
// saturates at FX_SAT, x below 2^-127 (or not positive) at -FX_SAT.
FX_HD fx fx_log2(const FxMath *__restrict__ mt, double x) {
  const fx b = fx_bits(x);
  const int k = (int)(b >> 52) - 1023;   // floor(log2 x); negative x: far below -127
  if (k < -127) return -FX_SAT;
  if (k > 126) return FX_SAT;
  const fx mant = b & 0xfffffffffffffLL;
  const int j = (int)(mant >> 44);
  // r = m c - 1, exact in Q62: |r| <= 2^-9 + 2^-10
  const fx R = (fx)((ufx)(mant | 0x10000000000000LL) * mt->c[j]) - (1LL << 62);
  const int p = (int)(R >> 23);          // 2^7 r in Q32 (r in Q39)
  const int lo = (int)(R & 0x7fffff);
  // ln(1 + r) = r - r^2/2 + r^2 (r s), s = 1/3 - r/4 + r^2/5 - r^3/6 (Q32; the
  // next term, r^7/7, is below 2^-61)
  int s = 52429 + fx_mulhi32(p, -341);   // 2^32 / (5 2^14), 2^32 / (6 2^21)
  s = -8388608 + fx_mulhi32(p, s);       // 2^32 / (4 2^7)
  s = 1431655765 + fx_mulhi32(p, s);     // 2^32 / 3
  const int rs = fx_mulhi32(p, s);       // r s in Q39
  const fx sq = (fx)p * p + (((fx)p * lo) >> 22);   // r^2 in Q78
  const fx ln = R - (sq >> 17) + (((fx)(int)(sq >> 32) * rs) >> 23);   // Q62
  // times log2(e) = 1 + 0.4427: Q62 -> Q55
  const fx l2 = ln + fx_mulhi(ln, 0x71547652B82FE177LL);   // (log2(e) - 1) in Q64
  return ((fx)k << FX_Q) + mt->lg[j] + ((l2 + 64) >> 7);
}

// 2^L, correctly rounded but for about 2^-55 relative
FX_HD double fx_exp2(const FxMath *__restrict__ mt, fx L) {
  const int n = (int)(L >> FX_Q), j = (int)(L >> 47) & 255;
  const fx g = (L & ((1LL << 47) - 1)) - (1LL << 46);   // Q55, |g| <= 2^-9
  const int q = (int)(g >> 15);                         // 2^8 g in Q32 (g in Q40)
  // 2^g = 1 + g (c1 + g (c2 + g (c3 + g (c4 + g c5)))), c_k = ln(2)^k / k!
  int h = 161365 + fx_mulhi32(q, 87);    // c4 2^32 / 2^8, c5 2^32 / 2^16
  h = 238388332 + fx_mulhi32(q, h);      // c3 2^32
  const fx h2 = 0x0F5FDEFFC162C754LL + (((fx)q * h) >> 10);              // c2 + .., Q62
  const fx g71 = g << 16;                                                // g in Q71
  const fx m1 = 0x2C5C85FDF473DE6BLL + (fx_mulhi(g71, h2) >> 7);         // c1 + .., Q62
  const fx m2 = fx_mulhi(g71, m1);                                       // 2^g - 1, Q69
  const ufx T = mt->ex[j];
  const ufx V = T + (ufx)(fx_mulhi((fx)T, m2 << 3) >> 8);                // Q62, in [1, 2]
  return fx_double(((fx)(n + 1022) << 52) + (fx)((V + 512) >> 10));
}

// a + w (b - a), w in Q64
FX_HD fx fx_lerp(fx a, fx b, ufx w) { return a + (fx_mulhi(b - a, (fx)(w >> 1)) << 1); }

// the fraction num / den in Q64, 0 <= num < den (< 1; error below 2^-50)
FX_HD ufx fx_frac(fx num, fx den) {
  const int z = fx_clz((ufx)den);
  const ufx D = (ufx)den << z, N = (ufx)num << z;   // D in [1/2, 1) of 2^64
  // FP32 reciprocal of D's 24 leading bits: R0 in Q23, (1, 2)
  float rf;
#ifdef __CUDA_ARCH__
  rf = __frcp_rn(__uint_as_float(0x3f000000u | ((unsigned)(D >> 40) & 0x7fffffu)));
  const unsigned rb = __float_as_uint(fminf(rf, 1.99999988f));
#else
  const unsigned db = 0x3f000000u | ((unsigned)(D >> 40) & 0x7fffffu);
  float df;
  memcpy(&df, &db, 4);
  rf = 1.0f / df;
  if (rf > 1.99999988f) rf = 1.99999988f;
  unsigned rb;
  memcpy(&rb, &rf, 4);
#endif
  const unsigned R = (rb & 0x7fffffu) | 0x800000u;
  // 1/D = R (1 + e + e^2), e = 1 - D R in Q55, |e| < 2^-21
  const fx e = FX_ONE - (fx)((ufx)(unsigned)(D >> 32) * R + (((ufx)(unsigned)D * R) >> 32));
  const int e53 = (int)(e >> 2);
  const fx c = e + (((fx)e53 * e53) >> 51);
  const fx q = (fx)((ufx)(unsigned)(N >> 32) * R + (((ufx)(unsigned)N * R) >> 32));   // N R, Q55
  fx s = q + (((fx)(int)(q >> 26) * (fx)(int)(c >> 2)) >> 27);   // Q29 x Q53
  s = s < 0 ? 0 : (s > FX_ONE - 1 ? FX_ONE - 1 : s);
  return (ufx)s << 9;
}

// ------------------------------- FP64 reciprocal and square roots by integers ----
//
// The same trade as above for the refined reciprocals of the hydro kernels: an
// FP32 seed of the significand (MUFU), a residual exact in 64 bits and a
// second-order correction give the reciprocal within 0.51 ulp and the roots
// within 0.52 (0.501, 0.516 and 0.514 over 4 M random arguments) in about 40
// integer instructions (20 cycles per warp and SM), where the FP64 refinement
// took 3 slots (48 cycles) for 1/d, 7 for sqrt(a/b), 5 for 1/sqrt(t).  For normal
// arguments whose result is normal; *_ok says so from the exponent fields.

FX_HD unsigned fx_seed(float x) {   // x in (1/2, 1], Q24, below 1
#ifdef __CUDA_ARCH__
  return (__float_as_uint(fminf(x, 0.99999994f)) & 0x7fffffu) | 0x800000u;
#else
  if (x > 0.99999994f) x = 0.99999994f;
  unsigned b;
  memcpy(&b, &x, 4);
  return (b & 0x7fffffu) | 0x800000u;
#endif
}
FX_HD float fx_float(unsigned b) {
#ifdef __CUDA_ARCH__
  return __uint_as_float(b);
#else
  float x;
  memcpy(&x, &b, 4);
  return x;
#endif
}
FX_HD float fx_rcpf(float x) {
#ifdef __CUDA_ARCH__
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
#else
  return 1.0f / x;
#endif
}
FX_HD float fx_rsqrtf(float x) {
#ifdef __CUDA_ARCH__
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
#else
  return 1.0f / __builtin_sqrtf(x);
#endif
}

// 1/d: the exponent field must be in [1, 2043]
FX_HD bool fx_rcp_ok(fx b) { return ((unsigned)(b >> 52) & 0x7ff) - 1u < 2043u; }
FX_HD double fx_rcp(fx b) {
  const ufx m = ((ufx)b & 0xfffffffffffffull) | 0x10000000000000ull;   // 1.f in Q52
  const unsigned R = fx_seed(fx_rcpf(fx_float(0x3f800000u | ((unsigned)(b >> 29) & 0x7fffffu))));
  const fx e = -(fx)(m * R);                // 1 - m R in Q76 (mod 2^64: |e| < 2^-21)
  const int eh = (int)(e >> 24);            // Q52
  // 1/m = R (1 + e + e^2): e's low part and e^2 (Q72) in Q76
  const ufx lo = (ufx)(e & 0xffffff) + ((ufx)(unsigned)fx_mulhi32(eh, eh) << 4);
  const ufx r = ((ufx)R << 39) + (ufx)(((fx)(int)R * eh) >> 13) + ((lo * R) >> 37);   // Q63
  const unsigned E = (unsigned)(b >> 52) & 0x7ff;
  return fx_double((fx)((ufx)(2044u - E) << 52) + (fx)((r + 512) >> 10) | (b & (fx)0x8000000000000000ull));
}

// 1/sqrt of V in Q62, 1 <= V < 4: Q63, in (1/2, 1]
FX_HD ufx fx_rsqrt62(ufx V) {
  // FP32 of V from its leading bits: [1, 2) or [2, 4)
  const unsigned top = (unsigned)(V >> 63);
  const float f = fx_float((0x3f800000u + (top << 23)) | ((unsigned)(V >> (39 + top)) & 0x7fffffu));
  const unsigned Y = fx_seed(fx_rsqrtf(f));
  const fx e = (1LL << 62) - (fx)fx_umulhi(V, (ufx)Y * Y << 16);   // 1 - V Y^2, Q62
  const int eh = (int)(e >> 10);                                   // Q52
  const fx c = e + ((3 * (fx)fx_mulhi32(eh, eh)) >> 12);           // e/2 + 3 e^2/8, Q63
  return ((ufx)Y << 39) + (ufx)(((c >> 4) * (fx)(int)Y) >> 20);
}

// sqrt(a / b) for positive normal a, b
FX_HD bool fx_pos_ok(fx b) { return (unsigned)(b >> 52) - 1u < 2046u; }
FX_HD double fx_sqrt_ratio(fx a, fx b) {
  const ufx A = (((ufx)a & 0xfffffffffffffull) | 0x10000000000000ull) << 11;   // Q63, [1, 2)
  const ufx B = (((ufx)b & 0xfffffffffffffull) | 0x10000000000000ull) << 11;
  const int ea = (int)(a >> 52) - 1023, eb = (int)(b >> 52) - 1023;
  // a b = t 2^E, t in [1, 4), E even
  const ufx p = fx_umulhi(A, B);            // Q62, [1, 4)
  const int odd = (ea + eb) & 1, two = (int)(p >> 63);
  // odd exponent: t = 2 p (p < 2) or p / 2 with E + 2 (p >= 2)
  const ufx V = odd ? (two ? p >> 1 : p << 1) : p;
  const int E = ea + eb - odd + (odd & two ? 2 : 0);
  // sqrt(a / b) = A 2^ea / sqrt(a b)
  ufx C = fx_umulhi(A, fx_rsqrt62(V));      // Q62, in (1/2, 2)
  int ex = ea - E / 2;
  if (!(C >> 62)) { C <<= 1; --ex; }        // Q62, [1, 2)
  return fx_double(((fx)(ex + 1022) << 52) + (fx)((C + 512) >> 10));
}

// 1/sqrt(t) for positive normal t
FX_HD double fx_rsqrt(fx t) {
  const ufx T = (((ufx)t & 0xfffffffffffffull) | 0x10000000000000ull) << 10;   // Q62, [1, 2)
  const int e = (int)(t >> 52) - 1023, odd = e & 1;
  const ufx y = fx_rsqrt62(T << odd);       // Q63, (1/2, 1]
  return fx_double(((fx)(1021 - (e - odd) / 2) << 52) + (fx)((y + 512) >> 10));
}

// ------------------------------------------- sums of neighbours by integers ----
//
// The multigrid's second differences: significands aligned to the largest exponent of the
// values, summed exactly, and the sum rounded to FP64.  Not where every value is below
// 2^-950, nor from 2^1018 up (where a sum may overflow, or a value is infinite or not a
// number): the sums are taken in FP64 there.

FX_HD bool fx_sum_ok(int emax) { return emax >= 70 && emax <= 2040; }   // exponent field of the largest
FX_HD int fx_min(int a, int b) {
#ifdef __CUDA_ARCH__
  return min(a, b);
#else
  return a < b ? a : b;
#endif
}
FX_HD int fx_max(int a, int b) {
#ifdef __CUDA_ARCH__
  return max(a, b);
#else
  return a > b ? a : b;
#endif
}
// as fx_double, opaque like fx_bits
FX_HD double fx_value(fx b) {
#ifdef __CUDA_ARCH__
  double x;
  asm("mov.b64 %0, %1;" : "=d"(x) : "l"(b));
  return x;
#else
  return fx_double(b);
#endif
}

// sum of the six neighbours n less six times the centre c, to about 2^-58 of the largest
// of them, with six guard bits (values below that count as zero, as they would in FP64);
// fp64(): the sum outside the range
template <class F>
FX_HD double fx_lap6(double c, const double n[6], F fp64) {
  fx b[7];
  b[0] = fx_bits(c);
#pragma unroll
  for (int q = 0; q < 6; ++q) b[q + 1] = fx_bits(n[q]);
  int ex[7], emax = 0;
#pragma unroll
  for (int q = 0; q < 7; ++q) {
    ex[q] = (int)(b[q] >> 52) & 0x7ff;
    emax = fx_max(emax, ex[q]);
  }
  if (!fx_sum_ok(emax)) return fp64();
  fx s = 0;   // (a zero's hidden bit shifts out: emax >= 70)
#pragma unroll
  for (int q = 0; q < 7; ++q) {
    const ufx m = ((ufx)b[q] & 0xfffffffffffffull) | 0x10000000000000ull;
    const fx sg = b[q] >> 63;
    const fx v = ((fx)((m << 6) >> fx_min(emax - ex[q], 63)) ^ sg) - sg;
    s += q == 0 ? -6 * v : v;
  }
  if (s == 0) return 0.0;
  const ufx a = s < 0 ? -(ufx)s : (ufx)s;
  const int z = fx_clz(a);               // at least 1
  const ufx w = a << z;                  // the exponent field less one: 11 to 2043
  const fx r = ((fx)(emax + 4 - z) << 52) + (fx)((w >> 11) + ((w >> 10) & 1));
  return fx_value(r | (s & (fx)0x8000000000000000ull));
}

// sum of the 24 values o around a 2 x 2 x 2 group of cells less three times the eight
// inside, q (the group's summed second differences: each cell is a neighbour of three
// others), as fx_lap6 with four guard bits (48 units of the largest value fit); false where
// it does not apply.  Values down to 1/16 of the largest enter exactly.
FX_HD bool fx_lap_group(const double q[8], const double o[24], double &sum) {
  int emax = 0;
#pragma unroll
  for (int u = 0; u < 8; ++u) emax = fx_max(emax, (int)(fx_bits(q[u]) >> 52) & 0x7ff);
#pragma unroll
  for (int u = 0; u < 24; ++u) emax = fx_max(emax, (int)(fx_bits(o[u]) >> 52) & 0x7ff);
  if (!fx_sum_ok(emax)) return false;
  auto part = [emax](double x) {   // (a zero's hidden bit shifts out: emax >= 70)
    const fx b = fx_bits(x), sg = b >> 63;
    const ufx m = ((ufx)b & 0xfffffffffffffull) | 0x10000000000000ull;
    return ((fx)((m << 4) >> fx_min(emax - ((int)(b >> 52) & 0x7ff), 63)) ^ sg) - sg;
  };
  fx in = 0, s = 0;
#pragma unroll
  for (int u = 0; u < 8; ++u) in += part(q[u]);
#pragma unroll
  for (int u = 0; u < 24; ++u) s += part(o[u]);
  s -= 3 * in;
  sum = 0.0;
  if (s == 0) return true;
  const ufx a = s < 0 ? -(ufx)s : (ufx)s;
  const int z = fx_clz(a);               // at least 1
  const ufx w = a << z;                  // the exponent field less one: 13 to 2045
  const fx r = ((fx)(emax + 6 - z) << 52) + (fx)((w >> 11) + ((w >> 10) & 1));
  sum = fx_value(r | (s & (fx)0x8000000000000000ull));
  return true;
}

// Is an entry outside the format at a corner of an nr x nt table?  (k = 0 .. 3)
FX_HD bool fx_outside(double v) { return (fx_bits(v) & 0x7fffffffffffffffLL) >= fx_bits(FX_MAX_LOG10); }
FX_HD bool corner_outside(int nr, int nt, int k, const double *le, const double *lp, const double *lc) {
  const long long at = ((k & 2) ? (long long)(nr - 1) * nt : 0) + ((k & 1) ? nt - 1 : 0);
  return fx_outside(le[at]) || fx_outside(lp[at]) || fx_outside(lc[at]);
}

// The table's axes in fixed point (the same function of the FP64 axes for every
// caller).  valid: the format takes them.
struct FxAxes {
  int valid;
  int sh;              // x (cell units along log rho) has sh fraction bits after the scaling
  fx L0, Dmax, tol;    // log2 of the lowest density, the range, half an FP64 ulp of log10 rho there
  ufx G;               // 1 / (cell width), 64-bit significand
  fx lt0, dlt;         // log2 T of the coldest node, cell width (Q55)
  unsigned dlt_lo;     // its next 32 bits
};

inline FxAxes fx_axes(int nr, int nt, double lr0, double lr1, double inv_dlr, double lt0, double dlt) {
  FxAxes a;
  memset(&a, 0, sizeof a);
  a.L0 = fx_of_log10(lr0);
  const fx l1 = fx_of_log10(lr1);
  a.lt0 = fx_of_log10(lt0);
  const fx lt1 = fx_of_log10(lt0 + (nt - 1) * dlt);
  if (a.L0 == FX_BAD || l1 == FX_BAD || a.lt0 == FX_BAD || lt1 == FX_BAD || !(inv_dlr > 0x1p-8 && inv_dlr < 0x1p20) ||
      !(dlt < 32.0) || nr > (1 << 24) || nt > (1 << 24))
    return a;
  a.Dmax = l1 - a.L0;
  const double m = (lr0 < 0 ? -lr0 : lr0) > (lr1 < 0 ? -lr1 : lr1) ? (lr0 < 0 ? -lr0 : lr0) : (lr1 < 0 ? -lr1 : lr1);
  int ex = 0;
  while ((double)(1u << (ex + 1)) <= m) ++ex;      // 2^ex <= largest |log10 rho| (or 1)
  a.tol = (fx)(3.3219 * (double)(1u << (ex + 2))); // half an ulp of it: 2^(ex - 53) log2(10) 2^55
  // 1 / (cell width in log2 units), by integer arithmetic: cells / range
  const long double G = (long double)inv_dlr * 0.30102999566398119521373889472449302677L;   // log10(2)
  int eg = 0;
  long double f = G;
  while (f >= 2.0L) { f /= 2.0L; ++eg; }
  while (f < 1.0L) { f *= 2.0L; --eg; }
  a.G = (ufx)(f * 9223372036854775808.0L);         // in [2^63, 2^64)
  a.sh = 54 - eg;
  const long double d2 = (long double)dlt * 3.3219280948873623478703194294893901759L * 36028797018963968.0L;   // Q55
  a.dlt = (fx)d2;
  a.dlt_lo = (unsigned)((d2 - (long double)a.dlt) * 4294967296.0L);
  a.valid = 1;
  return a;
}

// Density cell i and weight w (Q64) of rho; true if clamped to the table.  As in
// FP64, a density within the rounding of the table's edge is not clamped.
FX_HD bool fx_rho_cell(const FxMath *__restrict__ mt, const FxAxes &A, int nr, double rho, int &i, ufx &w) {
  fx D = fx_log2(mt, rho) - A.L0;
  bool cl = false;
  if (D < 0) { cl = D < -A.tol; D = 0; }
  const fx b = fx_bits(rho);
  if ((b & 0x7fffffffffffffffLL) > 0x7ff0000000000000LL) { cl = true; D = 0; }   // not a number
  if (D > A.Dmax) { cl = cl || D > A.Dmax + A.tol; D = A.Dmax; }
  const ufx x = fx_umulhi((ufx)D, A.G);
  i = (int)(x >> A.sh);
  w = x << (64 - A.sh);
  if (i > nr - 2) { i = nr - 2; w = ~0ull; }
  return cl;
}

// log2 T at fraction s (Q64) of temperature cell j
FX_HD fx fx_log2T(const FxAxes &A, int j, ufx s) {
  return A.lt0 + (fx)j * A.dlt + (fx)(((ufx)(unsigned)j * A.dlt_lo) >> 32) + (fx)fx_umulhi((ufx)A.dlt, s);
}

// tables of fx_log2 and fx_exp2 (host, extended precision)
const FxMath &fx_math();

}  // namespace tde
