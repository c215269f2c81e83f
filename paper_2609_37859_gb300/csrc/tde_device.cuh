// tde_device.cuh -- device-side building blocks of the hydro stage: the
// tabulated-EOS inversion, conserved -> primitive recovery with the dual-energy
// switch, PLM / PPM face reconstruction and the HLLC Riemann solver.
//
// Every routine is a per-cell or per-face function in registers; the kernels in
// tde_hydro.cu stage the data through shared memory and call them.  The FP64
// pipe is the limiting resource of this path on sm_103a (FP64 FMA issues at
// about 1/55 of the FP32 rate), so the routines avoid divisions where an algebraically
// equal form with fewer of them exists, and never branch on the Riemann wave
// pattern (a warp that diverged would pay for every branch).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "tde_fx.cuh"

namespace tde {

enum { EOS_IDEAL = 0, EOS_TABLE = 1 };
enum { PLM = 0, PPM = 1 };
enum { RIEMANN_HLLC = 0, RIEMANN_HLLE = 1 };

// The first statement of every kernel launched by pdl_launch: waits until the
// kernels before this one have completed and their writes are visible.  Nothing may
// be read before it that an earlier kernel writes; such pointers are not
// __restrict__ (a load through one may be moved over the wait).  The kernels do not
// release their successors early (griddepcontrol.launch_dependents): CTAs placed
// during a kernel wait on its registers and shared memory, which cost more than the
// launch latency it hides (a step of a 32^3 mesh: 134 us with ordinary launches, 177
// with the early release, 103 without it).
__device__ __forceinline__ void pdl_begin() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// ------------------------------------- comparisons on the integer pipe ----
//
// A double's bit pattern, read as a signed 64-bit integer, orders positive
// values like the values themselves; flipping the magnitude bits of negative
// patterns extends that to a total order (-0 just below +0).  Comparisons,
// minima and maxima written this way run on the integer ALUs, which sit idle
// while the FP64 pipe (where DSETP and DMNMX would issue) bounds the path.
// For NaN operands they are not the IEEE predicates; the kernels count
// non-finite states rather than rely on comparisons with NaN.

// The bits through an opaque move: the compiler recognises sign and magnitude
// masks and comparisons of a double's bits and turns them back into FP64
// instructions (a magnitude into an FP64 addition: 28 of them per cell in an
// eight-variable PPM sweep).
__device__ __forceinline__ long long dbits(double x) {
  long long b;
  asm("mov.b64 %0, %1;" : "=l"(b) : "d"(x));
  return b;
}
__device__ __forceinline__ double dfrom(long long b) {
  double x;
  asm("mov.b64 %0, %1;" : "=d"(x) : "l"(b));
  return x;
}
__device__ __forceinline__ long long dmag(double x) { return dbits(x) & 0x7fffffffffffffffLL; }   // bits of |x|
// order key: key(a) < key(b) iff a < b for non-NaN a, b (except -0 < +0)
__device__ __forceinline__ long long dkey(double x) {
  const long long b = dbits(x);
  return b ^ ((b >> 63) & 0x7fffffffffffffffLL);
}
__device__ __forceinline__ bool dgt0(double x) { return dbits(x) > 0; }          // x > 0
__device__ __forceinline__ bool dge0(double x) { return dkey(x) >= -1; }         // x >= 0 (incl. -0)
__device__ __forceinline__ bool dzero(double x) { return (dbits(x) << 1) == 0; }  // x == +-0
__device__ __forceinline__ bool dlt(double a, double b) { return dkey(a) < dkey(b); }
__device__ __forceinline__ bool dle(double a, double b) { return dkey(a) <= dkey(b); }
__device__ __forceinline__ double dmin(double a, double b) { return dkey(a) <= dkey(b) ? a : b; }
__device__ __forceinline__ double dmax(double a, double b) { return dkey(a) >= dkey(b) ? a : b; }
__device__ __forceinline__ bool dfinite(double x) { return ((dbits(x) >> 52) & 0x7ff) != 0x7ff; }
// -x and |x| by the sign bit
__device__ __forceinline__ double dneg(double x) { return dfrom(dbits(x) ^ (long long)0x8000000000000000ull); }
__device__ __forceinline__ double dabs(double x) { return dfrom(dmag(x)); }
// x truncated to FP32 on the integer pipe (a guide value: normal x with
// 2^-126 <= |x| < 2^128, or zero)
__device__ __forceinline__ float dguide(double x) {
  const long long b = dbits(x);
  const int e = (int)((b >> 52) & 0x7ff) - 1023 + 127;
  if (e <= 0) return 0.0f;
  return __uint_as_float((unsigned)((b >> 32) & 0x80000000u) | ((unsigned)e << 23) | (unsigned)((b >> 29) & 0x7fffff));
}
// the double value of a small integer |k| < 2^51, by one FP64 add
__device__ __forceinline__ double dint(long long k) {
  return __longlong_as_double(0x4338000000000000LL + k) - 6755399441055744.0;
}

// ------------------------------------------------ log10 / exp10 (FP64) ----
//
// Table-driven logarithm and exponential after P. T. P. Tang (ACM TOMS 15, 1989:
// exp; ACM TOMS 16, 1990: log), written for this library: an exact argument
// reduction onto one of 128 table points, a short polynomial of the small
// remainder, and a split (Cody-Waite) constant so that the reduction adds no
// rounding.  Fewer FP64 instructions than the general-purpose routines; within
// a few units in the last place (checked against CUDA's log10 / exp10 by
// tde_math_selftest).  Arguments outside the normal range go to the library.

struct MathTables {
  double logF[182];    // ln(j/128), j = 90 .. 181 (the reduced argument's table points)
  double invF[182];    // 128 / j
  double F[182];       // j / 128
  double exp2j[128];   // 2^(j/128)
};

__device__ __forceinline__ double fast_log10(const MathTables *__restrict__ mt, double x) {
  const long long bits = __double_as_longlong(x);
  const int ex = (int)((bits >> 52) & 0x7ff);
  if (ex == 0 || ex == 0x7ff || bits < 0) return log10(x);
  // x = 2^k m with m in [sqrt(1/2), sqrt(2)) (no cancellation near x = 1), and
  // m = F (1 + r) with F = j/128 the nearest table point, m - F exact
  const long long mant = bits & 0x000fffffffffffffLL;
  const bool upper = mant >= 0x6a09e667f3bcdLL;            // m0 = 1 + mant 2^-52 >= sqrt(2)
  const int k = upper ? ex - 1022 : ex - 1023;
  const double m = __longlong_as_double(mant | (upper ? 0x3fe0000000000000LL : 0x3ff0000000000000LL));
  const int j = upper ? 64 + (int)((mant + (1LL << 45)) >> 46) : 128 + (int)((mant + (1LL << 44)) >> 45);
  const double F = __ldg(&mt->F[j]);
  const double r = __dmul_rn(__dsub_rn(m, F), __ldg(&mt->invF[j]));    // |r| <= 2^-7.5
  // ln(1 + r) = r - r^2/2 + ... + r^7/7 (the next term, r^8/8, is below 2^-55.5
  // relative to the result for |r| <= 2^-7.5)
  double q = 1.0 / 7.0;
  q = __fma_rn(q, r, -1.0 / 6.0);
  q = __fma_rn(q, r, 1.0 / 5.0);
  q = __fma_rn(q, r, -1.0 / 4.0);
  q = __fma_rn(q, r, 1.0 / 3.0);
  q = __fma_rn(q, r, -0.5);
  const double lp = __fma_rn(__dmul_rn(q, r), r, r);
  const double kd = dint(k);
  const double ln2_hi = 0.6931471803691238;   // 32 significant bits: k * ln2_hi is exact
  const double ln2_lo = 1.9082149292705877e-10;
  const double hi = __fma_rn(kd, ln2_hi, __ldg(&mt->logF[j]));
  const double lo = __fma_rn(kd, ln2_lo, lp);
  return __dmul_rn(__dadd_rn(hi, lo), 0.4342944819032518);   // log10(e)
}

__device__ __forceinline__ double fast_exp10(const MathTables *__restrict__ mt, double x) {
  if (!((dbits(x) & 0x7fffffffffffffffLL) < dbits(300.0))) return exp10(x);   // |x| < 300
  // 10^x = 2^(n/128) 10^r with n = round(128 x log2 10), r = x - n log10(2)/128;
  // adding 1.5 2^52 rounds to an integer in the low mantissa bits
  const double big = __fma_rn(x, 425.20679614558236, 6755399441055744.0);   // 128 log2(10)
  const double n = __dsub_rn(big, 6755399441055744.0);
  const double c_hi = 0.002351796840230236;   // log10(2)/128, 32 significant bits
  const double c_lo = 8.946172576579561e-13;
  const double r = __fma_rn(-n, c_lo, __fma_rn(-n, c_hi, x));   // |r| <= log10(2)/256
  const double u = __dmul_rn(r, 2.302585092994046);             // ln 10
  // e^u - 1 = u + u^2/2 + ... + u^5/120, |u| <= 2.7e-3 (the next term, u^6/720,
  // is below 2^-60 relative to the result)
  double q = 1.0 / 120.0;
  q = __fma_rn(q, u, 1.0 / 24.0);
  q = __fma_rn(q, u, 1.0 / 6.0);
  q = __fma_rn(q, u, 0.5);
  const double eu = __fma_rn(__dmul_rn(q, u), u, u);
  const int ni = (int)dbits(big);   // n, from the low bits
  const int jj = ni & 127, kk = ni >> 7;
  const double tj = __ldg(&mt->exp2j[jj]);
  const double v = __fma_rn(tj, eu, tj);   // 2^(jj/128) e^u
  return __longlong_as_double(__double_as_longlong(v) + ((long long)kk << 52));
}

// Tabulated EOS on a uniform (log10 rho, log10 T) grid, [n_rho][n_T], cgs.
struct DTable {
  int nr, nt;
  double lr0, inv_dlr, lt0, dlt;
  double xr_max;                   // nr - 1 (the largest density coordinate)
  const double *__restrict__ le;   // log10 e
  const double *__restrict__ lp;   // log10 P
  const double *__restrict__ lc;   // log10 cs^2
  const float *__restrict__ le32;  // log10 e rounded to FP32 (the network's inputs; the FP64 form's search)
  const MathTables *__restrict__ mt;   // tables of fast_log10 / fast_exp10 (or null)
  // fixed-point form (tde_fx.cuh; log2 units, Q55), built at load where every
  // entry fits it.  node: per (density cell i, temperature node j) the pairs
  // (row i, row i + 1) of log e, log P, log cs^2 in three 16-byte words, so an
  // inversion's last lookups are two runs of 48 bytes; null: converted from the FP64
  // arrays as they are read (eos_invert_views)
  FxAxes fa;
  const FxMath *__restrict__ fm;       // tables of fx_log2 / fx_exp2
  const longlong2 *__restrict__ node;  // [nr - 1][nt][3]
  const int2 *__restrict__ n32;        // [nr - 1][nt] the log e pairs in Q23 (the search)
  union {   // (one word for both: the kernels' argument blocks keep their layout)
    // node given: per density cell and bucket of log e (2^bshift wide from y0), the first
    // and last temperature cell the inversion can end in (null: search the column)
    const ushort2 *__restrict__ bk;
    // node null: a caller's arrays, where this says whether a corner entry is outside the
    // format (null: a loaded table, whose fa says that)
    const int *outside;
  };
  fx y0;
  int bshift, nbk;
};

__device__ __forceinline__ double tlog10(const DTable &t, double x) {
  return t.mt ? fast_log10(t.mt, x) : log10(x);
}
__device__ __forceinline__ double texp10(const DTable &t, double x) {
  return t.mt ? fast_exp10(t.mt, x) : exp10(x);
}

struct Counters {
  unsigned long long rho_floor, p_floor, u_floor, table_clamp, excised, dual_aux_used, synced,
      nonfinite, surrogate_accepted;
};

// Scheme, physics and geometry constants, passed by value to every kernel.
struct Phys {
  int eos, recon, dual, nvar, nwv;
  int eos_mode;   // TDE_INVERT_*: how the table is inverted (the results are identical)
  int riemann;    // RIEMANN_HLLC or RIEMANN_HLLE
  double gamma, gm1, inv_gm1, eta1, eta2;
  double rho_floor, p_floor, u_floor;
  double unit_rho, unit_e, inv_unit_p, inv_unit_e;
  DTable tab;
  int N[3], bc[3], active[3], g[3], ng;
  double xmin[3], dx[3], idx[3], dxmin;
};

struct BH {
  int on, excise;
  double GM, rs2, rexc, t0, x0[3], v0[3], a0[3];
  int frame;          // inertial source of the accelerating frame
  double afr[3];
};

// padded geometry of one MeshBlock; origin (i0, j0, k0) on its level's grid
struct DevBlock {
  int i0, j0, k0, n[3], p[3], level;
  long long off;
};

// k + 1/2 for a small integer |k| < 2^49, by one FP64 add
__device__ __forceinline__ double dhalf(long long k) {
  return dfrom(0x4328000000000000LL + 2 * k + 1) - 3377699720527872.0;   // 1.5 2^51, units of 1/2
}

// 2^e for |e| < 1000, exact (built from the exponent field)
__host__ __device__ __forceinline__ double exp2i(int e) {
  unsigned long long b = (unsigned long long)(1023 + e) << 52;
  double r;
  memcpy(&r, &b, 8);
  return r;
}

// x 2^e for a normal x whose result is normal: an integer add on the exponent
// field (exact, and no FP64 instruction)
__device__ __forceinline__ double scale2i(double x, int e) {
  return dfrom(dbits(x) + ((long long)e << 52));
}

// cell width, its reciprocal and the grid size along a on block B's level
// (refinement halves the cells of the active directions only)
__device__ __forceinline__ double block_dx(const Phys &p, const DevBlock &B, int a) {
  return p.active[a] ? scale2i(p.dx[a], -B.level) : p.dx[a];
}
__device__ __forceinline__ double block_idx(const Phys &p, const DevBlock &B, int a) {
  return p.active[a] ? scale2i(p.idx[a], B.level) : p.idx[a];
}
__device__ __forceinline__ int level_n(const Phys &p, int a, int L) {
  return p.active[a] ? p.N[a] << L : 1;
}

__device__ __forceinline__ void count(unsigned long long *c) {
  if (c) atomicAdd(c, 1ull);
}

// Hardware seeds: approximate double reciprocal and reciprocal square root
// (relative error about 2^-20, under 2^-19, over the normal range, measured by
// tde_math_probe; flush-to-zero).
__device__ __forceinline__ double rcp_seed(double d) {
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(d));
  return r;
}
__device__ __forceinline__ double rsqrt_seed(double d) {
  double r;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(d));
  return r;
}

// 1/d within 0.51 ulp by integer arithmetic (fx_rcp) for normal d whose reciprocal
// is normal; otherwise (zero, infinite, not a number, at the ends of the range)
// from the hardware seed r: with e = 1 - d r, 1/d = r (1 + e + e^2 + ...).
// (The rare forms are calls: inlined, the compiler would evaluate them for every
// thread and select, on the FP64 pipe.)
static __device__ __noinline__ double rcp_fp64(double d) {
  const double r = rcp_seed(d);
  const double e = fma(-d, r, 1.0);
  return fma(r, fma(e, e, e), r);
}
__device__ __forceinline__ double rcp_nr(double d) {
  const long long b = dbits(d);
  return fx_rcp_ok(b) ? fx_rcp(b) : rcp_fp64(d);
}

// sqrt(a / b) for a, b > 0 within 0.52 ulp by integer arithmetic (the wave speeds
// of the Riemann solver and of the time-step condition); the IEEE form where a or
// b is not a positive normal number.
static __device__ __noinline__ double sqrt_ratio_ieee(double a, double b) { return sqrt(a / b); }
__device__ __forceinline__ double sqrt_ratio(double a, double b) {
  const long long ka = dbits(a), kb = dbits(b);
  if (fx_pos_ok(ka) && fx_pos_ok(kb)) return fx_sqrt_ratio(ka, kb);
  return sqrt_ratio_ieee(a, b);
}

// 1/sqrt(t) for t > 0, likewise
static __device__ __noinline__ double rsqrt_ieee(double t) { return 1.0 / sqrt(t); }
__device__ __forceinline__ double rsqrt_nr(double t) {
  const long long k = dbits(t);
  return fx_pos_ok(k) ? fx_rsqrt(k) : rsqrt_ieee(t);
}

// sqrt(r2) < r for r2 >= 0, decided as with the correctly rounded square root:
// away from the boundary the comparison of r2 with r^2 (1 -+ 2^-40) gives the
// same answer (the roundings of r^2 and of the square root are below 2^-51
// relative), and only within that band is the square root taken.  A negative
// or NaN r gives false, as the comparison does.
// The thresholds depend on r alone, so a kernel that tests many cells against one
// sphere forms them once (sphere_of) and tests with inside_sphere; inside_radius
// does both.
struct Sphere {
  double r, lo, hi;   // radius; r^2 (1 - 2^-40), r^2 (1 + 2^-40)
  int mode;           // 0: the band test; 1: r^2 near the subnormals (root test); 2: never inside
};
__device__ __forceinline__ Sphere sphere_of(double r) {
  Sphere s;
  s.r = r;
  const double r2b = r * r;
  s.lo = r2b * (1.0 - 0x1p-40);
  s.hi = r2b * (1.0 + 0x1p-40);
  s.mode = (unsigned long long)dbits(r) > 0x7ff0000000000000ull ? 2 : (((dbits(r2b) >> 52) & 0x7ff) < 64 ? 1 : 0);
  return s;
}
__device__ __forceinline__ bool inside_sphere(double r2, const Sphere &s) {
  if (s.mode == 2) return false;
  if (s.mode == 1) return dlt(sqrt(r2), s.r);   // r^2 near the subnormals
  if (dlt(r2, s.lo)) return true;
  if (dlt(s.hi, r2)) return false;
  return dlt(sqrt(r2), s.r);
}
__device__ __forceinline__ bool inside_radius(double r2, double r) { return inside_sphere(r2, sphere_of(r)); }

// Squared distance of a cell centre from the point mass, in one fixed order of
// roundings for every kernel (a cell's potential and excision flag then agree
// wherever they are evaluated); d0 enters last, so the two transverse terms of
// an x pencil can be summed once per pencil.
__device__ __forceinline__ double bh_r2_yz(double d1, double d2) { return fma(d1, d1, d2 * d2); }
__device__ __forceinline__ double bh_r2(double d0, double d1, double d2) { return fma(d0, d0, bh_r2_yz(d1, d2)); }

// The square of the point mass's time-step limit (the CFL condition with the
// point mass, Sec. 7.1): dt_g^2 = dx / |g| with |g| = GM r / (r^2 + r_s^2)^(3/2),
// written as (dx / GM) s2^2 / (sqrt(s2) r) with s2 = r^2 + r_s^2 from refined
// reciprocals (a few ulps); infinity where there is no limit (GM <= 0, r = 0).
// Its square root is taken once per block, after the minimum (the square root
// is monotonic, so the minimum of the roots is the root of the minimum).
// dxg = bh_dxg(dx, GM), the per-block factor dx / GM (infinite without a limit).
__device__ __forceinline__ double bh_dxg(double dx, double GM) {
  return dgt0(GM) ? dx * rcp_nr(GM) : INFINITY;
}
__device__ __forceinline__ double bh_dt2(double dxg, double r2, double rs2) {
  if (!dgt0(r2)) return INFINITY;
  const double s2 = r2 + rs2;
  return dxg * (s2 * s2) * (rsqrt_nr(s2) * rsqrt_nr(r2));
}

// ---------------------------------------------------------------- EOS ----

// Density cell i and weight w of log10 rho (clamped to the table).
__device__ __forceinline__ bool rho_cell(const DTable &t, double rho, int &i, double &w) {
  double x = (tlog10(t, rho) - t.lr0) * t.inv_dlr;
  bool cl = false;
  if (!dge0(x) || (dbits(x) & 0x7fffffffffffffffLL) > 0x7ff0000000000000LL) { x = 0.0; cl = true; }  // < 0, NaN
  if (dlt(t.xr_max, x)) { x = t.xr_max; cl = true; }
  // i = floor(x) and w = x - i from the bit fields (0 <= x <= nr - 1 < 2^31); the
  // same values as the FP64 floor and subtraction, without the FP64 pipe
  const long long b = dbits(x);
  const int e = (int)((b >> 52) & 0x7ff) - 1023;
  int ii;
  if (e < 0) {
    ii = 0;
    w = x;
  } else {
    const long long m = (b & 0xfffffffffffffLL) | 0x10000000000000LL;
    ii = (int)(m >> (52 - e));
    w = __longlong_as_double(0x3ff0000000000000LL | ((m << e) & 0xfffffffffffffLL)) - 1.0;
  }
  if (ii > t.nr - 2) { ii = t.nr - 2; w = 1.0; }   // x = nr - 1 exactly
  i = ii;
  return cl;
}

// Interpolation formulas are written with explicit rounding so that every kernel
// computes the same bits for the same cell (the surrogate's accepted path must
// equal the bisection path exactly, whatever the compiler fuses around it).
__device__ __forceinline__ double lerp_rn(double w, double a, double b) {
  return __fma_rn(w, b, __dmul_rn(__dsub_rn(1.0, w), a));
}

__device__ __forceinline__ double bilin(const double *__restrict__ f, int nt, int i, double w, int j,
                                        double s) {
  const double *a = f + (size_t)i * nt + j;
  const double *b = a + nt;
  const double lo = lerp_rn(s, __ldg(a), __ldg(a + 1));
  const double hi = lerp_rn(s, __ldg(b), __ldg(b + 1));
  return lerp_rn(w, lo, hi);
}

// Exact linear solve inside temperature cell j of the interpolated column: the
// fraction s of the cell at which it reaches y (g0 <= y < g1), and log10 T
// there.  Shared by every inversion so that all of them compute the same bits.
__device__ __forceinline__ double cell_solve(double y, double g0, double g1) {
  return __dmul_rn(__dsub_rn(y, g0), rcp_nr(__dsub_rn(g1, g0)));
}
__device__ __forceinline__ double cell_log10T(const DTable &t, int j, double s) {
  return __fma_rn(__dadd_rn(dint(j), s), t.dlt, t.lt0);
}

// (rho, e) -> P, cs2 (cgs): the temperature cell of the interpolated log e column
// at fixed density weight, then an exact linear solve inside it (Sec. 4.2, runtime
// map).  Returns true if the input was clamped to the table edge; then *e_used is
// the table's e at the clamped point.  WANT_CS2 = false computes P only (cs2, T
// and e_used are left untouched).
//
// The FP64 form, for entries that the fixed-point format does not take.  The search runs on
// the FP32 copy of log e (le32; null: in FP64) and is confirmed by the FP64 bracket.
template <bool WANT_CS2>
__device__ __forceinline__ void fp64_cell(const DTable &t, int i, double w, int j, double s, bool cl, double e, double &P,
                                          double &cs2, double &e_used, double *T) {
  const int nt = t.nt;
  P = texp10(t, bilin(t.lp, nt, i, w, j, s));
  if (WANT_CS2) {
    cs2 = texp10(t, bilin(t.lc, nt, i, w, j, s));
    if (T) *T = texp10(t, cell_log10T(t, j, s));
    e_used = cl ? texp10(t, bilin(t.le, nt, i, w, j, s)) : e;
  }
}
template <bool WANT_CS2>
__device__ __forceinline__ bool eos_invert_fp64(const DTable &t, double rho, double e, double &P,
                                                double &cs2, double &e_used, double *T) {
  int i;
  double w;
  bool cl = rho_cell(t, rho, i, w);
  const int nt = t.nt;
  const double *__restrict__ a = t.le + (size_t)i * nt;
  const double *__restrict__ b = a + nt;
  auto g = [&](int j) { return lerp_rn(w, __ldg(a + j), __ldg(b + j)); };
  const double y = dgt0(e) ? tlog10(t, e) : -INFINITY;
  int j;
  double s;
  if (!dlt(g(0), y)) {
    j = 0; s = 0.0; cl = true;
  } else if (dle(g(nt - 1), y)) {
    j = nt - 2; s = 1.0; cl = true;
  } else {
    int lo = 0, hi = nt - 1;
    if (t.le32) {
      const float *__restrict__ a32 = t.le32 + (size_t)i * nt;
      const float *__restrict__ b32 = a32 + nt;
      const float w32 = dguide(w), y32 = dguide(y);
      while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        const float a0 = __ldg(a32 + mid);
        if (fmaf(w32, __ldg(b32 + mid) - a0, a0) <= y32) lo = mid; else hi = mid;
      }
    }
    j = lo;
    double g0 = g(j), g1 = g(j + 1);
    if (!(dle(g0, y) && dlt(y, g1))) {
      lo = 0;
      hi = nt - 1;
      while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (dle(g(mid), y)) lo = mid; else hi = mid;
      }
      j = lo;
      g0 = g(j);
      g1 = g(j + 1);
    }
    s = cell_solve(y, g0, g1);
  }
  fp64_cell<WANT_CS2>(t, i, w, j, s, cl, e, P, cs2, e_used, T);
  return cl;
}

// The fixed-point results in temperature cell j of density cell i, every table value
// converted as it is read; false if the cell does not hold y (nor clamps it), or one of its
// entries is outside the format (then out is set).  The same bits as eos_invert's.
template <bool WANT_CS2>
__device__ __forceinline__ bool fx_cell_views(const DTable &t, int i, ufx w, fx y, int j, bool &cl, bool &out, double e,
                                              double &P, double &cs2, double &e_used, double *T) {
  const size_t a = (size_t)i * t.nt + j, b = a + t.nt;
  int top = 0;   // the largest high word of a magnitude (38 has a low word of zero)
  auto g = [&](const double *f, int k) {
    const double u = __ldg(f + a + k), v = __ldg(f + b + k);
    top = max(top, max((int)(dmag(u) >> 32), (int)(dmag(v) >> 32)));
    return fx_lerp(fx_of_log10_in(u), fx_of_log10_in(v), w);
  };
  auto outside = [&] { return top >= (int)(fx_bits(FX_MAX_LOG10) >> 32); };
  const fx g0 = g(t.le, 0), g1 = g(t.le, 1);
  out = outside();
  if (out) return false;
  ufx s;
  bool c = true;
  if (j == 0 && y <= g0) s = 0;
  else if (j == t.nt - 2 && y >= g1) s = ~0ull;
  else if (g0 <= y && y < g1) { s = fx_frac(y - g0, g1 - g0); c = false; }
  else return false;
  const bool clamped = cl || c;
  P = fx_exp2(t.fm, fx_lerp(g(t.lp, 0), g(t.lp, 1), s));
  if (WANT_CS2) {
    cs2 = fx_exp2(t.fm, fx_lerp(g(t.lc, 0), g(t.lc, 1), s));
    if (T) *T = fx_exp2(t.fm, fx_log2T(t.fa, j, s));
    e_used = clamped ? fx_exp2(t.fm, fx_lerp(g0, g1, s)) : e;
  }
  out = outside();
  if (!out) cl = clamped;
  return !out;
}

// Without the prepared table.  One with an entry outside the format at a corner (where a
// table that increases along both axes has its extremes) is inverted in FP64 as a whole: no
// cell pays for both forms (2^22 inversions 0.73 ms; 0.89 to 0.98 with a choice per cell).
// Others -- a caller's arrays, a table loaded without room for the prepared form, entries
// outside elsewhere in the table -- cell by cell: in fixed point, with eos_invert's
// bits, where the cell's entries are inside the format, else in FP64.  Which of the two
// depends on the table and the input alone: where the cell of the FP32 search (on truncations
// of log e) does not hold log e or an entry is outside, the 64-bit search decides, with
// entries outside the format taken at its ends (the columns increase, so a cell inside is
// found).
// (Calls within calls, so that the kernels that never get here save no registers for it.)
template <bool WANT_CS2>
__device__ __forceinline__ int eos_invert_cells(const DTable &t, double rho, double e, double &P, double &cs2,
                                             double &e_used, double *T) {   // -1: FP64
  int i;
  ufx w;
  bool cl = fx_rho_cell(t.fm, t.fa, t.nr, rho, i, w), out;
  const int nt = t.nt;
  const double *__restrict__ a = t.le + (size_t)i * nt;
  const double *__restrict__ b = a + nt;
  const fx y = dgt0(e) ? fx_log2(t.fm, e) : -FX_SAT;
  int lo = 0, hi = nt - 1;
  bool all = !t.le32 && !t.outside;   // every step in 64 bits
  if (!all) {
    const float w32 = (float)(unsigned)(w >> 32) * 2.3283064e-10f;   // 2^-32
    const float y32 = (float)(int)(y >> 32) * 3.5885572e-8f;         // 2^-23 log10(2)
    while (hi - lo > 1) {
      const int mid = (lo + hi) >> 1;
      const float u = dguide(__ldg(a + mid));
      if (fmaf(w32, dguide(__ldg(b + mid)) - u, u) <= y32) lo = mid; else hi = mid;
    }
    if (fx_cell_views<WANT_CS2>(t, i, w, y, lo, cl, out, e, P, cs2, e_used, T)) return cl;
    lo = 0;
    hi = nt - 1;
  }
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (fx_lerp(fx_of_log10_sat(__ldg(a + mid)), fx_of_log10_sat(__ldg(b + mid)), w) <= y) lo = mid; else hi = mid;
  }
  return fx_cell_views<WANT_CS2>(t, i, w, y, lo, cl, out, e, P, cs2, e_used, T) ? (int)cl : -1;
}
template <bool WANT_CS2>
__device__ __noinline__ bool eos_invert_views(const DTable &t, double rho, double e, double &P, double &cs2,
                                              double &e_used, double *T) {
  int r = -1;
  if (t.fa.valid && !(t.outside && *t.outside)) r = eos_invert_cells<WANT_CS2>(t, rho, e, P, cs2, e_used, T);
  return r < 0 ? eos_invert_fp64<WANT_CS2>(t, rho, e, P, cs2, e_used, T) : r > 0;
}

// a pair (row i, row i + 1) of the prepared table interpolated in density
__device__ __forceinline__ fx fx_pair(const longlong2 *__restrict__ q, ufx w) {
  const longlong2 v = __ldg(q);
  return fx_lerp(v.x, v.y, w);
}

// the results at fraction s of cell (i, j); nd = the cell's first node
template <bool WANT_CS2>
__device__ __forceinline__ void eos_at(const DTable &t, const longlong2 *__restrict__ nd, ufx w, int j, ufx s,
                                       bool cl, double e, double &P, double &cs2, double &e_used, double *T) {
  P = fx_exp2(t.fm, fx_lerp(fx_pair(nd + 1, w), fx_pair(nd + 4, w), s));
  if (WANT_CS2) {
    cs2 = fx_exp2(t.fm, fx_lerp(fx_pair(nd + 2, w), fx_pair(nd + 5, w), s));
    if (T) *T = fx_exp2(t.fm, fx_log2T(t.fa, j, s));
    e_used = cl ? fx_exp2(t.fm, fx_lerp(fx_pair(nd, w), fx_pair(nd + 3, w), s)) : e;
  }
}

// The inversion on the prepared table.  The cell with g_j <= y < g_{j+1} is
// unique, so any search that ends in a bracketing cell gives the same result: the
// bucket of log e bounds it to a few cells, a bisection on the 32-bit pairs
// picks one, the 64-bit bracket the solve needs anyway confirms it, and the rare
// miss (log e within 2^-22 of a node) bisects the column in 64 bits.  What bounds
// it for scattered inputs is the gathers (one 16-byte word per lane and load), so
// the buckets (1 or 2 search loads instead of 8) and the node pairs (6 loads for
// all of a cell's 12 values) matter as much as the arithmetic.
template <bool WANT_CS2 = true>
__device__ __forceinline__ bool eos_invert_node(const DTable &t, double rho, double e, double &P,
                                                double &cs2, double &e_used, double *T = nullptr) {
  int i;
  ufx w;
  bool cl = fx_rho_cell(t.fm, t.fa, t.nr, rho, i, w);
  const int nt = t.nt;
  const longlong2 *__restrict__ row = t.node + (size_t)i * nt * 3;
  const fx y = dgt0(e) ? fx_log2(t.fm, e) : -FX_SAT;
  int lo = 0, hi = nt - 1;
  if (t.n32) {
    if (t.bk) {
      const fx q = (y - t.y0) >> t.bshift;
      const int qi = q < 0 ? 0 : (q >= t.nbk ? t.nbk - 1 : (int)q);
      const ushort2 r = __ldg(t.bk + (size_t)i * t.nbk + qi);
      lo = r.x;
      hi = r.y + 1;
    }
    const int2 *__restrict__ r32 = t.n32 + (size_t)i * nt;
    const int y32 = (int)(y >> 32), w32 = (int)(w >> 33);
    while (hi - lo > 1) {
      const int mid = (lo + hi) >> 1;
      const int2 v = __ldg(r32 + mid);
      if (v.x + 2 * __mulhi(v.y - v.x, w32) <= y32) lo = mid; else hi = mid;
    }
  } else {   // every step in 64 bits
    while (hi - lo > 1) {
      const int mid = (lo + hi) >> 1;
      if (fx_pair(row + 3 * mid, w) <= y) lo = mid; else hi = mid;
    }
  }
  int j = lo;
  fx g0 = fx_pair(row + 3 * j, w), g1 = fx_pair(row + 3 * j + 3, w);
  ufx s;
  for (;;) {   // at most twice
    if (j == 0 && y <= g0) { s = 0; cl = true; break; }
    if (j == nt - 2 && y >= g1) { s = ~0ull; cl = true; break; }
    if (g0 <= y && y < g1) { s = fx_frac(y - g0, g1 - g0); break; }
    lo = 0;
    hi = nt - 1;
    while (hi - lo > 1) {
      const int mid = (lo + hi) >> 1;
      if (fx_pair(row + 3 * mid, w) <= y) lo = mid; else hi = mid;
    }
    j = lo;
    g0 = fx_pair(row + 3 * j, w);
    g1 = fx_pair(row + 3 * j + 3, w);
  }
  eos_at<WANT_CS2>(t, row + 3 * j, w, j, s, cl, e, P, cs2, e_used, T);
  return cl;
}

// the inversion for whatever table the kernel got
template <bool WANT_CS2 = true>
__device__ __forceinline__ bool eos_invert(const DTable &t, double rho, double e, double &P,
                                           double &cs2, double &e_used, double *T = nullptr) {
  if (!t.node) return eos_invert_views<WANT_CS2>(t, rho, e, P, cs2, e_used, T);   // uniform
  return eos_invert_node<WANT_CS2>(t, rho, e, P, cs2, e_used, T);
}

// The table's inputs (cgs density and specific internal energy) of a cell with
// density rho and internal energy density U in code units.
__device__ __forceinline__ void eos_inputs(const Phys &p, double rho, double U, double &rho_c,
                                           double &e_c) {
  rho_c = rho * p.unit_rho;
  e_c = (U * rcp_nr(rho)) * p.unit_e;
}

// Table results of a cell computed by a separate pass (the learned-guess
// inversion runs as its own launches): P, cs2 in cgs and eu = the clamped
// table energy, or 0 where the input was inside the table.
struct EOSBuf {
  const double *P, *cs2, *eu;
};

// EOS closure in code units: internal energy density U at density rho ->
// P, cs^2 and the internal energy the table actually represents.  EOSB = 1: take
// the table results of the cell at index flat from eb instead of inverting; 2: the
// table has the prepared form (no call that the kernel keeps registers for).
template <int EOSK, int EOSB = 0>
__device__ __forceinline__ void eos_closure(const Phys &p, double rho, double U, double &P,
                                            double &cs2, double &Uu, Counters *cnt,
                                            const EOSBuf *eb = nullptr, long long flat = 0) {
  if (EOSK == EOS_IDEAL) {
    P = p.gm1 * U;
    cs2 = p.gamma * P / rho;
    Uu = U;
  } else {
    double Pc, c2c, eu;
    bool cl;
    if (EOSB == 1) {
      Pc = eb->P[flat];
      c2c = eb->cs2[flat];
      eu = eb->eu[flat];
      cl = dgt0(eu);
    } else {
      double rc, ec;
      eos_inputs(p, rho, U, rc, ec);
      cl = EOSB == 2 ? eos_invert_node(p.tab, rc, ec, Pc, c2c, eu) : eos_invert(p.tab, rc, ec, Pc, c2c, eu);
    }
    if (cl && cnt) count(&cnt->table_clamp);
    P = Pc * p.inv_unit_p;
    cs2 = c2c * p.inv_unit_e;
    Uu = cl ? rho * (eu * p.inv_unit_e) : U;
  }
}

// Pressure of internal energy density U at density rho (code units), table EOS
// (the compression source of Eq. dual-tabulated-compression needs P only).  PREP: the
// table has its prepared form.
template <int PREP>
__device__ __forceinline__ double table_pressure(const Phys &p, double rho, double U,
                                                 Counters *cnt) {
  double Pc, c2c, eu;
  const double rc = rho * p.unit_rho, ec = (U * rcp_nr(rho)) * p.unit_e;
  const bool cl = PREP ? eos_invert_node<false>(p.tab, rc, ec, Pc, c2c, eu) : eos_invert<false>(p.tab, rc, ec, Pc, c2c, eu);
  if (cl && cnt) count(&cnt->table_clamp);
  return Pc * p.inv_unit_p;
}

// Density (floored), velocities and the internal energy density the EOS gets
// (Eq. dual-econs with the dual-energy switch of Eq. dual-primitive-switch).
template <int DUAL>
__device__ __forceinline__ void c2p_energy(const Phys &p, const double *u, double &rho, double &vx,
                                           double &vy, double &vz, double &Ue, Counters *cnt) {
  rho = u[0];
  if (dlt(rho, p.rho_floor)) { rho = p.rho_floor; if (cnt) count(&cnt->rho_floor); }
  double ir = rcp_nr(rho);
  vx = u[1] * ir; vy = u[2] * ir; vz = u[3] * ir;
  double Uc = u[4] - 0.5 * (u[1] * vx + u[2] * vy + u[3] * vz);   // Eq. dual-econs
  Ue = Uc;
  if (DUAL) {
    if (!(dgt0(Uc) && dlt(p.eta1 * u[4], Uc))) { Ue = u[5]; if (cnt) count(&cnt->dual_aux_used); }
  }
}

// The primitives w = (rho, vx, vy, vz, P[, Gamma_e, Gamma_1][, U_aux]) from the
// floored density, the velocities and the closure's P, cs^2 and represented U
// (code units), with the pressure floor.
template <int EOSK, int DUAL>
__device__ __forceinline__ void c2p_prims(const Phys &p, double uaux, double rho, double vx, double vy, double vz,
                                          double P, double cs2, double Uu, double *w, Counters *cnt) {
  if (dlt(P, p.p_floor)) { P = p.p_floor; if (cnt) count(&cnt->p_floor); }
  w[0] = rho; w[1] = vx; w[2] = vy; w[3] = vz; w[4] = P;
  if (EOSK == EOS_TABLE) {
    w[5] = 1.0 + P * rcp_nr(Uu);         // Gamma_e
    w[6] = rho * cs2 * rcp_nr(P);        // Gamma_1
    if (DUAL) w[7] = uaux;
  } else {
    if (DUAL) w[5] = uaux;
  }
}

// Conserved (rho, m, E[, U_aux]) -> primitives with the dual-energy switch of
// Eq. dual-primitive-switch and the density / pressure floors.
template <int EOSK, int DUAL, int EOSB = 0>
__device__ __forceinline__ void cons_to_prim(const Phys &p, const double *u, double *w,
                                             Counters *cnt, const EOSBuf *eb = nullptr,
                                             long long flat = 0) {
  double rho, vx, vy, vz, Ue;
  c2p_energy<DUAL>(p, u, rho, vx, vy, vz, Ue, cnt);
  double P, cs2, Uu;
  eos_closure<EOSK, EOSB>(p, rho, Ue, P, cs2, Uu, cnt, eb, flat);
  c2p_prims<EOSK, DUAL>(p, DUAL ? u[5] : 0.0, rho, vx, vy, vz, P, cs2, Uu, w, cnt);
}

// ------------------------------------------------------- reconstruction ----
//
// Both schemes work on the differences D of neighbouring cells along a pencil; a
// thread walks a run of cells of one variable, so each cell value is read once
// and each difference formed once.

// PLM, van Leer limiter, cell q0 with the differences dl, dr to its neighbours:
// half-slope h = dl dr / (dl + dr) if dl dr > 0; faces q0 -+ h.  (Where a product
// is added to something, the rounding is spelt out here and in the Riemann
// solvers, so that every kernel they are compiled into gives the same bits.)
__device__ __forceinline__ void plm(double q0, double dl, double dr, double &left, double &right) {
  const long long kl = dbits(dl), kr = dbits(dr);
  left = q0;
  right = q0;
  // dl dr > 0: by the signs, and by the product, which is zero where it underflows
  // (differences of 1e-310, say, whose sum has no finite reciprocal)
  if ((kl ^ kr) >= 0 && (kl << 1) != 0 && (kr << 1) != 0) {
    const double pr = __dmul_rn(dl, dr);
    if (!dzero(pr)) {
      const double ir = rcp_nr(__dadd_rn(dl, dr));
      left = __fma_rn(-pr, ir, q0);
      right = __fma_rn(pr, ir, q0);
    }
  }
}
// a - b, without the subtraction where a = b on every lane that votes.  (The votes of the
// reconstruction are over whichever lanes are still in the loop: a vote only skips work whose
// outcome is known, so no result depends on who votes.  But for equal infinities, whose
// difference is not a number: whether their face values are infinite or none depends on it,
// and the cells beside them are non-finite, and counted as such, either way.)
__device__ __forceinline__ double diff_or_zero(double a, double b) {
  double d = 0.0;
  if (__any_sync(__activemask(), dbits(a) != dbits(b))) d = a - b;
  return d;
}

// PPM interface between cells q0 and q1 = q0 + D1, with D0 and D2 the differences
// below and above: the 4th-order value 7/12 (q0 + q1) - 1/12 (qm1 + q2) is
// q0 + T/2 with T = D1 + (D0 - D2)/6; clipped to [q0, q1] (T to between 0 and
// 2 D1, by its sign and magnitude on the integer pipe).  At |T| = 2 |D1| the value is q1
// itself, not q0 + D1: D1 is rounded, and where q1 is below half an ulp of q0 (a floor
// beside a star) q0 + D1 is zero.  For smaller |T| the exact q0 + T/2 lies short of q1 --
// T/2 is at least an FP64 step below D1, which is within half a step of q1 - q0 -- and
// rounding keeps it in [q0, q1].  The limited values q0 - T and q0 + V of ppm_limit are
// bounded by the neighbours in the same way.  Returns the value and twice its distance
// from q0 (T) and from q1 (V = 2 D1 - T).
__device__ __forceinline__ double ppm_iface(double q0, double q1, double D0, double D1, double D2, double &T,
                                            double &V) {
  double t = fma(D0 - D2, 1.0 / 6.0, D1);
  const long long bt = dbits(t), b1 = dbits(D1);
  const long long m1 = b1 & 0x7fffffffffffffffLL;
  const bool over = (bt & 0x7fffffffffffffffLL) >= m1 + 0x10000000000000LL && (bt ^ b1) >= 0;   // |t| >= 2 |D1|
  if ((bt ^ b1) < 0 || m1 < 0x10000000000000LL) t = 0.0;   // the other sign, or D1 zero (or subnormal)
  T = t;
  V = fma(2.0, D1, -t);
  double a = fma(0.5, t, q0);
  if (over && m1 >= 0x10000000000000LL) {
    T = scale2i(D1, 1);
    V = 0.0;
    a = q1;
  }
  return a;
}

// Colella-Woodward (1984) monotonicity constraints on the parabola (aL, q0, aR),
// given V = 2 (q0 - aL) and T = 2 (aR - q0).  The textbook tests
// (aR - q0)(q0 - aL) <= 0, da^2 < da q6 and da q6 < -da^2 (da = aR - aL,
// q6 = 6 (q0 - (aL + aR) / 2)) read, in these distances: V and T of opposite
// sign or zero; |V| > 2 |T|; |T| > 2 |V|.  All on the integer pipe; the limited
// values 3 q0 - 2 aR = q0 - T and 3 q0 - 2 aL = q0 + V take one FP64 operation
// where a limit acts.
__device__ __forceinline__ void ppm_limit(double q0, double V, double T, double &aL, double &aR) {
  const long long bv = dbits(V), bt = dbits(T);
  const long long mv = bv & 0x7fffffffffffffffLL, mt = bt & 0x7fffffffffffffffLL;
  const bool flat = (bv ^ bt) < 0 || mv == 0 || mt == 0;
  const bool low = !flat && mv > mt + 0x10000000000000LL, high = !flat && mt > mv + 0x10000000000000LL;
  if (flat) {
    aL = q0;
    aR = q0;
  }
  // (a vote, so that the addition is skipped where no lane of the warp needs it
  // rather than evaluated and selected)
  if (__any_sync(__activemask(), low || high)) {
    const double x = q0 + (low ? dneg(T) : V);
    if (low) aL = x;
    if (high) aR = x;
  }
}

// ------------------------------------------------------------------ HLLC ----

// Face state: rho, v[3], P, Gamma_e (or gamma), Gamma_1 (or gamma), U_aux.
struct FState {
  double r, v[3], P, ge, g1, A;
};

// HLLC flux across a face normal to direction D (Toro, Spruce & Speares) with
// Davis wave-speed estimates; F[0..4] = mass, momentum, energy; F[5] = U_aux
// flux (Eq. dual-flux); vf = face velocity (Eq. dual-face-velocity).  The wave
// pattern is selected without branching on it.
//
// Every speed enters relative to the chosen side's gas (sigma = S - u,
// w = S_M - u), which keeps the contact's distance from the gas to full precision
// in flows far faster than sound, and the star state's flux is written by its
// contact: mass m = r chi S_M with chi = sigma / (S - S_M), momentum m v plus
// P* = P + r sigma w, energy (E* + P*) S_M, auxiliary A chi S_M, instead of
// F_K + S (U*_K - U_K).  Outside the wave fan chi = 1, w = 0 and S_M = u give the
// side's own flux by the same expressions.  33 FP64 operations a face
// instead of 73 (the square roots and reciprocals are integer arithmetic).
template <int D, int EOSK, int DUAL>
__device__ __forceinline__ void hllc(const Phys &p, const FState &L, const FState &R, double *F,
                                     double &vf) {
  const int t1 = D == 0 ? 1 : 0, t2 = D == 2 ? 1 : 2;
  const double ul = L.v[D], ur = R.v[D];
  const double cl = sqrt_ratio(L.g1 * L.P, L.r), cr = sqrt_ratio(R.g1 * R.P, R.r);
  // S_L - u_L = min(-c_L, du - c_R), S_R - u_R = max(c_R, c_L - du), du = u_R - u_L
  const double du = ur - ul;
  const double sl = dmin(dneg(cl), du - cr), sr = dmax(cr, cl - du);
  const double al = __dmul_rn(L.r, sl), ar = __dmul_rn(R.r, sr);
  // S_M - u_L = (P_R - P_L - a_R du) / (a_L - a_R)
  const double wl = __dmul_rn(fma(-ar, du, R.P - L.P), rcp_nr(__dsub_rn(al, ar)));
  const double SM = __dadd_rn(ul, wl);
  const bool supL = dle(dneg(ul), sl), supR = dle(sr, dneg(ur));   // S_L >= 0, S_R <= 0
  const bool useL = supL || (!supR && dge0(SM)), sup = supL || supR;
  const double r = useL ? L.r : R.r, un = useL ? ul : ur, P = useL ? L.P : R.P;
  const double v0 = useL ? L.v[0] : R.v[0], v1 = useL ? L.v[1] : R.v[1], v2 = useL ? L.v[2] : R.v[2];
  const double vt1 = useL ? L.v[t1] : R.v[t1], vt2 = useL ? L.v[t2] : R.v[t2];
  const double sg = useL ? sl : sr, rs = useL ? al : ar;
  // E + P
  const double ig = EOSK == EOS_IDEAL ? p.inv_gm1 : rcp_nr((useL ? L.ge : R.ge) - 1.0);
  const double EP = fma(0.5 * r, fma(v2, v2, fma(v1, v1, v0 * v0)), fma(P, ig, P));
  const double wk = useL ? wl : __dsub_rn(wl, du);
  double den = __dsub_rn(sg, wk);
  if (dzero(den)) den = 1.0;   // only outside the fan
  const double inv = rcp_nr(den);
  const double uf = sup ? un : SM, w = sup ? 0.0 : wk;
  const double q = sup ? uf : (sg * inv) * uf;   // chi times the face's normal velocity
  // E* + P* = E + P + w ((E + P + r sigma S_M) / (S - S_M) + r sigma)
  const double H = fma(w, fma(fma(rs, uf, EP), inv, rs), EP);
  const double m = r * q;
  F[0] = m;
  F[1 + D] = fma(m, uf, fma(rs, w, P));
  F[1 + t1] = m * vt1;
  F[1 + t2] = m * vt2;
  F[4] = H * uf;
  if (DUAL) {
    // the chosen side is the upwind one of the mass flux
    F[5] = q * (useL ? L.A : R.A);
    vf = q;
  } else {
    F[5] = 0.0;
    vf = 0.0;
  }
}

// HLLE flux across a face normal to direction D (Harten, Lax and van Leer with
// Einfeldt's two-wave form; the production solver of Table 1) with the same
// Davis wave-speed bounds as hllc: b- = min(S_L, 0), b+ = max(S_R, 0),
// F = (b+ F_L - b- F_R + b+ b- (U_R - U_L)) / (b+ - b-), written by what each
// side carries: with alpha = b+ / (b+ - b-) and beta = 1 - alpha, side L enters
// with the velocity a_L = alpha (u_L - b-) and the pressure share alpha P_L, side R
// with a_R = beta (u_R - b+) and beta P_R (about 45 FP64 operations instead of
// 90); F[5] and vf follow the sign of the mass flux as for hllc.
template <int D, int EOSK, int DUAL>
__device__ __forceinline__ void hlle(const Phys &p, const FState &L, const FState &R, double *F,
                                     double &vf) {
  const double ul = L.v[D], ur = R.v[D];
  const double cl = sqrt_ratio(L.g1 * L.P, L.r), cr = sqrt_ratio(R.g1 * R.P, R.r);
  const double igl = EOSK == EOS_IDEAL ? p.inv_gm1 : rcp_nr(L.ge - 1.0);
  const double igr = EOSK == EOS_IDEAL ? p.inv_gm1 : rcp_nr(R.ge - 1.0);
  const double El = fma(0.5 * L.r, fma(L.v[2], L.v[2], fma(L.v[1], L.v[1], L.v[0] * L.v[0])), __dmul_rn(L.P, igl));
  const double Er = fma(0.5 * R.r, fma(R.v[2], R.v[2], fma(R.v[1], R.v[1], R.v[0] * R.v[0])), __dmul_rn(R.P, igr));
  const double bm = dmin(dmin(ul - cl, ur - cr), 0.0);
  const double bp = dmax(dmax(ul + cl, ur + cr), 0.0);
  double den = bp - bm;
  if (dzero(den)) den = 1.0;   // both fluxes vanish there
  const double inv = rcp_nr(den), al = __dmul_rn(bp, inv), be = __dmul_rn(dneg(bm), inv);
  const double cL = __dmul_rn(al, __dsub_rn(ul, bm)), cR = __dmul_rn(be, __dsub_rn(ur, bp));
  const double ml = __dmul_rn(cL, L.r), mr = __dmul_rn(cR, R.r);
  const double pl = __dmul_rn(al, L.P), pr = __dmul_rn(be, R.P);
  F[0] = __dadd_rn(ml, mr);
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    const double f = __fma_rn(ml, L.v[q], __dmul_rn(mr, R.v[q]));
    F[1 + q] = q == D ? __dadd_rn(f, __dadd_rn(pl, pr)) : f;
  }
  F[4] = fma(El, cL, fma(pl, ul, fma(Er, cR, __dmul_rn(pr, ur))));
  if (DUAL) {
    double f = F[0];
    bool up = dgt0(f);
    double ru = up ? L.r : R.r, Au = up ? L.A : R.A;
    double iru = rcp_nr(ru);
    F[5] = !dzero(f) ? f * (Au * iru) : 0.0;
    vf = !dzero(f) ? f * iru : 0.0;
  } else {
    F[5] = 0.0;
    vf = 0.0;
  }
}

}  // namespace tde
