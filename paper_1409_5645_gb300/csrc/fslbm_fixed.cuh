// fslbm_fixed.cuh -- the TRT collision of the FP64 form in 64-bit fixed point.
//
// GB300 issues two FP64 operations per cycle and SM against 64 or more 32-bit
// integer ones, and the FP64 collision (about 210 FP64 instructions a cell)
// kept the bulk kernel on that pipe at a tenth of the copy bandwidth.  The
// collision needs no floating exponent: in a cell of a flow near rho = 1
// every operand lies in (-8, 8), so it is done on 64-bit integers in units of
// 2^-60.  Sums are exact; a product (64 x 64 bits, the high word kept, rounded
// to nearest up to 0.6 unit, its mean error zero) errs by at most about 2^-60.
// An FP64 value in the range of the moving populations (2^-6 .. 2^-4) has a
// spacing of 2^-58 or 2^-57, so the result before its one rounding back to FP64
// is nearer to the exact collision than a chain of FP64 operations comes (400 000
// states of each of five kinds: rms error of a population 4.0e-18 against
// 0.9e-17 to 3.0e-17; mean error of a cell's mass and momentum in a step near
// equilibrium, tau 0.8, g_x = 1e-6, 0.4e-19 and 1e-21 against 3.5e-19 and
// 5.2e-19).  The weights are the FP64 values of 1/3, 1/18 and 1/36, whose sum
// is 1 - 2^-54: with exact ones the density would not relax toward
// (1 - 2^-54) rho as it does in FP64, and a film's interface mass leaves the
// FP64 run's by 1e-15 of its value a step.
//
// A cell whose populations are not all in [0, 1/4) (rest: [0, 1)), whose
// density is not in [1/2, 2), whose momentum reaches 1/2, or whose result
// leaves [2^-28, 8) takes collide<double> (or, for the last, the hardware
// conversion): negative populations, NaN and states far from rho = 1 included.  Values below 2^-8
// are rounded to the unit, which FP64's own sums with their neighbours do too.
#pragma once
#include <math.h>
#include <string.h>

#include "fslbm_dev.cuh"

namespace fsl {

// high 64 bits of a signed product, to about 0.6 unit: the low halves enter
// with 31 bits, and `mean` (units of 2^-31) stands for the mean of what is
// dropped: half a unit by the shift, a0 b0 / 2^64 of the low words and half a
// high word for an odd low word.
__host__ __device__ __forceinline__ long long mul_hi_near(long long a, long long b, long long mean) {
  const int ah = (int)(a >> 32), bh = (int)(b >> 32);
  const int al = (int)((unsigned)a >> 1), bl = (int)((unsigned)b >> 1);
  const long long t = (long long)ah * bl + (long long)al * bh + mean;
  return (long long)ah * bh + (t >> 31);
}
// The means.  Of a constant operand c beside one of random low bits (its low
// word's mean is 2^31), even or of either parity; of a square and of a product
// of two even operands of random low bits (1/2 + 1/3 and 1/2 + 1/4).  One
// value for them all (3/4) made an error of fixed sign of every step: 6.9e-18
// in a cell's mass and 1e-18 to 2e-18 in its momentum, a body force that a
// film's velocity followed.
__host__ __device__ __forceinline__ constexpr long long mean_even(long long c) {
  return 0x40000000LL + (long long)((unsigned)c >> 2);
}
__host__ __device__ __forceinline__ constexpr long long mean_any(long long c) { return mean_even(c) + (c >> 34); }
constexpr long long MEAN_SQUARE = 0x6aaaaaabLL, MEAN_PRODUCT = 0x60000000LL;

// x >> s with s >= 64 giving 0
__host__ __device__ __forceinline__ unsigned long long shr_clamped(unsigned long long x, unsigned s) {
#ifdef __CUDA_ARCH__
  unsigned long long r;
  asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(x), "r"(s));
  return r;
#else
  return s < 64 ? x >> s : 0;
#endif
}

// an FP64 value in [0, 1) (its bits) in units of 2^-60
__host__ __device__ __forceinline__ long long fix_of(unsigned long long bits) {
  const unsigned e = (unsigned)(bits >> 52);
  const unsigned long long m = ((bits & 0xfffffffffffffULL) | 0x10000000000000ULL) << 10;
  return (long long)shr_clamped(m, 1025u - e);
}

// the same rounded to nearest (ties to even), for values that may have bits
// under 2^-60 (those below 2^-8): cut off they would be an error of fixed sign
__host__ __device__ __forceinline__ long long fix_near(unsigned long long bits) {
  const unsigned e = (unsigned)(bits >> 52), s = 1025u - e;
  if (s > 63u) return 0;  // (below half a unit, and zero)
  const unsigned long long m = ((bits & 0xfffffffffffffULL) | 0x10000000000000ULL) << 10;
  return (long long)((m + ((1ULL << (s - 1u)) - 1ULL) + ((m >> s) & 1ULL)) >> s);
}
// bits of an FP64 value's high word: [2^-8, 1/4) and [2^-8, 1) convert exactly
constexpr unsigned FIX_LOW = 0x3f700000u, FIX_MOVING = 0x3fd00000u, FIX_REST = 0x3ff00000u;

// the FP64 value nearest to x 2^-60 (ties to even), for x >= 2^32
__host__ __device__ __forceinline__ unsigned long long bits_of(long long x) {
#ifdef __CUDA_ARCH__
  const int n = __clz((int)(x >> 32));
#else
  const int n = __builtin_clz((unsigned)(x >> 32));
#endif
  unsigned long long a = (unsigned long long)x << (n - 1);  // the leading bit at bit 62
  a += 0x1ffULL + ((a >> 10) & 1ULL);
  return (a >> 10) + ((unsigned long long)(unsigned)(1025 - n) << 52);
}

__host__ __device__ __forceinline__ unsigned long long bits_of_double(double v) {
#ifdef __CUDA_ARCH__
  return (unsigned long long)__double_as_longlong(v);
#else
  unsigned long long b;
  memcpy(&b, &v, 8);
  return b;
#endif
}
__host__ __device__ __forceinline__ double double_of_bits(unsigned long long b) {
#ifdef __CUDA_ARCH__
  return __longlong_as_double((long long)b);
#else
  double v;
  memcpy(&v, &b, 8);
  return v;
#endif
}
// x 2^-60 for any x
__host__ __device__ __forceinline__ double double_of_fix(long long x) { return (double)x * 0x1p-60; }

// The constants of Par from its rates and forces: |lambda| < 2 holds for every
// tau > 1/2; the forces must leave the operands in range, and u_max^2 must be
// some units of 2^-60 (a guard near 1e-9 is kept by the FP64 collision).
inline void fix_constants(Par& p) {
  bool ok = !p.compressible && !p.linear_eq;
  for (int a = 0; a < 3; ++a) {
    const double gl = p.g[a] * p.inv_lam_m;
    ok = ok && fabs(p.g[a]) < 1.0 / 32.0 && fabs(gl) < 1.0 / 8.0;
    p.fx_hg[a] = ok ? llround(p.g[a] * 0x1p59) : 0;
    p.fx_gl[a] = ok ? llround(gl * 0x1p60) : 0;
    p.fx_gm[a] = ok ? llround((gl * 0x1p60 - (double)p.fx_gl[a]) * (0x1p31 / 3.0)) : 0;
  }
  ok = ok && p.lam_p > -2.0 && p.lam_p < 0.0 && p.lam_m > -2.0 && p.lam_m < 0.0;
  p.fx_lp = ok ? llround(p.lam_p * 0x1p62) : 0;
  p.fx_lm = ok ? llround(p.lam_m * 0x1p62) : 0;
  ok = ok && !(p.umax2 > 0.0 && p.umax2 < 0x1p-30);
  p.fx_um2 = p.umax2 > 0.0 && p.umax2 < 4.0 ? llround(p.umax2 * 0x1p60) : 0x7fffffffffffffffLL;
  p.fix_ok = ok;
}

// Density in [1/2, 2), |j| < 1/2.  With the populations' range the upper bounds
// keep every product below (4 rho fits).  The lower one is for the unit, which
// is absolute: at a density of 1/2 FP64's own chain still errs twice as far (8e-18
// rms), below 1/4 it is the nearer one, and a density of zero has to reach its
// check there.
__host__ __device__ __forceinline__ bool fix_range(long long r, long long jx, long long jy, long long jz) {
  auto half = [](long long j) { return (unsigned)((int)(j >> 32) + 0x08000000) < 0x10000000u; };
  return (unsigned)((int)(r >> 32) - 0x08000000) < 0x18000000u && half(jx) && half(jy) && half(jz);
}

// What a cell's populations share, and the collision of the rest population
// and of a link pair from it.  The differences 2 n that the rates multiply are
// taken in units of 2^-62, where their quarters and halves are whole.
struct FixTerms {
  long long lp, lm, lp2, lm2;  // lambda_+- in units of 2^-62 and 2^-61
  long long k0, kp, kq, km;    // the means of their products: rest, axis pairs, diagonal pairs, odd parts
  long long xx, yy, zz, xy, xz, yz, usq;
  long long d4, a4, bx, by, bz;  // 4 (rho - 3/2 u.u), that / 36, 4 u^eq / 12
  __host__ __device__ __forceinline__ FixTerms(const Par& p, long long r, long long jx, long long jy, long long jz) {
    // fl(1/36) and fl(3 fl(1/36)), units of 2^-64
    constexpr long long K36 = 0x071c71c71c71c700LL, K12 = 0x1555555555555500LL;
    lp = p.fx_lp;
    lp2 = p.fx_lp >> 1;
    lm2 = p.fx_lm >> 1;
    k0 = mean_any(lp);
    kp = mean_even(lp2);
    kq = mean_any(lp2);
    km = mean_even(lm2);
    const long long ux = (jx + p.fx_hg[0]) << 2, uy = (jy + p.fx_hg[1]) << 2, uz = (jz + p.fx_hg[2]) << 2;
    xx = mul_hi_near(ux, ux, MEAN_SQUARE);
    yy = mul_hi_near(uy, uy, MEAN_SQUARE);
    zz = mul_hi_near(uz, uz, MEAN_SQUARE);
    xy = mul_hi_near(ux, uy, MEAN_PRODUCT);
    xz = mul_hi_near(ux, uz, MEAN_PRODUCT);
    yz = mul_hi_near(uy, uz, MEAN_PRODUCT);
    usq = xx + yy + zz;
    // e^+ = w rho + 9/2 w (c.u)^2 - 3/2 w u.u: a = (rho - 3/2 u.u) / 36 is the
    // diagonal links' part (the axis links' twice that), 9/2 w = 1/8 and 1/4
    d4 = (r << 2) - 6 * usq;
    a4 = mul_hi_near(d4, K36, mean_even(K36));
    // e^- = 3 w (c.u^eq): 1/12 of u^eq (diagonal links), twice that (axis links)
    // (g / lambda_- to a unit would be a force to 4e-19, 4e-13 of a film's 1e-6:
    // what its rounding leaves joins the product's mean)
    bx = mul_hi_near((jx - p.fx_gl[0]) << 2, K12, mean_even(K12) - p.fx_gm[0]);
    by = mul_hi_near((jy - p.fx_gl[1]) << 2, K12, mean_even(K12) - p.fx_gm[1]);
    bz = mul_hi_near((jz - p.fx_gl[2]) << 2, K12, mean_even(K12) - p.fx_gm[2]);
  }
  __host__ __device__ __forceinline__ long long rest(long long x) const {
    constexpr long long K3 = 0x5555555555555400LL;  // fl(1/3)
    return x + mul_hi_near(lp, (x << 2) - mul_hi_near(d4, K3, mean_even(K3)), k0);
  }
  // the pair of odd link q (population x) and its opposite (xb): f + l+ n^+ +- l- n^-
  __host__ __device__ __forceinline__ void pair(int q, long long x, long long xb, long long& y, long long& yb) const {
    long long e8, m8;  // 8 e^+, 8 e^-
    if (q <= 6) {
      e8 = 4 * a4 + 2 * (q == 1 ? xx : (q == 3 ? yy : zz));
      m8 = 4 * (q == 1 ? bx : (q == 3 ? by : bz));
    } else {
      const long long s = q <= 10 ? xx + yy : (q <= 14 ? xx + zz : yy + zz);
      const long long c = q <= 10 ? xy : (q <= 14 ? xz : yz);
      const bool same = cx(q) * cy(q) + cx(q) * cz(q) + cy(q) * cz(q) > 0;  // the two components' signs
      e8 = 2 * a4 + (same ? s + 2 * c : s - 2 * c);
      m8 = 2 * (cx(q) * bx + cy(q) * by + cz(q) * bz);
    }
    const long long rp = mul_hi_near(lp2, 4 * (x + xb) - e8, q <= 6 ? kp : kq);
    const long long rm = mul_hi_near(lm2, 4 * (x - xb) - m8, km);
    y = x + rp + rm;
    yb = xb + rp - rm;
  }
};

// The collision in place: f <- f + l+ n^+ + l- n^- with the density sum f in
// units of 2^-60; fast = the speed guard's test (|u|^2 > u_max^2).  False, with
// f untouched, where the cell is out of range.
__host__ __device__ __forceinline__ bool collide_fixed(const Par& p, double (&f)[19], long long& rho, bool& fast) {
  if (!p.fix_ok) return false;
  // (as unsigned, a negative value's or a NaN's high word is above the bounds,
  // and one below 2^-8 wraps above them too)
  unsigned top = 0u;
#pragma unroll
  for (int q = 1; q < 19; ++q) {
    const unsigned h = (unsigned)(bits_of_double(f[q]) >> 32) - FIX_LOW;
    top = h > top ? h : top;
  }
  const unsigned h0 = (unsigned)(bits_of_double(f[0]) >> 32);
  long long x[19];
  if (top < FIX_MOVING - FIX_LOW && h0 - FIX_LOW < FIX_REST - FIX_LOW) {
#pragma unroll
    for (int q = 0; q < 19; ++q) x[q] = fix_of(bits_of_double(f[q]));
  } else {
    bool in = h0 < FIX_REST;
#pragma unroll
    for (int q = 1; q < 19; ++q) in = in && (unsigned)(bits_of_double(f[q]) >> 32) < FIX_MOVING;
    if (!in) return false;
#pragma unroll
    for (int q = 0; q < 19; ++q) x[q] = fix_near(bits_of_double(f[q]));
  }
  long long r = x[0], jx = 0, jy = 0, jz = 0;
#pragma unroll
  for (int q = 1; q < 19; ++q) r += x[q];
#pragma unroll
  for (int q = 1; q < 19; q += 2) {
    const long long d = x[q] - x[q + 1];
    jx += cx(q) * d;
    jy += cy(q) * d;
    jz += cz(q) * d;
  }
  if (!fix_range(r, jx, jy, jz)) return false;
  const FixTerms T(p, r, jx, jy, jz);
  x[0] = T.rest(x[0]);
  long long low = x[0];
#pragma unroll
  for (int q = 1; q < 19; q += 2) {
    T.pair(q, x[q], x[q + 1], x[q], x[q + 1]);
    low = x[q] < low ? x[q] : low;
    low = x[q + 1] < low ? x[q + 1] : low;
  }
  if (low >= (1LL << 32)) {
#pragma unroll
    for (int q = 0; q < 19; ++q) f[q] = double_of_bits(bits_of(x[q]));
  } else {  // a negative or a tiny result
#pragma unroll
    for (int q = 0; q < 19; ++q) f[q] = double_of_fix(x[q]);
  }
  rho = r;
  fast = T.usq > p.fx_um2;
  return true;
}

#ifdef __CUDACC__
// collide_fixed with population q on lane q of a warp (q = 0 on the lanes from
// 19 on): the same integers, so the same bits.  False, with f untouched, where
// the cell is out of range.
__device__ __forceinline__ bool collide_warp(const Par& p, int q, double& f, long long& rho) {
  const unsigned FULL = 0xffffffffu;
  if (!p.fix_ok) return false;
  const int lane = threadIdx.x & 31, qb = q == 0 ? 0 : ((q & 1) ? q + 1 : q - 1);
  const unsigned h = (unsigned)(bits_of_double(f) >> 32);
  if (!__all_sync(FULL, h < (q ? FIX_MOVING : FIX_REST))) return false;
  const long long x = fix_near(bits_of_double(f));
  long long m[4] = {0, 0, 0, 0};
  if (lane < 19) {
    m[0] = x;
    m[1] = cx(q) * x;
    m[2] = cy(q) * x;
    m[3] = cz(q) * x;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1)
#pragma unroll
    for (int k = 0; k < 4; ++k) m[k] += __shfl_xor_sync(FULL, m[k], o);
  if (!fix_range(m[0], m[1], m[2], m[3])) return false;  // (the same on every lane)
  const FixTerms T(p, m[0], m[1], m[2], m[3]);
  const long long xb = __shfl_sync(FULL, x, qb);
  long long y, yb;
  if (q == 0) {
    y = T.rest(x);
  } else {  // the pair's terms from its odd link, on both of its lanes
    const bool odd = (q & 1) != 0;
    T.pair(odd ? q : qb, odd ? x : xb, odd ? xb : x, y, yb);
    if (!odd) y = yb;
  }
  // (both conversions round the same; a thread chooses one for its 19)
  f = y >= (1LL << 32) ? double_of_bits(bits_of(y)) : double_of_fix(y);
  rho = m[0];
  return true;
}
#endif

// Density less 1 and momentum of populations in the collision's range, in units
// of 2^-60; false where they are not, or where one of the four reaches 7/16
// (so that eighteen cells' sum fits 64 bits)
__host__ __device__ __forceinline__ bool moments_fixed(const double (&f)[19], long long& dev, long long (&j)[3]) {
  bool in = (unsigned)(bits_of_double(f[0]) >> 32) < FIX_REST;
#pragma unroll
  for (int q = 1; q < 19; ++q) in = in && (unsigned)(bits_of_double(f[q]) >> 32) < FIX_MOVING;
  if (!in) return false;
  dev = fix_near(bits_of_double(f[0])) - (1LL << 60);
  j[0] = j[1] = j[2] = 0;
#pragma unroll
  for (int q = 1; q < 19; q += 2) {
    const long long a = fix_near(bits_of_double(f[q])), b = fix_near(bits_of_double(f[q + 1]));
    dev += a + b;
    j[0] += cx(q) * (a - b);
    j[1] += cy(q) * (a - b);
    j[2] += cz(q) * (a - b);
  }
  auto small = [](long long v) { return (unsigned)((int)(v >> 32) + 0x07000000) < 0x0e000000u; };
  return small(dev) && small(j[0]) && small(j[1]) && small(j[2]);
}

}  // namespace fsl
