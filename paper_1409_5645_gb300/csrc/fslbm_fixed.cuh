// fslbm_fixed.cuh -- the TRT collision of the FP64 form in 64-bit fixed point.
//
// GB300 issues two FP64 operations per cycle and SM against 64 or more 32-bit
// integer ones, and the FP64 collision (about 210 FP64 instructions a cell)
// kept the bulk kernel on that pipe at a seventh of the copy bandwidth.  The
// collision needs no floating exponent: in a cell of a flow near rho = 1
// every operand lies in (-8, 8), so it is done on 64-bit integers in units of
// 2^-60.  Sums are exact; a product (64 x 64 bits, the high word kept, rounded
// to nearest up to 0.6 unit) errs by at most about 2^-60.  An FP64 value in
// the range of the moving populations (2^-6 .. 2^-4) has a spacing of 2^-58 or
// 2^-57, so the result before its one rounding back to FP64 is nearer to the
// exact collision than a chain of FP64 operations comes (rms error over random
// states 5e-18 against 2.3e-17).  The weights are the FP64 values of 1/3, 1/18
// and 1/36, whose sum is 1 - 2^-54: with exact ones the density would not
// relax toward (1 - 2^-54) rho as it does in FP64, and a film's interface mass
// leaves the FP64 run's by 1e-15 of its value a step.
//
// A cell whose populations are not all in [0, 1/4) (rest: [0, 1)), whose
// momentum reaches 1/2, or whose result leaves [2^-28, 8) takes collide<double>
// (or, for the last, the hardware conversion): negative populations, NaN and
// states far from rho = 1 included.  Values below 2^-8 lose the bits under
// 2^-60, which FP64's own sums with their neighbours lose too.
#pragma once
#include <string.h>

#include "fslbm_dev.cuh"

namespace fsl {

// high 64 bits of a signed product, to about 0.6 unit: the low halves enter
// with 31 bits, and 3/4 of a unit stands for the mean of what is dropped
__host__ __device__ __forceinline__ long long mul_hi_near(long long a, long long b) {
  const int ah = (int)(a >> 32), bh = (int)(b >> 32);
  const int al = (int)((unsigned)a >> 1), bl = (int)((unsigned)b >> 1);
  const long long t = (long long)ah * bl + (long long)al * bh + 0x60000000LL;
  return (long long)ah * bh + (t >> 31);
}

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

// The collision in place: f <- f + l+ n^+ + l- n^- with the density sum f in
// units of 2^-60; fast = the speed guard's test (|u|^2 > u_max^2).  False, with
// f untouched, where the cell is out of range.
__host__ __device__ __forceinline__ bool collide_fixed(const Par& p, double (&f)[19], long long& rho, bool& fast) {
  if (!p.fix_ok) return false;
  unsigned top = 0u;  // (as unsigned, a negative value's or a NaN's high word is above the bound)
#pragma unroll
  for (int q = 1; q < 19; ++q) {
    const unsigned h = (unsigned)(bits_of_double(f[q]) >> 32);
    top = h > top ? h : top;
  }
  const unsigned h0 = (unsigned)(bits_of_double(f[0]) >> 32);
  bool ok = top < 0x3fd00000u && h0 < 0x3ff00000u;
  long long x[19];
#pragma unroll
  for (int q = 0; q < 19; ++q) x[q] = fix_of(bits_of_double(f[q]));
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
  // |j| < 1/2 (also bounds every product below)
  auto half = [](long long j) { return (unsigned)((int)(j >> 32) + 0x08000000) < 0x10000000u; };
  ok = ok && half(jx) && half(jy) && half(jz);
  if (!ok) return false;
  const long long ux = (jx + p.fx_hg[0]) << 2, uy = (jy + p.fx_hg[1]) << 2, uz = (jz + p.fx_hg[2]) << 2;
  const long long xx = mul_hi_near(ux, ux), yy = mul_hi_near(uy, uy), zz = mul_hi_near(uz, uz);
  const long long xy = mul_hi_near(ux, uy), xz = mul_hi_near(ux, uz), yz = mul_hi_near(uy, uz);
  const long long usq = xx + yy + zz;
  // fl(1/36), fl(1/3) and fl(3 fl(1/36)), units of 2^-64
  constexpr long long K36 = 0x071c71c71c71c700LL, K3 = 0x5555555555555400LL, K12 = 0x1555555555555500LL;
  // e^+ = w rho + 9/2 w (c.u)^2 - 3/2 w u.u: a = (rho - 3/2 u.u) / 36 is the
  // diagonal links' part (the axis links' twice that), 9/2 w = 1/8 and 1/4
  const long long dens = r - usq - (usq >> 1), a = mul_hi_near(dens, K36);
  // e^- = 3 w (c.u^eq): 1/12 of u^eq (diagonal links), twice that (axis links)
  const long long bx = mul_hi_near(jx - p.fx_gl[0], K12), by = mul_hi_near(jy - p.fx_gl[1], K12),
                  bz = mul_hi_near(jz - p.fx_gl[2], K12);
  x[0] += mul_hi_near(p.fx_lp, (x[0] - mul_hi_near(dens, K3)) << 2);
  long long low = x[0];
#pragma unroll
  for (int q = 1; q < 19; q += 2) {
    const int qb = q + 1;
    long long e2, m2;  // 2 e^+, 2 e^-
    if (q <= 6) {
      e2 = 4 * a + ((q == 1 ? xx : (q == 3 ? yy : zz)) >> 1);
      m2 = 4 * (q == 1 ? bx : (q == 3 ? by : bz));
    } else {
      const long long s = q <= 10 ? xx + yy : (q <= 14 ? xx + zz : yy + zz);
      const long long c = q <= 10 ? xy : (q <= 14 ? xz : yz);
      const bool same = cx(q) * cy(q) + cx(q) * cz(q) + cy(q) * cz(q) > 0;  // the two components' signs
      e2 = 2 * a + ((same ? s + 2 * c : s - 2 * c) >> 2);
      m2 = 2 * (cx(q) * bx + cy(q) * by + cz(q) * bz);
    }
    // the relaxations l+ n^+ and l- n^- (2 n in units of 2^-61)
    const long long rp = mul_hi_near(p.fx_lp, (x[q] + x[qb] - e2) << 1);
    const long long rm = mul_hi_near(p.fx_lm, (x[q] - x[qb] - m2) << 1);
    x[q] = x[q] + rp + rm;
    x[qb] = x[qb] + rp - rm;
    low = x[q] < low ? x[q] : low;
    low = x[qb] < low ? x[qb] : low;
  }
  if (low >= (1LL << 32)) {
#pragma unroll
    for (int q = 0; q < 19; ++q) f[q] = double_of_bits(bits_of(x[q]));
  } else {  // a negative or a tiny result
#pragma unroll
    for (int q = 0; q < 19; ++q) f[q] = double_of_fix(x[q]);
  }
  rho = r;
  fast = usq > p.fx_um2;
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
  bool ok = __all_sync(FULL, h < (q ? 0x3fd00000u : 0x3ff00000u));
  const long long x = ok ? fix_of(bits_of_double(f)) : 0;
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
  auto half = [](long long j) { return (unsigned)((int)(j >> 32) + 0x08000000) < 0x10000000u; };
  ok = ok && half(m[1]) && half(m[2]) && half(m[3]);  // (the same on every lane)
  if (!ok) return false;
  const long long ux = (m[1] + p.fx_hg[0]) << 2, uy = (m[2] + p.fx_hg[1]) << 2, uz = (m[3] + p.fx_hg[2]) << 2;
  const long long xx = mul_hi_near(ux, ux), yy = mul_hi_near(uy, uy), zz = mul_hi_near(uz, uz);
  const long long xy = mul_hi_near(ux, uy), xz = mul_hi_near(ux, uz), yz = mul_hi_near(uy, uz);
  const long long usq = xx + yy + zz, dens = m[0] - usq - (usq >> 1);
  constexpr long long K36 = 0x071c71c71c71c700LL, K3 = 0x5555555555555400LL, K12 = 0x1555555555555500LL;
  const long long a = mul_hi_near(dens, K36);
  const long long bx = mul_hi_near(m[1] - p.fx_gl[0], K12), by = mul_hi_near(m[2] - p.fx_gl[1], K12),
                  bz = mul_hi_near(m[3] - p.fx_gl[2], K12);
  const long long xb = __shfl_sync(FULL, x, qb);
  long long y;
  if (q == 0) {
    y = x + mul_hi_near(p.fx_lp, (x - mul_hi_near(dens, K3)) << 2);
  } else {
    // the odd link's terms, as collide_fixed takes them, on both lanes of a pair
    const int qo = (q & 1) ? q : qb;
    long long e2, m2;
    if (qo <= 6) {
      e2 = 4 * a + ((qo == 1 ? xx : (qo == 3 ? yy : zz)) >> 1);
      m2 = 4 * (qo == 1 ? bx : (qo == 3 ? by : bz));
    } else {
      const long long s = qo <= 10 ? xx + yy : (qo <= 14 ? xx + zz : yy + zz);
      const long long c = qo <= 10 ? xy : (qo <= 14 ? xz : yz);
      const int cxo = cx(qo), cyo = cy(qo), czo = cz(qo);
      const bool same = cxo * cyo + cxo * czo + cyo * czo > 0;
      e2 = 2 * a + ((same ? s + 2 * c : s - 2 * c) >> 2);
      m2 = 2 * (cxo * bx + cyo * by + czo * bz);
    }
    const long long d = (q & 1) ? x - xb : xb - x;
    const long long rp = mul_hi_near(p.fx_lp, (x + xb - e2) << 1), rm = mul_hi_near(p.fx_lm, (d - m2) << 1);
    y = x + rp + ((q & 1) ? rm : -rm);
  }
  // (both conversions round the same; a thread chooses one for its 19)
  f = y >= (1LL << 32) ? double_of_bits(bits_of(y)) : double_of_fix(y);
  rho = m[0];
  return true;
}
#endif

// density and momentum of populations in the collision's range, in units of
// 2^-60; false where they are not
__host__ __device__ __forceinline__ bool moments_fixed(const double (&f)[19], long long& rho, long long (&j)[3]) {
  unsigned top = 0u;
#pragma unroll
  for (int q = 1; q < 19; ++q) {
    const unsigned h = (unsigned)(bits_of_double(f[q]) >> 32);
    top = h > top ? h : top;
  }
  if (!(top < 0x3fd00000u && (unsigned)(bits_of_double(f[0]) >> 32) < 0x3ff00000u)) return false;
  rho = fix_of(bits_of_double(f[0]));
  j[0] = j[1] = j[2] = 0;
#pragma unroll
  for (int q = 1; q < 19; q += 2) {
    const long long a = fix_of(bits_of_double(f[q])), b = fix_of(bits_of_double(f[q + 1]));
    rho += a + b;
    j[0] += cx(q) * (a - b);
    j[1] += cy(q) * (a - b);
    j[2] += cz(q) * (a - b);
  }
  return true;
}

}  // namespace fsl
