// fslbm_slow.cuh -- a bulk cell's general path, out of line: the liquid cells
// of the segment masks' third word (next to a WALL cell, on a periodic face,
// CLI link fractions, a moving wall on a face), for the kernels that walk the
// masks (k_bulk_pairs, k_bulk_fixed).
#pragma once
#include "fslbm_dev.cuh"
#include "fslbm_fixed.cuh"
#include "fslbm_pull.cuh"

namespace fsl {

// k_bulk's test for a liquid cell whose sources are plain offsets or lie
// beyond a non-periodic face (bounce-back from its own slots)
__device__ __forceinline__ bool fast_cell(const Par& p, uint8_t fl, int x, int y, int z) {
  const bool ax = x == 0 || x == p.nx - 1, ay = y == 0 || y == p.ny - 1, az = z == 0 || z == p.nz - 1;
  if ((fl & KIND) != LIQ) return false;
  if (p.has_wd || p.has_uw) return !(fl & NEARB) && !ax && !ay && !az;
  return !(fl & NEARW) && !(ax && p.px) && !(ay && p.py) && !(az && p.pz);
}

// the general pull of k_bulk for one liquid cell (walls, periodic faces, CLI)
template <int P>
__device__ __forceinline__ void general_cell(const Par& p, const View<P>& v, long long i, int x, int y, int z,
                                             typename Form<P>::R (&f)[19]) {
  using R = typename Form<P>::R;
  const size_t N = (size_t)p.N;
  unsigned wallm, gasm, liqm;
  int srcs[19];
  f[0] = ld<P, 0>(v.fin, (size_t)i);
  pull_table<P>(p, v, x, y, z, f, wallm, gasm, liqm, srcs);
  if (gasm) atomicOr(v.err, ERRB_STATE);  // liquid must not touch gas
  wallm |= gasm;
  if (wallm) {
    R own[19];
#pragma unroll
    for (int q = 0; q < 19; ++q) own[q] = ldq<P>(v.fin, (size_t)q * N + (size_t)i, q);
    wall_links<P>(p, v, i, wallm, 0u, own, f);
  }
}

// One liquid cell of a segment that needs the general pull, as k_bulk
// treats it; returns its density for the mass balance (0 if not owned).
template <int P>
__device__ __noinline__ double slow_cell(const Par& p, const View<P>& v, long long i, int x, int y, int z,
                                         uint8_t fl) {
  using R = typename Form<P>::R;
  constexpr bool SH = Form<P>::SH;
  const size_t N = (size_t)p.N;
  const long long sy = p.nx, sz = (long long)p.nx * p.ny;
  R f[19];
  if (fast_cell(p, fl, x, y, z)) {
    // plain offsets, bounce-back beyond a non-periodic face
    const bool ax0 = x == 0, ax1 = x == p.nx - 1, ay0 = y == 0, ay1 = y == p.ny - 1, az0 = z == 0,
               az1 = z == p.nz - 1;
    f[0] = ld<P, 0>(v.fin, (size_t)i);
#pragma unroll
    for (int q = 1; q < 19; ++q) {
      const bool bbq = (cx(q) == 1 && ax0) || (cx(q) == -1 && ax1) || (cy(q) == 1 && ay0) || (cy(q) == -1 && ay1) ||
                       (cz(q) == 1 && az0) || (cz(q) == -1 && az1);
      f[q] = bbq ? ldq<P>(v.fin, (size_t)inv(q) * N + (size_t)i, inv(q))
                 : ldq<P>(v.fin, (size_t)q * N + (size_t)FSL_CK(p, i - (cx(q) + sy * cy(q) + sz * cz(q)), p.N), q);
    }
  } else {
    general_cell<P>(p, v, i, x, y, z, f);
  }
  R rho, ux, uy, uz;
  if constexpr (P == P64) {
    long long rf;
    bool over;
    if (collide_fixed(p, f, rf, over)) {
      if (over) atomicOr(v.err, ERRB_SPEED);
#pragma unroll
      for (int q = 0; q < 19; ++q) stq<P>(v.fout, (size_t)q * N + (size_t)i, q, f[q]);
      return owned(p, x, y, z) ? double_of_fix(rf) : 0.0;
    }
  }
  collide<R, SH>(p, f, rho, ux, uy, uz);
  if (rho_bad<SH>(rho)) atomicOr(v.err, ERRB_UNSTABLE);
  if (speed_bad(p, ux, uy, uz)) atomicOr(v.err, ERRB_SPEED);
#pragma unroll
  for (int q = 0; q < 19; ++q) stq<P>(v.fout, (size_t)q * N + (size_t)i, q, f[q]);
  return owned(p, x, y, z) ? rho_full<SH>(rho) : 0.0;
}

}  // namespace fsl
