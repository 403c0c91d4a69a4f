// fslbm_pull.cuh -- device helpers of the stream step shared by the bulk
// kernels: the warp-aggregated list append, the general pull next to walls,
// faces and gas, and the wall closures.
#pragma once
#include "fslbm_dev.cuh"

namespace fsl {

// ---------------------------------------------------------------------------
// warp-aggregated append of `pred` lanes' values to list[*count ...]
// (all 32 lanes of the warp must call it)
// ---------------------------------------------------------------------------
__device__ __forceinline__ void warp_append(bool pred, int value, int* list, int* count, int cap, int* err) {
  unsigned bal = __ballot_sync(0xffffffffu, pred);
  if (!bal) return;
  int lane = threadIdx.x & 31;
  int leader = __ffs(bal) - 1;
  int base = 0;
  if (lane == leader) base = atomicAdd(count, __popc(bal));
  base = __shfl_sync(0xffffffffu, base, leader);
  if (pred) {
    int k = base + __popc(bal & ((1u << lane) - 1u));
    if (k < cap) list[k] = value;
    else atomicOr(err, ERRB_OVERFLOW);
  }
}

// ---------------------------------------------------------------------------
// General pull for a cell next to a wall, a face or gas.  Fills f[q] from
// fluid sources and returns masks of wall and gas sources.
// ---------------------------------------------------------------------------
template <int P, bool IN = false>
__device__ __forceinline__ void pull_general(const Par& p, const View<P>& v, int x, int y, int z,
                                             typename Form<P>::R (&f)[19], unsigned& wallm, unsigned& gasm,
                                             unsigned* liqm = nullptr) {
  const size_t N = (size_t)p.N;
  wallm = 0u;
  gasm = 0u;
  unsigned lm = 0u;
  // away from the faces the sources are plain offsets
  // (IN: the caller knows the cell is at least one cell away from every face)
  const bool in1 = IN || (x >= 1 && x < p.nx - 1 && y >= 1 && y < p.ny - 1 && z >= 1 && z < p.nz - 1);
  const long long i = (long long)x + (long long)p.nx * ((long long)y + (long long)p.ny * z);
  const long long sy = p.nx, sz = (long long)p.nx * p.ny;
  if constexpr (IN) {
    // every source lies inside the lattice: issue the population and flag
    // loads together (a gas source's stale populations are read and dropped)
#pragma unroll
    for (int q = 1; q < 19; ++q) {
      const long long s = i - (cx(q) + sy * cy(q) + sz * cz(q));
      const uint8_t ks = v.flags[s] & KIND;
      const typename Form<P>::R fq = ldq<P>(v.fin, (size_t)q * N + (size_t)s, q);
      if (is_fluid(ks)) {
        f[q] = fq;
        if (ks == LIQ) lm |= 1u << q;
      } else if (ks == WALL) { wallm |= 1u << q; f[q] = 0; }
      else { gasm |= 1u << q; f[q] = 0; }
    }
  } else {
    // a lattice without periodic axes: a source past a face is a wall
    const bool bounded = !p.px && !p.py && !p.pz;
#pragma unroll
    for (int q = 1; q < 19; ++q) {
      long long s;
      if (in1) {
        s = i - (cx(q) + sy * cy(q) + sz * cz(q));
      } else if (bounded) {
        const bool inside = (unsigned)(x - cx(q)) < (unsigned)p.nx && (unsigned)(y - cy(q)) < (unsigned)p.ny &&
                            (unsigned)(z - cz(q)) < (unsigned)p.nz;
        s = inside ? i - (cx(q) + sy * cy(q) + sz * cz(q)) : -1;
      } else {
        s = nbr(p, x, y, z, -cx(q), -cy(q), -cz(q));
      }
      uint8_t ks = kind_at(v.flags, s);
      if (is_fluid(ks)) {
        f[q] = ldq<P>(v.fin, (size_t)q * N + (size_t)s, q);
        if (ks == LIQ) lm |= 1u << q;
      } else if (ks == WALL) { wallm |= 1u << q; f[q] = 0; }
      else { gasm |= 1u << q; f[q] = 0; }
    }
  }
  if (liqm) *liqm = lm;
}

// The sources x - c_q of a cell's pull, -1 past a non-periodic face: each axis'
// three neighbour coordinates (the x wrap shifts z) are taken once and a source
// is the sum of three of them.  (nbr() unrolled 18 times is over a thousand
// instructions.)
__device__ __forceinline__ void pull_sources(const Par& p, int x, int y, int z, int (&srcs)[19]) {
  int xo[3], yo[3], zo[3][3];
  bool xv[3], yv[3], zv[3][3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    int X = x + k - 1, Y = y + k - 1, sh = 0;
    if (p.px) {
      if (X < 0) { X += p.nx; sh = p.zshift; }
      else if (X >= p.nx) { X -= p.nx; sh = -p.zshift; }
    }
    if (p.py) Y += Y < 0 ? p.ny : (Y >= p.ny ? -p.ny : 0);
    xo[k] = X;
    xv[k] = (unsigned)X < (unsigned)p.nx;
    yo[k] = Y * p.nx;
    yv[k] = (unsigned)Y < (unsigned)p.ny;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      int Z = z + c - 1 + sh;
      if (p.pz) Z += Z < 0 ? p.nz : (Z >= p.nz ? -p.nz : 0);
      zv[k][c] = (unsigned)Z < (unsigned)p.nz;
      zo[k][c] = Z * (p.nx * p.ny);
    }
  }
  srcs[0] = xo[1] + yo[1] + zo[1][1];
#pragma unroll
  for (int q = 1; q < 19; ++q) {
    const int ka = 1 - cx(q), kb = 1 - cy(q), kc = 1 - cz(q);
    srcs[q] = xv[ka] && yv[kb] && zv[ka][kc] ? xo[ka] + yo[kb] + zo[ka][kc] : -1;
  }
}

// The pull of a cell that may lie on a face, for the interface kernel's edge
// cells and the bulk kernels' out-of-line cells, which a warp meets one at a
// time: sources from pull_sources, kinds and populations loaded together
// (pull_general loads a population after its source's kind).
template <int P>
__device__ __forceinline__ void pull_table(const Par& p, const View<P>& v, int x, int y, int z,
                                           typename Form<P>::R (&f)[19], unsigned& wallm, unsigned& gasm,
                                           unsigned& liqm, int (&srcs)[19]) {
  const size_t N = (size_t)p.N;
  pull_sources(p, x, y, z, srcs);
  wallm = gasm = liqm = 0u;
#pragma unroll
  for (int q = 1; q < 19; ++q) {
    const bool in = srcs[q] >= 0;
    const int s = in ? srcs[q] : 0;
    const uint8_t ks = in ? (uint8_t)(v.flags[s] & KIND) : (uint8_t)WALL;
    const typename Form<P>::R fq = ldq<P>(v.fin, (size_t)q * N + (size_t)s, q);
    f[q] = is_fluid(ks) ? fq : typename Form<P>::R(0);
    if (ks == LIQ) liqm |= 1u << q;
    else if (ks == WALL) wallm |= 1u << q;
    else if (ks != IFC) gasm |= 1u << q;
  }
}

// Wall closure for the links in wallm (needs the cell's own f~ and the
// pulled values): half-way bounce-back f_q = f~_p(x), p = qbar, or CLI with
// kappa = (1 - 2 dw)/(1 + 2 dw): f_q = f~_p(x) + kappa (f~_p(x - c_p) - f~_q(x)),
// where f~_p(x - c_p) is the value pulled along p (used only if that source is
// fluid).
template <int P>
__device__ __forceinline__ void wall_links(const Par& p, const View<P>& v, long long i, unsigned wallm,
                                           unsigned gasm, const typename Form<P>::R (&own)[19],
                                           typename Form<P>::R (&f)[19]) {
  using R = typename Form<P>::R;
  const size_t N = (size_t)p.N;
#pragma unroll
  for (int q = 1; q < 19; ++q) {
    if (!(wallm & (1u << q))) continue;
    const int pq = inv(q);
    R val = own[pq];
    if (p.has_wd) {
      R dw = (R)v.wd[(size_t)pq * N + (size_t)i];
      bool up_fluid = !((wallm | gasm) & (1u << pq));
      if (dw >= R(0) && up_fluid) {
        R kap = (R(1) - R(2) * dw) / (R(1) + R(2) * dw);
        val = val + kap * (f[pq] - own[q]);
      }
    } else if (p.has_uw) {
      // moving wall (half-way bounce-back): + 6 w_q rho_0 (c_q.u_w), rho_0 = 1
      val = val + R(6) * wq<R>(q) *
                      (R(cx(q)) * R(p.wall_u[0]) + R(cy(q)) * R(p.wall_u[1]) + R(cz(q)) * R(p.wall_u[2]));
    }
    f[q] = val;
  }
}

}  // namespace fsl
