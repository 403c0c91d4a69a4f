// fslbm_step.cuh -- the stream-collide kernels of one FSLBM time step (the
// segment scan k_segments, which lists the step's segments and interface
// cells before them, is in fslbm_step.cu).
//
// k_bulk   (FP32/FP16; the FP64 form's is in fslbm_bulk64.cu) every warp walks
//          the segment list on its own, one lane per cell.
//          Liquid cells pull their 19 populations (Eq. lbe1), apply half-way
//          bounce-back / CLI at walls, collide (Eq. lbe2) and store.  The
//          liquid density is reduced per warp for the mass balance.
// k_iface  one thread (short lists: one warp) per interface cell: pulls,
//          rebuilds the populations arriving from gas cells by the FSK rule
//          (Eq. koerner) or the FSL rule (Eq. closure, Table 1, D = 0) with the
//          link fraction from the height-function plane (Sec. 2.2, Sec. 5),
//          exchanges mass with its neighbours (Sec. 2.3), collides, stores, and
//          marks fill / empty conversions into compact lists.
//
// Templates over the precision form; each fslbm_step_p*.cu instantiates
// the launcher for one form, so that the forms compile in parallel.
#pragma once
#include "fslbm_dev.cuh"
#include "fslbm_fixed.cuh"
#include "fslbm_kernels.h"
#include "fslbm_pull.cuh"

namespace fsl {

// ---------------------------------------------------------------------------
// k_bulk: every warp walks the segment list on its own (no block barrier),
// one lane per cell; the liquid density is summed per warp.
// ---------------------------------------------------------------------------
template <int P>
__global__ void __launch_bounds__(128, 8) k_bulk(Par p, View<P> v, const int* __restrict__ seglist,
                                              const int* __restrict__ segcount) {
  pdl_begin();
  using R = typename Form<P>::R;
  const int nseg = *((volatile const int*)segcount);
  const int lane = threadIdx.x & 31;
  const int gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int nw = (gridDim.x * blockDim.x) >> 5;
  double msum = 0.0;
  for (int si = gw; si < nseg; si += nw) {
    const int4 sd = reinterpret_cast<const int4*>(seglist)[si];  // x0, y, z, first cell
    const int x = sd.x + lane, y = sd.y, z = sd.z;
    const bool in = x < p.nx;
    const long long i = FSL_CK_IF(p, in, (long long)sd.w + lane, p.N);
    const uint8_t fl = in ? v.flags[i] : (uint8_t)GAS;
    const uint8_t k = fl & KIND;
    const size_t N = (size_t)p.N;
    R f[19];
    // Fast path: every source is a fluid cell at a plain offset, or lies beyond
    // a non-periodic face (half-way bounce-back f_q = f~_qbar(x), read by
    // selecting the cell's own slot).  Cells next to a WALL cell, on a
    // periodic face, or with CLI link fractions take the general path.
    const bool ax0 = x == 0, ax1 = x == p.nx - 1, ay0 = y == 0, ay1 = y == p.ny - 1, az0 = z == 0,
               az1 = z == p.nz - 1;
    const bool onface = ax0 || ax1 || ay0 || ay1 || az0 || az1;
    const bool fast = k == LIQ &&
                      ((p.has_wd || p.has_uw) ? !(fl & NEARB) && !onface
                                : !(fl & NEARW) && !((ax0 || ax1) && p.px) && !((ay0 || ay1) && p.py) &&
                                      !((az0 || az1) && p.pz));
    const bool face_warp = __any_sync(0xffffffffu, fast && onface);
    if (k != LIQ) continue;
    if (fast && !face_warp) {
      const long long sy = p.nx, sz = (long long)p.nx * p.ny;
#define FSL_LD(q) \
  f[q] = ld<P, q>(v.fin, (size_t)q * N + (size_t)FSL_CK(p, i - (cx(q) + sy * cy(q) + sz * cz(q)), p.N));
      FSL_LD(0) FSL_LD(1) FSL_LD(2) FSL_LD(3) FSL_LD(4) FSL_LD(5) FSL_LD(6) FSL_LD(7) FSL_LD(8)
      FSL_LD(9) FSL_LD(10) FSL_LD(11) FSL_LD(12) FSL_LD(13) FSL_LD(14) FSL_LD(15) FSL_LD(16)
      FSL_LD(17) FSL_LD(18)
#undef FSL_LD
    } else if (fast) {
      const long long sy = p.nx, sz = (long long)p.nx * p.ny;
#define FSL_LDF(q)                                                                                              \
  {                                                                                                             \
    const bool bb = (cx(q) == 1 && ax0) || (cx(q) == -1 && ax1) || (cy(q) == 1 && ay0) || (cy(q) == -1 && ay1) || \
                    (cz(q) == 1 && az0) || (cz(q) == -1 && az1);                                                \
    const size_t k_ = bb ? (size_t)inv(q) * N + (size_t)i                                                       \
                         : (size_t)q * N + (size_t)FSL_CK(p, i - (cx(q) + sy * cy(q) + sz * cz(q)), p.N);      \
    f[q] = bb ? ld<P, inv(q)>(v.fin, k_) : ld<P, q>(v.fin, k_);                                                 \
  }
      f[0] = ld<P, 0>(v.fin, (size_t)i);
      FSL_LDF(1) FSL_LDF(2) FSL_LDF(3) FSL_LDF(4) FSL_LDF(5) FSL_LDF(6) FSL_LDF(7) FSL_LDF(8)
      FSL_LDF(9) FSL_LDF(10) FSL_LDF(11) FSL_LDF(12) FSL_LDF(13) FSL_LDF(14) FSL_LDF(15) FSL_LDF(16)
      FSL_LDF(17) FSL_LDF(18)
#undef FSL_LDF
    } else {
      unsigned wallm, gasm;
      f[0] = ld<P, 0>(v.fin, (size_t)i);
      pull_general<P>(p, v, x, y, z, f, wallm, gasm);
      if (gasm) atomicOr(v.err, ERRB_STATE);  // liquid must not touch gas
      wallm |= gasm;
      if (wallm) {
        R own[19];
#pragma unroll
        for (int q = 0; q < 19; ++q) own[q] = ldq<P>(v.fin, (size_t)q * N + (size_t)i, q);
        wall_links<P>(p, v, i, wallm, 0u, own, f);
      }
    }
    R rho, ux, uy, uz;
    collide<R, Form<P>::SH>(p, f, rho, ux, uy, uz);
    if (rho_bad<Form<P>::SH>(rho)) atomicOr(v.err, ERRB_UNSTABLE);
    if (speed_bad(p, ux, uy, uz)) atomicOr(v.err, ERRB_SPEED);
#define FSL_ST(q) st<P, q>(v.fout, (size_t)q * N + (size_t)i, f[q]);
    FSL_ST(0) FSL_ST(1) FSL_ST(2) FSL_ST(3) FSL_ST(4) FSL_ST(5) FSL_ST(6) FSL_ST(7) FSL_ST(8)
    FSL_ST(9) FSL_ST(10) FSL_ST(11) FSL_ST(12) FSL_ST(13) FSL_ST(14) FSL_ST(15) FSL_ST(16)
    FSL_ST(17) FSL_ST(18)
#undef FSL_ST
    if (owned(p, x, y, z)) msum += rho_full<Form<P>::SH>(rho);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) msum += __shfl_down_sync(0xffffffffu, msum, o);
  if (lane == 0) v.partials[gw] = msum;
}

// ---------------------------------------------------------------------------
// k_iface
// ---------------------------------------------------------------------------
// The work of one interface cell (pull, mass exchange, wall and gas-link
// closures, collision, store, fill/empty marks); returns its mass m.  IN:
// every cell within 3 of it lies inside the lattice, so all stencil offsets
// are plain (the hot path, kept apart from the face and wrap logic).
// Velocity of a fluid cell from its stored post-collision populations
// (sum_q c_q f~_q = rho_0 U + F, u = U + F/(2 rho_0)); only the FSL closure
// with u_b extrapolated along the link calls it (the extended k_iface instance).
template <class R>
struct Vel3 {
  R x, y, z;
};
template <int P>
__device__ __forceinline__ Vel3<typename Form<P>::R> cell_velocity(const typename Form<P>::S* __restrict__ fin,
                                                                 size_t N, size_t s, int compressible, double gx,
                                                                 double gy, double gz) {
  using R = typename Form<P>::R;
  R r = R(0), jx = R(0), jy = R(0), jz = R(0);
#pragma unroll
  for (int q = 0; q < 19; ++q) {
    const R fq = ldq<P>(fin, (size_t)q * N + s, q);
    r += fq;
    if (cx(q)) jx += R(cx(q)) * fq;
    if (cy(q)) jy += R(cy(q)) * fq;
    if (cz(q)) jz += R(cz(q)) * fq;
  }
  const R ir0 = compressible ? R(1) / rho_full_r<Form<P>::SH>(r) : R(1);
  return Vel3<R>{jx * ir0 - R(0.5) * R(gx), jy * ir0 - R(0.5) * R(gy), jz * ir0 - R(0.5) * R(gz)};
}

template <int P, bool IN, bool EXT>
__device__ __forceinline__ double iface_cell(const Par& p, const View<P>& v, int li, long long i, int x, int y,
                                             int z, bool& fill, bool& empty) {
  using R = typename Form<P>::R;
  const size_t N = (size_t)p.N;
  R own[19], f[19];
#pragma unroll
  for (int q = 0; q < 19; ++q) own[q] = ldq<P>(v.fin, (size_t)q * N + (size_t)i, q);
  constexpr bool SH = Form<P>::SH;
  R rt, utx, uty, utz;  // rt: rho(t), or rho(t) - 1 in the shifted forms
  moments_post<R, SH>(p, own, rt, utx, uty, utz);
  f[0] = own[0];
  unsigned wallm, gasm, liqm;
  int srcs[19];  // sources of the pull (only kept off the interior path)
  if constexpr (IN) pull_general<P, true>(p, v, x, y, z, f, wallm, gasm, &liqm);
  else pull_table<P>(p, v, x, y, z, f, wallm, gasm, liqm, srcs);
  const long long sy = p.nx, sz = (long long)p.nx * p.ny;
  const R phic = v.phin[i];
  // mass exchange (Sec. 2.3) with the pulled values, before any rebuild
  double dm = 0.0;
  if (!p.freeze) {
#pragma unroll
    for (int q = 1; q < 19; ++q) {
      if ((wallm | gasm) & (1u << q)) continue;
      const long long sq = IN ? i - (cx(q) + sy * cy(q) + sz * cz(q)) : (long long)srcs[q];
      const R phs = v.phin[sq];  // (loaded whatever the kind, so the loads overlap)
      R sw = (liqm & (1u << q)) ? R(1) : R(0.5) * (phic + phs);
      dm += (double)(sw * (f[q] - own[inv(q)]));
    }
  }
  if (wallm) wall_links<P>(p, v, i, wallm, gasm, own, f);
  if (gasm || (EXT && p.recon_nc)) {
    // the plane and curvature of k_geom (FSK without surface tension, the
    // boundary shear term or the normal links needs neither)
    R n[3] = {R(0), R(0), R(0)}, d = R(0), kap = R(0);
    if (p.rule != 0 || p.sigma != 0.0 || (EXT && (p.stress || p.recon_nc))) {
      const size_t cap = (size_t)v.cap;
      n[0] = v.geo[li];
      n[1] = v.geo[cap + li];
      n[2] = v.geo[2 * cap + li];
      d = v.geo[3 * cap + li];
      kap = v.geo[4 * cap + li];
    }
    const bool ok = true;  // no normal is stored as n = 0: c.n > 0 fails and delta stays 1/2
    // links to rebuild: the gas links, and with recon_nc the links p toward a
    // fluid node with n.c_p > 0 (Koerner et al.'s reconstruction along the
    // normal; margin 1e-6 for links tangent to the surface)
    unsigned rmask = gasm;
    R pulled[19];  // the pulled values, kept apart from the rebuilt ones
    if (EXT && p.recon_nc) {
#pragma unroll
      for (int q = 1; q < 19; ++q) {
        pulled[q] = f[q];
        const int pq = inv(q);
        const R cn = R(cx(pq)) * n[0] + R(cy(pq)) * n[1] + R(cz(pq)) * n[2];
        if (!((wallm | gasm) & (1u << q)) && cn > R(1e-6)) rmask |= 1u << q;
      }
    }
    R rb = R(p.rho_G);
    if (p.sigma != 0.0) rb = rb + R(3.0 * p.sigma) * kap;
    const R r0b = p.compressible ? rb : R(1);
    const R r0t = p.compressible ? rho_full_r<SH>(rt) : R(1);
    if (SH) rb = rb - R(1);  // e^+ below in the arithmetic of the stored values
    const R usq = utx * utx + uty * uty + utz * utz;
    const R lp = R(p.lam_p);
    // boundary shear rate S^b of Eq. bterm (stress mode): S from the cell's
    // own non-equilibrium part, sum_q c_qa c_qb n_q^+ = (2 c_s^2 / lambda_+) S_ab
    // (leading order of Eq. nqp), with its normal-tangential components set to
    // zero in the basis of the normal (Eq. proj2 through Eq. bstress):
    // S^b = S - (S n) n^T - n (S n)^T + 2 (n.S.n) n n^T
    R Sb[6] = {R(0), R(0), R(0), R(0), R(0), R(0)};  // xx yy zz xy xz yz
    if (EXT && p.stress == 2) {  // prescribed S^b
#pragma unroll
      for (int k = 0; k < 6; ++k) Sb[k] = R(p.shear_b[k]);
    } else if (EXT && p.stress) {
#pragma unroll
      for (int q = 1; q < 19; q += 2) {  // each pair once: n_q^+ = n_qbar^+
        const R et = eplus_q<R>(p, q, rt, r0t, utx, uty, utz, usq);
        const R np2 = R(2) * (R(0.5) * (own[q] + own[q + 1]) - et) * R(p.inv_1plp);
        Sb[0] += R(cx(q) * cx(q)) * np2; Sb[1] += R(cy(q) * cy(q)) * np2; Sb[2] += R(cz(q) * cz(q)) * np2;
        Sb[3] += R(cx(q) * cy(q)) * np2; Sb[4] += R(cx(q) * cz(q)) * np2; Sb[5] += R(cy(q) * cz(q)) * np2;
      }
#pragma unroll
      for (int k = 0; k < 6; ++k) Sb[k] *= R(1.5) * lp;
      const R Sn0 = Sb[0] * n[0] + Sb[3] * n[1] + Sb[4] * n[2];
      const R Sn1 = Sb[3] * n[0] + Sb[1] * n[1] + Sb[5] * n[2];
      const R Sn2 = Sb[4] * n[0] + Sb[5] * n[1] + Sb[2] * n[2];
      const R snn = n[0] * Sn0 + n[1] * Sn1 + n[2] * Sn2;
      Sb[0] += R(2) * (snn * n[0] * n[0] - Sn0 * n[0]);
      Sb[1] += R(2) * (snn * n[1] * n[1] - Sn1 * n[1]);
      Sb[2] += R(2) * (snn * n[2] * n[2] - Sn2 * n[2]);
      Sb[3] += R(2) * snn * n[0] * n[1] - Sn0 * n[1] - n[0] * Sn1;
      Sb[4] += R(2) * snn * n[0] * n[2] - Sn0 * n[2] - n[0] * Sn2;
      Sb[5] += R(2) * snn * n[1] * n[2] - Sn1 * n[2] - n[1] * Sn2;
    }
    const R Dk = R(-3.0 * (p.tau_m_half));  // D = -alpha_+ Lambda_+ w_p / c_s^2, without alpha_+ w_p
#pragma unroll
    for (int q = 1; q < 19; ++q) {
      if (!(rmask & (1u << q))) continue;
      const int pq = inv(q);  // boundary link: x + c_p is gas (or a normal link), rebuilt f_pbar = f_q
      R eb = eplus_q<R>(p, pq, rb, r0b, utx, uty, utz, usq);
      bool up_fluid = !((wallm | gasm) & (1u << pq));
      // D c_p.S^b.c_p / alpha_+ (Eq. bterm, Table 1)
      R dterm = R(0);
      if (EXT && p.stress) {
        const R cSc = R(cx(pq) * cx(pq)) * Sb[0] + R(cy(pq) * cy(pq)) * Sb[1] + R(cz(pq) * cz(pq)) * Sb[2] +
                      R(2 * cx(pq) * cy(pq)) * Sb[3] + R(2 * cx(pq) * cz(pq)) * Sb[4] +
                      R(2 * cy(pq) * cz(pq)) * Sb[5];
        dterm = Dk * wq<R>(pq) * cSc;
      }
      if (p.rule == 0 || !up_fluid) {
        f[q] = -own[pq] + R(2) * eb + R(2) * dterm;  // FSK, Eq. koerner (alpha_+ = 2)
      } else {
        R dl = R(0.5);
        if (ok) {
          R cn = R(cx(pq)) * n[0] + R(cy(pq)) * n[1] + R(cz(pq)) * n[2];
          if (cn > R(0)) {
            dl = qdiv(d, cn);
            dl = dl < R(p.delta_min) ? R(p.delta_min) : (dl > R(1) ? R(1) : dl);
          }
        }
        if (EXT && p.ub_extrap) {
          // u_b at the surface point x_b + delta c_p, linear along the link
          // through u(x_b) and u(x_b - c_p)
          const long long su = IN ? i - (cx(pq) + sy * cy(pq) + sz * cz(pq)) : (long long)srcs[pq];
          const Vel3<R> uu = cell_velocity<P>(v.fin, N, (size_t)su, p.compressible, p.g[0], p.g[1], p.g[2]);
          const R wx = utx + dl * (utx - uu.x), wy = uty + dl * (uty - uu.y), wz = utz + dl * (utz - uu.z);
          eb = eplus_q<R>(p, pq, rb, r0b, wx, wy, wz, wx * wx + wy * wy + wz * wz);
        }
        R et = eplus_q<R>(p, pq, rt, r0t, utx, uty, utz, usq);
        R nplus = (R(0.5) * (own[pq] + own[q]) - et) * R(p.inv_1plp);
        R C = lp * (R(0.5) + dl) - R(2) * lp;
        const R fup = (EXT && p.recon_nc) ? pulled[pq] : f[pq];  // f~_p(x_b - c_p)
        f[q] = (R(0.5) - dl) * own[pq] + R(0.5) * own[q] + (dl - R(1)) * fup + C * nplus + eb + dterm;
      }
    }
  }
  R rho, ux, uy, uz;
  collide<R, SH>(p, f, rho, ux, uy, uz);
  // (the velocity guard is the liquid cells': an isolated interface cell of
  // the spray, with a few fluid neighbours, carries spurious speeds of 0.4
  // and more in a stable flow)
  if (rho_bad<SH>(rho)) atomicOr(v.err, ERRB_UNSTABLE);
#pragma unroll
  for (int q = 0; q < 19; ++q) stq<P>(v.fout, (size_t)q * N + (size_t)i, q, f[q]);
  double mm = v.m[i];
  if (!p.freeze) {
    const double rhof = rho_full<SH>(rho);
    mm = mm + dm;
    v.m[i] = mm;
    v.phout[i] = (R)(mm / rhof);
    // thresholds, plus the isolated-cell rules: no gas neighbour -> fill,
    // no liquid/interface neighbour -> empty
    fill = mm > (1.0 + p.eps) * rhof || ((p.cleanup & 1) && gasm == 0u);
    empty = !fill && (mm < -p.eps * rhof || ((p.cleanup & 2) && (wallm | gasm) == 0x7fffeu));
    if (fill) v.mark[i] = MK_FILL;  // marks are zero between steps; each cell writes only its own
    else if (empty) v.mark[i] = MK_EMPTY;
  }
  return mm;
}

// The FP64 form's default interface cell.  Its FP64 pipe (two operations a
// cycle and SM) bounds it, so the arithmetic is laid out for few of them: the
// equilibria, the non-equilibrium part and the quotient d / (n.c) are taken
// once per link pair (a pair has at most one link with the FSL closure: its
// upstream node must be fluid), both directions of a pair run the same
// instructions on selected operands, and the collision is the fixed-point one.
// It comes for a thread per cell and, where the list is short, for a warp per
// cell with a link per lane; the roundings are written out (but a wall link's,
// where both leave the one product and sum to the compiler), so the two give
// the same bits and the choice does not show; the tests of the two paths hold
// that for every closure.
//
// c . a for a link with components 0 or +-1 (one rounding, of the sum)
__device__ __forceinline__ double link_dot(int ax, int ay, int az, const double (&a)[3]) {
  return fx_fma((double)ax, a[0], fx_fma((double)ay, a[1], fx_mul((double)az, a[2])));
}

__device__ __forceinline__ float link_dot32(int ax, int ay, int az, float a0, float a1, float a2) {
  return fx_fma((float)ax, a0, fx_fma((float)ay, a1, fx_mul((float)az, a2)));
}

// what the links of a cell share
struct Surface64 {
  double n[3], d;        // the plane of k_geom
  double rb, rt;         // rho_b and rho(t)
  double r0b, r0t;       // rho_0 beside them
  double u[3], usq, nl;  // u_b, its square, 0 for the linear equilibrium
};

// The closure of the pair of links q (components a) and its opposite qb:
// o / ob the cell's own populations, f / fb the pulled ones, ga / gb whether
// they come from gas, blocked whether from gas or a wall; w the weight.
// Rebuilds f and fb.
__device__ __forceinline__ void gas_pair64(const Par& p, const Surface64& S, double w, int ax, int ay, int az, double o,
                                           double ob, bool ga, bool gb, bool ba, bool bb, double& f, double& fb) {
  // e^+ of both directions: w rho + 3/2 w rho_0 (3 (c.u)^2 - u.u)
  const double cu = link_dot(ax, ay, az, S.u);
  const double k = fx_mul(fx_mul(S.nl, fx_mul(1.5, w)), fx_fma(fx_mul(3.0, cu), cu, -S.usq));
  const double eb = fx_fma(S.r0b, k, fx_mul(w, S.rb));
  // FSL (Table 1): the rebuilt population's own link has a fluid upstream node
  const bool fa = p.rule != 0 && ga && !bb, fo = p.rule != 0 && gb && !ba;
  double val = 0.0;
  if (fa || fo) {
    const double hs = fx_mul(0.5, fx_add(o, ob));
    const double nplus = fx_mul(fx_sub(hs, fx_fma(S.r0t, k, fx_mul(w, S.rt))), p.inv_1plp);
    const double op = fa ? ob : o, fup = fa ? fb : f;
    const double cq = link_dot(ax, ay, az, S.n), cn = fa ? -cq : cq;
    double dl = 0.5;
    if (cn > 0.0) {
      dl = __ddiv_rn(S.d, cn);
      dl = dl < p.delta_min ? p.delta_min : (dl > 1.0 ? 1.0 : dl);
    }
    val = fx_add(fx_add(fx_sub(hs, fup), eb), fx_fma(dl, fx_sub(fup, op), fx_mul(fx_mul(p.lam_p, fx_sub(dl, 1.5)), nplus)));
  }
  const double ska = fx_fma(2.0, eb, -ob), skb = fx_fma(2.0, eb, -o);  // FSK, Eq. koerner
  if (ga) f = fa ? val : ska;
  if (gb) fb = fo ? val : skb;
}

// plane, densities and velocity of a cell from its geometry and the moments of
// its own populations
__device__ __forceinline__ void surface64(const Par& p, const View<P64>& v, int li, double rt, const double (&j)[3],
                                          Surface64& S) {
  S.n[0] = S.n[1] = S.n[2] = S.d = 0.0;
  S.rb = p.rho_G;
  if (p.rule != 0 || p.sigma != 0.0) {
    const size_t cap = (size_t)v.cap;
    S.n[0] = v.geo[li];
    S.n[1] = v.geo[cap + li];
    S.n[2] = v.geo[2 * cap + li];
    S.d = v.geo[3 * cap + li];
    S.rb = fx_fma(fx_mul(3.0, p.sigma), v.geo[4 * cap + li], S.rb);
  }
  S.rt = rt;
  S.r0t = p.compressible ? rt : 1.0;
  S.r0b = p.compressible ? S.rb : 1.0;
#pragma unroll
  for (int a = 0; a < 3; ++a) S.u[a] = fx_fma(-0.5, p.g[a], p.compressible ? __ddiv_rn(j[a], rt) : j[a]);
  S.usq = fx_fma(S.u[2], S.u[2], fx_fma(S.u[1], S.u[1], fx_mul(S.u[0], S.u[0])));
  S.nl = p.linear_eq ? 0.0 : 1.0;
}

// the cell's new mass and fill level and its conversion marks (one thread)
__device__ __forceinline__ double finish64(const Par& p, const View<P64>& v, long long i, double dm, double rho,
                                           unsigned wallm, unsigned gasm, bool& fill, bool& empty) {
  double mm = v.m[i];
  if (!p.freeze) {
    mm = fx_add(mm, dm);
    v.m[i] = mm;
    v.phout[i] = __ddiv_rn(mm, rho);
    fill = mm > fx_mul(1.0 + p.eps, rho) || ((p.cleanup & 1) && gasm == 0u);
    empty = !fill && (mm < fx_mul(-p.eps, rho) || ((p.cleanup & 2) && (wallm | gasm) == 0x7fffeu));
    if (fill) v.mark[i] = MK_FILL;
    else if (empty) v.mark[i] = MK_EMPTY;
  }
  return mm;
}

template <bool IN>
__device__ __forceinline__ double iface_cell64(const Par& p, const View<P64>& v, int li, long long i, int x, int y,
                                               int z, bool& fill, bool& empty) {
  const size_t N = (size_t)p.N;
  double own[19], f[19];
#pragma unroll
  for (int q = 0; q < 19; ++q) own[q] = v.fin[(size_t)q * N + (size_t)i];
  f[0] = own[0];
  unsigned wallm, gasm, liqm;
  int srcs[19];  // sources of the pull (only kept off the interior path)
  if constexpr (IN) pull_general<P64, true>(p, v, x, y, z, f, wallm, gasm, &liqm);
  else pull_table<P64>(p, v, x, y, z, f, wallm, gasm, liqm, srcs);
  const long long sy = p.nx, sz = (long long)p.nx * p.ny;
  const double phic = v.phin[i];
  double dm = 0.0;  // mass exchange (Sec. 2.3), twice its value
  if (!p.freeze) {
#pragma unroll
    for (int q = 1; q < 19; ++q) {
      if ((wallm | gasm) & (1u << q)) continue;
      const long long sq = IN ? FSL_CK(p, i - (cx(q) + sy * cy(q) + sz * cz(q)), p.N) : (long long)srcs[q];
      const double phs = v.phin[sq];
      dm = fx_fma((liqm & (1u << q)) ? 2.0 : fx_add(phic, phs), fx_sub(f[q], own[inv(q)]), dm);
    }
    dm = fx_mul(0.5, dm);
  }
  if (wallm) wall_links<P64>(p, v, i, wallm, gasm, own, f);
  if (gasm) {
    double rt = own[0], j[3] = {0.0, 0.0, 0.0};
#pragma unroll
    for (int q = 1; q < 19; q += 2) {
      const double s = fx_add(own[q], own[q + 1]), e = fx_sub(own[q], own[q + 1]);
      rt = fx_add(rt, s);
      if (cx(q)) j[0] = fx_add(j[0], cx(q) * e);
      if (cy(q)) j[1] = fx_add(j[1], cy(q) * e);
      if (cz(q)) j[2] = fx_add(j[2], cz(q) * e);
    }
    Surface64 S;
    surface64(p, v, li, rt, j, S);
    const unsigned blocked = wallm | gasm;
#pragma unroll
    for (int q = 1; q < 19; q += 2) {
      const int qb = q + 1;
      const bool ga = (gasm >> q) & 1u, gb = (gasm >> qb) & 1u;
      if (ga || gb)
        gas_pair64(p, S, q <= 6 ? 1.0 / 18.0 : 1.0 / 36.0, cx(q), cy(q), cz(q), own[q], own[qb], ga, gb,
                   (blocked >> q) & 1u, (blocked >> qb) & 1u, f[q], f[qb]);
    }
  }
  double rho;
  long long rf;
  bool over;
  if (collide_fixed(p, f, rf, over)) {
    rho = double_of_fix(rf);
  } else {
    double ux, uy, uz;
    collide<double>(p, f, rho, ux, uy, uz);
    if (rho_bad<false>(rho)) atomicOr(v.err, ERRB_UNSTABLE);
  }
#pragma unroll
  for (int q = 0; q < 19; ++q) v.fout[(size_t)q * N + (size_t)i] = f[q];
  return finish64(p, v, i, dm, rho, wallm, gasm, fill, empty);
}

// A cell by a warp, link q on lane q (the lanes from 19 on repeat the rest
// population and write nothing); fill, empty and the returned mass are lane 0's.
__device__ __forceinline__ double iface_warp64(const Par& p, const View<P64>& v, int li, long long i, int x, int y,
                                               int z, bool& fill, bool& empty) {
  const unsigned FULL = 0xffffffffu;
  const size_t N = (size_t)p.N;
  const int lane = threadIdx.x & 31, q = lane < 19 ? lane : 0, qb = q == 0 ? 0 : ((q & 1) ? q + 1 : q - 1);
  const int ax = cx(q), ay = cy(q), az = cz(q);
  const long long s = nbr(p, x, y, z, -ax, -ay, -az);
  const uint8_t ks = kind_at(v.flags, s);
  const double own = v.fin[(size_t)q * N + (size_t)i];
  double f = v.fin[(size_t)q * N + (size_t)(s < 0 ? 0 : s)];
  const double phic = v.phin[i], phs = s < 0 ? 0.0 : v.phin[s];
  if (!is_fluid(ks)) f = 0.0;
  const bool link = lane >= 1 && lane < 19;
  const unsigned wallm = __ballot_sync(FULL, link && ks == WALL);
  const unsigned gasm = __ballot_sync(FULL, link && ks != WALL && !is_fluid(ks));
  const unsigned blocked = wallm | gasm;
  const double ownb = __shfl_sync(FULL, own, qb);
  double dm = 0.0;
  if (!p.freeze) {
    const double wgt = ks == LIQ ? 2.0 : fx_add(phic, phs), dif = fx_sub(f, ownb);
#pragma unroll
    for (int l = 1; l < 19; ++l) {  // in link order, as a thread sums it
      const double a = __shfl_sync(FULL, wgt, l), b = __shfl_sync(FULL, dif, l);
      if (!((blocked >> l) & 1u)) dm = fx_fma(a, b, dm);
    }
    dm = fx_mul(0.5, dm);
  }
  double fb = __shfl_sync(FULL, f, qb);  // the opposite link's pulled value
  if ((wallm >> q) & 1u) {  // (wall_links)
    double val = ownb;
    if (p.has_wd) {
      const double dw = v.wd[(size_t)qb * N + (size_t)i];
      if (dw >= 0.0 && !((blocked >> qb) & 1u)) {
        const double kap = (1.0 - 2.0 * dw) / (1.0 + 2.0 * dw);
        val = val + kap * (fb - own);
      }
    } else if (p.has_uw) {
      val = val + 6.0 * (q <= 6 ? 1.0 / 18.0 : 1.0 / 36.0) * (ax * p.wall_u[0] + ay * p.wall_u[1] + az * p.wall_u[2]);
    }
    f = val;
  }
  if (gasm) {
    double rt = __shfl_sync(FULL, own, 0), j[3] = {0.0, 0.0, 0.0};
    const double sum = fx_add(own, ownb), dif = (q & 1) ? fx_sub(own, ownb) : 0.0;
#pragma unroll
    for (int l = 1; l < 19; l += 2) {
      const double e = __shfl_sync(FULL, dif, l);
      rt = fx_add(rt, __shfl_sync(FULL, sum, l));
      if (cx(l)) j[0] = fx_add(j[0], cx(l) * e);
      if (cy(l)) j[1] = fx_add(j[1], cy(l) * e);
      if (cz(l)) j[2] = fx_add(j[2], cz(l) * e);
    }
    Surface64 S;
    surface64(p, v, li, rt, j, S);
    // both lanes of a pair run its closure, as the thread does from the odd link
    const bool odd = (q & 1) != 0;
    const int sg = odd ? 1 : -1, qo = odd ? q : qb, qe = odd ? qb : q;
    double fo = odd ? f : fb, fe = odd ? fb : f;
    const bool ga = q && ((gasm >> qo) & 1u), gb = q && ((gasm >> qe) & 1u);
    if (ga || gb) {
      gas_pair64(p, S, q <= 6 ? 1.0 / 18.0 : 1.0 / 36.0, sg * ax, sg * ay, sg * az, odd ? own : ownb, odd ? ownb : own,
                 ga, gb, (blocked >> qo) & 1u, (blocked >> qe) & 1u, fo, fe);
      if ((gasm >> q) & 1u) f = odd ? fo : fe;
    }
  }
  double rho;
  long long rf;
  if (!collide_warp(p, q, f, rf)) {  // out of the fixed-point range: as a thread, on every lane
    double g[19], ux, uy, uz;
#pragma unroll
    for (int l = 0; l < 19; ++l) g[l] = __shfl_sync(FULL, f, l);
    collide<double>(p, g, rho, ux, uy, uz);
    if (lane == 0 && rho_bad<false>(rho)) atomicOr(v.err, ERRB_UNSTABLE);
#pragma unroll
    for (int l = 0; l < 19; ++l) f = l == q ? g[l] : f;
  } else {
    rho = double_of_fix(rf);
  }
  if (lane < 19) v.fout[(size_t)q * N + (size_t)i] = f;
  return lane == 0 ? finish64(p, v, i, dm, rho, wallm, gasm, fill, empty) : 0.0;
}

// The default interface cell of the FP32 and FP16 forms by a warp, link q on
// lane q (the lanes from 19 on repeat the rest population and write nothing):
// the operations of iface_cell<P, ., false>, sums in its order.  The roundings
// are written out here as the compiler takes them there (written out there too,
// the thread's kernel was slower: 100 steps of a 128x64x64 FP32 splash 8.16 ->
// 8.34 ms); the tests of the two paths hold them to the same bits for every
// closure.  fill, empty and the returned mass are lane 0's.
template <int P>
__device__ __forceinline__ double iface_warp32(const Par& p, const View<P>& v, int li, long long i, int x, int y, int z,
                                               bool& fill, bool& empty) {
  static_assert(sizeof(typename Form<P>::R) == 4 && Form<P>::SH, "the reduced forms");
  const unsigned FULL = 0xffffffffu;
  const size_t N = (size_t)p.N;
  const int lane = threadIdx.x & 31, q = lane < 19 ? lane : 0, qb = q == 0 ? 0 : ((q & 1) ? q + 1 : q - 1);
  const int ax = cx(q), ay = cy(q), az = cz(q);
  const long long s = nbr(p, x, y, z, -ax, -ay, -az);
  const uint8_t ks = kind_at(v.flags, s);
  const float own = ldq<P>(v.fin, (size_t)q * N + (size_t)i, q);
  float f = ldq<P>(v.fin, (size_t)q * N + (size_t)(s < 0 ? 0 : s), q);
  const float phic = v.phin[i], phs = s < 0 ? 0.f : v.phin[s];
  if (!is_fluid(ks)) f = 0.f;
  const bool link = lane >= 1 && lane < 19;
  const unsigned wallm = __ballot_sync(FULL, link && ks == WALL);
  const unsigned gasm = __ballot_sync(FULL, link && ks != WALL && !is_fluid(ks));
  const unsigned blocked = wallm | gasm;
  const float ownb = __shfl_sync(FULL, own, qb);
  double dm = 0.0;
  if (!p.freeze) {
    const float sw = ks == LIQ ? 1.f : fx_mul(0.5f, fx_add(phic, phs)), flux = fx_mul(sw, fx_sub(f, ownb));
#pragma unroll
    for (int l = 1; l < 19; ++l) {
      const float a = __shfl_sync(FULL, flux, l);
      if (!((blocked >> l) & 1u)) dm += (double)a;
    }
  }
  const float fb = __shfl_sync(FULL, f, qb);  // the opposite link's pulled value
  if ((wallm >> q) & 1u) {                    // (wall_links)
    float val = ownb;
    if (p.has_wd) {
      const float dw = (float)v.wd[(size_t)qb * N + (size_t)i];
      if (dw >= 0.f && !((blocked >> qb) & 1u)) {
        const float kap = __fdiv_rn(fx_fma(-2.f, dw, 1.f), fx_fma(2.f, dw, 1.f));
        val = fx_fma(kap, fx_sub(fb, own), val);
      }
    } else if (p.has_uw) {
      const float w6 = 6.f * (q <= 6 ? wq<float>(1) : wq<float>(7));
      val = fx_fma(w6, link_dot32(ax, ay, az, (float)p.wall_u[0], (float)p.wall_u[1], (float)p.wall_u[2]), val);
    }
    f = val;
  }
  if (gasm) {
    // the moments of the cell's own populations
    float rt = 0.f, ux = 0.f, uy = 0.f, uz = 0.f;
#pragma unroll
    for (int l = 0; l < 19; ++l) {
      const float a = __shfl_sync(FULL, own, l);
      rt = fx_add(rt, a);
      if (cx(l)) ux = cx(l) > 0 ? fx_add(ux, a) : fx_sub(ux, a);
      if (cy(l)) uy = cy(l) > 0 ? fx_add(uy, a) : fx_sub(uy, a);
      if (cz(l)) uz = cz(l) > 0 ? fx_add(uz, a) : fx_sub(uz, a);
    }
    const float ir0 = p.compressible ? 1.f / rho_full_r<true>(rt) : 1.f;
    ux = fx_fma(ux, ir0, -fx_mul(0.5f, (float)p.g[0]));
    uy = fx_fma(uy, ir0, -fx_mul(0.5f, (float)p.g[1]));
    uz = fx_fma(uz, ir0, -fx_mul(0.5f, (float)p.g[2]));
    float n0 = 0.f, n1 = 0.f, n2 = 0.f, d = 0.f, kap = 0.f;
    if (p.rule != 0 || p.sigma != 0.0) {
      const size_t cap = (size_t)v.cap;
      n0 = v.geo[li];
      n1 = v.geo[cap + li];
      n2 = v.geo[2 * cap + li];
      d = v.geo[3 * cap + li];
      kap = v.geo[4 * cap + li];
    }
    float rb = (float)p.rho_G;
    if (p.sigma != 0.0) rb = fx_fma((float)(3.0 * p.sigma), kap, rb);
    const float r0b = p.compressible ? rb : 1.f, r0t = p.compressible ? rho_full_r<true>(rt) : 1.f;
    rb = fx_sub(rb, 1.f);
    if ((gasm >> q) & 1u) {
      // boundary link p = qb (x + c_p is gas), rebuilt f_q
      const float usq = fx_fma(uz, uz, fx_fma(ux, ux, fx_mul(uy, uy))), w = q <= 6 ? wq<float>(1) : wq<float>(7);
      const float cu = link_dot32(-ax, -ay, -az, ux, uy, uz);
      float eb = fx_mul(w, rb), et = fx_mul(w, rt);
      if (!p.linear_eq) {
        const float t = fx_fma(fx_mul(3.f, cu), cu, -usq);
        eb = fx_fma(fx_mul(fx_mul(w, 1.5f), r0b), t, eb);
        et = fx_fma(fx_mul(fx_mul(w, 1.5f), r0t), t, et);
      }
      if (p.rule == 0 || ((blocked >> qb) & 1u)) {
        f = fx_fma(2.f, eb, -ownb);
      } else {
        float dl = 0.5f;
        const float cn = link_dot32(-ax, -ay, -az, n0, n1, n2);
        if (cn > 0.f) {
          dl = qdiv(d, cn);
          dl = dl < (float)p.delta_min ? (float)p.delta_min : (dl > 1.f ? 1.f : dl);
        }
        const float nplus = fx_mul(fx_fma(0.5f, fx_add(ownb, own), -et), (float)p.inv_1plp), lp = (float)p.lam_p;
        const float C = fx_fma(lp, fx_add(0.5f, dl), -fx_mul(2.f, lp));
        float r = fx_fma(fx_sub(0.5f, dl), ownb, fx_mul(0.5f, own));
        r = fx_fma(fx_sub(dl, 1.f), fb, r);
        r = fx_fma(C, nplus, r);
        f = fx_add(r, eb);
      }
    }
  }
  // the collision (collide): moments in population order, then the link's pair
  float r, jx = 0.f, jy = 0.f, jz = 0.f;
  r = __shfl_sync(FULL, f, 0);
#pragma unroll
  for (int l = 1; l < 19; ++l) {
    const float a = __shfl_sync(FULL, f, l);
    r = fx_add(r, a);
    if (cx(l)) jx = cx(l) > 0 ? fx_add(jx, a) : fx_sub(jx, a);
    if (cy(l)) jy = cy(l) > 0 ? fx_add(jy, a) : fx_sub(jy, a);
    if (cz(l)) jz = cz(l) > 0 ? fx_add(jz, a) : fx_sub(jz, a);
  }
  const float fo = __shfl_sync(FULL, f, qb);
  const float r0 = p.compressible ? rho_full_r<true>(r) : 1.f, i0 = p.compressible ? 1.f / r0 : 1.f;
  const float Ux = fx_mul(jx, i0), Uy = fx_mul(jy, i0), Uz = fx_mul(jz, i0);
  const float gx = (float)p.g[0], gy = (float)p.g[1], gz = (float)p.g[2], ilm = (float)p.inv_lam_m;
  const float ux = fx_fma(0.5f, gx, Ux), uy = fx_fma(0.5f, gy, Uy), uz = fx_fma(0.5f, gz, Uz);
  const float vx = fx_fma(-gx, ilm, Ux), vy = fx_fma(-gy, ilm, Uy), vz = fx_fma(-gz, ilm, Uz);
  const float usq = fx_fma(uz, uz, fx_fma(uy, uy, fx_mul(ux, ux)));
  const float lp = (float)p.lam_p, lm = (float)p.lam_m, nl = p.linear_eq ? 0.f : 1.f;
  const float w = q == 0 ? wq<float>(0) : (q <= 6 ? wq<float>(1) : wq<float>(7));
  const float kw = fx_mul(fx_mul(1.5f * w, r0), nl);
  float out;
  if (q == 0) {
    out = fx_fma(lp, fx_sub(f, fx_fma(kw, -usq, fx_mul(w, r))), f);
  } else {
    constexpr float m7f = 1.f / 12.f, m1f = (1.f - 8.f * m7f) * 0.5f;
    const float mw = fx_mul(q <= 6 ? m1f : m7f, r0);
    const bool odd = (q & 1) != 0;
    const int sg = odd ? 1 : -1;  // (the pair's terms from its odd link)
    const float fq = odd ? f : fo, fqb = odd ? fo : f;
    const float cu = link_dot32(sg * ax, sg * ay, sg * az, ux, uy, uz);
    const float cv = link_dot32(sg * ax, sg * ay, sg * az, vx, vy, vz);
    const float ep = fx_fma(kw, fx_fma(fx_mul(3.f, cu), cu, -usq), fx_mul(w, r)), em = fx_mul(mw, cv);
    const float np = fx_fma(0.5f, fx_add(fq, fqb), -ep), nm = fx_fma(0.5f, fx_sub(fq, fqb), -em);
    out = fx_fma(odd ? lm : -lm, nm, fx_fma(lp, np, f));
  }
  if (lane < 19) stq<P>(v.fout, (size_t)q * N + (size_t)i, q, out);
  if (lane != 0) return 0.0;
  if (rho_bad<true>(r)) atomicOr(v.err, ERRB_UNSTABLE);
  double mm = v.m[i];
  if (!p.freeze) {
    const double rhof = rho_full<true>(r);
    mm = mm + dm;
    v.m[i] = mm;
    v.phout[i] = (float)(mm / rhof);
    fill = mm > (1.0 + p.eps) * rhof || ((p.cleanup & 1) && gasm == 0u);
    empty = !fill && (mm < -p.eps * rhof || ((p.cleanup & 2) && blocked == 0x7fffeu));
    if (fill) v.mark[i] = MK_FILL;
    else if (empty) v.mark[i] = MK_EMPTY;
  }
  return mm;
}

// ---------------------------------------------------------------------------
// k_geom: plane (normal, offset) and curvature of every listed interface cell
// from phi(t) (Sec. 2.2, Sec. 5) into v.geo; kept apart from k_iface so that
// each kernel holds fewer registers and less code.
//
// A thread per cell has the higher throughput (its 89 samples and their sums
// are about 1700 instructions for 32 cells) but is a chain of that length,
// 25 to 35 us however few cells there are; a warp per cell spends about 550
// instructions on one cell and is done with it in 3 to 5 us.  So each end of
// the list, the interior cells and the edge cells (within 3 of a face, whose
// samples need the neighbour rule), takes a thread per cell above
// geom_warp_max cells and a warp per cell up to it; in FP64 the line is lower,
// as a warp's finish holds the FP64 pipe as long for one cell as for 32.
// Alone, with warm caches, thread -> warp: 16 FP64 cells of a 4x4x32 film 94
// -> 13 us, 12.7 k FP32 cells of a 128x64x64 splash 28 -> 16 us, 17.4 k cells
// with curvature of a 128^3 FP16 wave 93 -> 33 us; 57 k FP64 cells by threads
// 55 us.
// ---------------------------------------------------------------------------
template <int P>
constexpr int geom_warp_max() { return P == P64 ? 2432 : 49152; }
// SIG: the instance that also computes the curvature (surface tension); ELV:
// the one with the ELVIRA normal where the height columns are open
// The thread path waits for the gathers of its cell, so blocks in flight beside
// the bulk kernel count for more than registers: 10 an SM for FP16 (48 registers,
// from 64 and 128: a pass of a 128^3 wave 5.02 -> 4.79 ms, of a 512x256x256 splash
// 17.36 -> 17.23) and 9 for plain FP32 (56: 19.38 -> 19.08).  FP64 keeps the
// compiler's choice (5 blocks: a splash 7.26 -> 7.37 ms), FP32 with surface tension
// or the elevation form has no measurement for a bound (0: none).
template <int P, bool SIG, bool ELV>
__global__ void __launch_bounds__(128, P == P16 ? 10 : P == P64 || SIG || ELV ? 0 : 9) k_geom(Par p, View<P> v) {
  pdl_begin();
  using R = typename Form<P>::R;
  const int n_in = min(*((volatile int*)&v.cnt[0]), v.cap), n_edge = min(*((volatile int*)&v.cnt[6]), v.cap - n_in);
  const size_t cap = (size_t)v.cap;
  auto put = [&](int pos, const Geo<R>& G) {
    v.geo[pos] = G.ok ? G.n[0] : R(0);
    v.geo[cap + pos] = G.ok ? G.n[1] : R(0);
    v.geo[2 * cap + pos] = G.ok ? G.n[2] : R(0);
    v.geo[3 * cap + pos] = G.d;
    v.geo[4 * cap + pos] = G.kap;
  };
  // interior cells at the front of the list, edge cells at the back
  const int t_in = n_in > geom_warp_max<P>() ? n_in : 0, t_edge = n_edge > geom_warp_max<P>() ? n_edge : 0;
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < t_in + t_edge; e += gridDim.x * blockDim.x) {
    const bool in3 = e < t_in;
    const int pos = in3 ? e : v.cap - 1 - (e - t_in);
    const long long i = FSL_CK(p, v.ilist[pos], p.N);
    int x, y, z;
    coords(p, i, x, y, z);
    if (!FSL_OK(p, !in3 || (x >= 3 && x < p.nx - 3 && y >= 3 && y < p.ny - 3 && z >= 3 && z < p.nz - 3))) continue;
    const R phic = v.phin[i];
    Geo<R> G;  // (in registers)
    if (in3) geometry<R, 1, SIG, ELV>(p, v.flags, v.phin, x, y, z, phic, G);
    else if (!p.px && !p.py && !p.pz) geometry<R, 2, SIG, ELV>(p, v.flags, v.phin, x, y, z, phic, G);
    else geometry<R, 0, SIG, ELV>(p, v.flags, v.phin, x, y, z, phic, G);
    put(pos, G);
  }
  // a warp per cell, from the grid's last warps on
  const int w_in = n_in - t_in, nc = w_in + n_edge - t_edge;
  const int lane = threadIdx.x & 31, warps = (gridDim.x * blockDim.x) >> 5;
  const int wid = warps - 1 - (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
  for (int e = wid; e < nc; e += warps) {
    const bool in3 = e < w_in;
    const int pos = in3 ? e : v.cap - 1 - (e - w_in);
    const long long i = FSL_CK(p, v.ilist[pos], p.N);
    int x, y, z;
    coords(p, i, x, y, z);
    if (!FSL_OK(p, !in3 || (x >= 3 && x < p.nx - 3 && y >= 3 && y < p.ny - 3 && z >= 3 && z < p.nz - 3))) continue;
    const R phic = v.phin[i];
    Geo<R> G;
    R nn, kopen;
    const bool ok = coop_stencil<R, SIG>(p, v.flags, v.phin, x, y, z, in3, (int)i, phic, nn, kopen, G);
    if (ok) coop_finish<R, SIG, ELV>(p, v.flags, v.phin, x, y, z, phic, nn, kopen, G);
    if (lane == 0) put(pos, G);
  }
}

// EXT: the instance with the boundary shear-rate term, the extrapolated u_b
// and the normal links (separate, so that the default instance carries none
// of their code).  LEAN: the FP64 form's instance with few FP64 operations
// (where the fixed-point collision applies)
//
// A list of up to IFACE_WARP_MAX cells goes by a warp per cell, a longer one by
// a thread per cell: the thread is a chain of 20 to 24 us however few cells
// there are, the warp one of 11.5 us (16 FP64 cells of a 4x4x32 film, alone,
// warm caches).  The line lies at 8 cells an SM: a warp's FP64 operations (in
// the reduced forms those of the cell's mass) hold the FP64 pipe as long for
// one cell as for 32, and 12.7 k FP32 cells of a 128x64x64 splash took 74 us by
// warps against 20 us by threads.
constexpr int IFACE_WARP_MAX = 152 * 8;
template <int P, bool EXT, bool LEAN = false>
__global__ void __launch_bounds__(128, (EXT ? 2 : (P == P64 ? 3 : 5))) k_iface(Par p, View<P> v, int part_base) {
  pdl_begin();
  const int n_in = min(*((volatile int*)&v.cnt[0]), v.cap), n_edge = min(*((volatile int*)&v.cnt[6]), v.cap);
  const int count = min(n_in + n_edge, v.cap);
  const int stride = gridDim.x * blockDim.x;
  const int rounds = (count + stride - 1) / stride;
  double msum = 0.0;
  // a short list by a warp per cell (the default instances)
  constexpr bool WARP = LEAN || (P != P64 && !EXT);
  const bool warp = WARP && count <= IFACE_WARP_MAX;
  if constexpr (WARP) {
    if (warp) {
      const int lane = threadIdx.x & 31;
      for (int e = (threadIdx.x >> 5) * gridDim.x + blockIdx.x; e < count; e += (blockDim.x >> 5) * gridDim.x) {
        const int pos = e < n_in ? e : v.cap - 1 - (e - n_in);
        const long long i = FSL_CK(p, v.ilist[pos], p.N);
        int x, y, z;
        coords(p, i, x, y, z);
        bool fill = false, empty = false;
        double mm;
        if constexpr (P == P64) mm = iface_warp64(p, v, pos, i, x, y, z, fill, empty);
        else mm = iface_warp32<P>(p, v, pos, i, x, y, z, fill, empty);
        if (lane == 0 && owned(p, x, y, z)) msum += mm;
        warp_append(lane == 0 && fill, (int)i, v.flist, &v.cnt[1], v.cap, v.err);
        warp_append(lane == 0 && empty, (int)i, v.elist, &v.cnt[2], v.cap, v.err);
      }
    }
  }
  for (int r = 0; r < rounds; ++r) {
    if (warp) break;
    const int li = r * stride + blockIdx.x * blockDim.x + threadIdx.x;
    const bool act = li < count;
    bool fill = false, empty = false;
    int icell = 0;
    if (act) {
      const bool in3 = li < n_in;  // interior cells at the front, edge cells at the back
      const int pos = in3 ? li : v.cap - 1 - (li - n_in);
      const long long i = FSL_CK(p, v.ilist[pos], p.N);
      icell = (int)i;
      int x, y, z;
      coords(p, i, x, y, z);
      if (FSL_OK(p, !in3 || (x >= 3 && x < p.nx - 3 && y >= 3 && y < p.ny - 3 && z >= 3 && z < p.nz - 3))) {
        double mm;
        if constexpr (LEAN) {
          mm = in3 ? iface_cell64<true>(p, v, pos, i, x, y, z, fill, empty)
                   : iface_cell64<false>(p, v, pos, i, x, y, z, fill, empty);
        } else {
          mm = in3 ? iface_cell<P, true, EXT>(p, v, pos, i, x, y, z, fill, empty)
                   : iface_cell<P, false, EXT>(p, v, pos, i, x, y, z, fill, empty);
        }
        if (owned(p, x, y, z)) msum += mm;
      }
    }
    warp_append(fill, icell, v.flist, &v.cnt[1], v.cap, v.err);
    warp_append(empty, icell, v.elist, &v.cnt[2], v.cap, v.err);
  }
  // per-warp partial sums, after the bulk warps' ones
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) msum += __shfl_down_sync(0xffffffffu, msum, o);
  if ((threadIdx.x & 31) == 0) v.partials[part_base + ((blockIdx.x * blockDim.x + threadIdx.x) >> 5)] = msum;
}

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------
// a launch without the programmatic-serialization attribute (after a wait
// on another stream's event)
template <typename... KArgs, typename... Args>
inline int launch_plain(void (*kernel)(KArgs...), unsigned grid, unsigned block, cudaStream_t st, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(block);
  cfg.stream = st;
  return (int)cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}

template <int P>
int launch_step_kernels(const Par& p, const View<P>& v, cudaStream_t st, int bulk_blocks, int iface_blocks,
                        int* seglist, int* segcount, void* timing_handle, int bulk_mode,
                        const CUtensorMap* tmap, const Fork* fork) {
  if (launch_segments(p, v.flags, seglist, segcount, v.ilist, v.cnt, v.cap, v.err, st))
    return 1;
  // the interface geometry reads phi(t), the flags and the interface list of
  // the segment scan, and writes only its scratch: it runs on the side stream
  // beside the bulk kernel.  Beside the pair kernel (whose grid then leaves
  // room on every SM) the interface kernel follows it there: it reads f~(t),
  // phi(t), m and the flags, and writes the interface cells' populations, m,
  // phi(t+1), marks and lists, none of which the bulk kernel touches
  const bool geo = p.rule != 0 || p.sigma != 0.0 || p.stress || p.recon_nc;
  auto kgeo = p.elvira ? (p.sigma != 0.0 ? k_geom<P, true, true> : k_geom<P, false, true>)
                       : (p.sigma != 0.0 ? k_geom<P, true, false> : k_geom<P, false, false>);
  auto kif = (p.stress || p.ub_extrap || p.recon_nc) ? k_iface<P, true> : k_iface<P, false>;
  if constexpr (P == P64) {
    if (p.fix_ok && !(p.stress || p.ub_extrap || p.recon_nc)) kif = k_iface<P, false, true>;
  }
  const bool pairs = P != P64 && bulk_mode == BULK_PAIRS;
  const bool side_geo = geo && fork;
  const bool side_if = (pairs || P == P64) && fork;
  if (side_geo || side_if) {
    if (cudaEventRecord(fork->fork, st) != cudaSuccess) return 1;
    if (cudaStreamWaitEvent(fork->side, fork->fork, 0) != cudaSuccess) return 1;
    if (side_geo && launch_plain(kgeo, iface_blocks, 128, fork->side, p, v)) return 1;
    // the interface partials follow the bulk warps' ones
    if (side_if && launch_plain(kif, iface_blocks, 128, fork->side, p, v, bulk_blocks * 4)) return 1;
    if (cudaEventRecord(fork->join, fork->side) != cudaSuccess) return 1;
  }
  if (timing_handle && fslbm_mark(timing_handle, 0)) return 1;  // the bulk group times the bulk kernel alone
  bool launched = false;
  if constexpr (P != P64) {
    if (bulk_mode == BULK_TMA && tmap) {
      if (launch_bulk_tma<P>(p, v, tmap, st, bulk_blocks, seglist, segcount)) return 1;
      launched = true;
    } else if (bulk_mode == BULK_ASYNC) {
      if (launch_bulk_async<P>(p, v, st, bulk_blocks, seglist, segcount)) return 1;
      launched = true;
    } else if (bulk_mode == BULK_PAIRS) {
      if (launch_bulk_pairs<P>(p, v, st, bulk_blocks, seglist, segcount, side_if)) return 1;
      launched = true;
    }
  }
  if constexpr (P == P64) {
    if (launch_bulk_fixed(p, v, st, bulk_blocks, seglist, segcount)) return 1;
  } else {
    if (!launched && launch_k(k_bulk<P>, bulk_blocks, 128, 0, st, p, v, (const int*)seglist, (const int*)segcount))
      return 1;
  }
  if (timing_handle && fslbm_mark(timing_handle, 1)) return 1;
  if (geo && !side_geo && launch_k(kgeo, iface_blocks, 128, 0, st, p, v)) return 1;
  if (side_geo || side_if) {
    if (cudaStreamWaitEvent(st, fork->join, 0) != cudaSuccess) return 1;
  }
  if (!side_if) {
    if (side_geo ? launch_plain(kif, iface_blocks, 128, st, p, v, bulk_blocks * 4)
                 : launch_k(kif, iface_blocks, 128, 0, st, p, v, bulk_blocks * 4))
      return 1;
  }
  return (int)cudaGetLastError();
}

}  // namespace fsl
