// fslbm_conv.cuh -- the stages of the cell conversions as device functions
// over whatever grid calls them (fslbm_conv.cu describes them), with the grid
// barrier and the mass reduction of the kernels that run them in one launch.
#pragma once
#include "fslbm_dev.cuh"
#include "fslbm_fixed.cuh"
#include "fslbm_kernels.h"
#include "fslbm_pull.cuh"

namespace fsl {

__device__ __forceinline__ uint8_t or_u8(uint8_t* base, long long j, unsigned bits) {
  unsigned* w = (unsigned*)(base + (j & ~3LL));
  unsigned sh = (unsigned)(j & 3) * 8u;
  unsigned old = atomicOr(w, bits << sh);
  return (uint8_t)(old >> sh);
}
__device__ __forceinline__ void clear_u8(uint8_t* base, long long j, unsigned bits) {
  unsigned* w = (unsigned*)(base + (j & ~3LL));
  unsigned sh = (unsigned)(j & 3) * 8u;
  atomicAnd(w, ~(bits << sh));
}
// append `value` for every converged lane with `pred`, one atomic per warp
__device__ __forceinline__ void push(bool pred, int* list, int* count, int cap, int value, int* err) {
  const unsigned act = __activemask();
  const unsigned bal = __ballot_sync(act, pred);
  if (!bal) return;
  const int lane = threadIdx.x & 31, leader = __ffs(bal) - 1;
  int base = 0;
  if (lane == leader) base = atomicAdd(count, __popc(bal));
  base = __shfl_sync(act, base, leader);
  if (pred) {
    int k = base + __popc(bal & ((1u << lane) - 1u));
    if (k < cap) list[k] = value;
    else atomicOr(err, ERRB_OVERFLOW);
  }
}
__device__ __forceinline__ int load_count(const int* c) { return *((volatile const int*)c); }

// density of cell i at t+1 (summed in q order in the arithmetic type)
template <int P>
__device__ __forceinline__ double rho_out(const Par& p, const View<P>& v, long long i) {
  using R = typename Form<P>::R;
  R r = R(0);
#pragma unroll
  for (int q = 0; q < 19; ++q) r += ldq<P>(v.fout, (size_t)q * (size_t)p.N + (size_t)i, q);
  return rho_full<Form<P>::SH>(r);
}

// fill cell k by a warp, lane q (1..18) takes link q
template <int P>
__device__ __forceinline__ void fill_cell(const Par& p, const View<P>& v, int k) {
  const int lane = threadIdx.x & 31;
  const int q = (lane >= 1 && lane < 19) ? lane : 0;
  {
    const long long i = FSL_CK(p, v.flist[k], p.N);
    int x, y, z;
    coords(p, i, x, y, z);
    bool won = false;
    long long j = -1;
    if (q) {
      j = nbr(p, x, y, z, cx(q), cy(q), cz(q));
      const uint8_t kj = j < 0 ? (uint8_t)WALL : (uint8_t)(v.flags[j] & KIND);
      if (kj == GAS) {
        const uint8_t old = or_u8(v.mark, j, MK_NEWG);
        won = !(old & MK_NEWG);  // the first claimant lists the new cell
      }
    }
    push(won, v.nglist, &v.cnt[3], v.cap, (int)j, v.err);
  }
}
// The FP64 form's new cell from its neighbours' fixed-point moments (rho - 1,
// j; lanes with `use`): f^eq of the means, collided; lane q builds population q.
// The sums are exact (moments_fixed).  The cell's density and momentum are the
// means themselves (the weights' sums), as a sum over the lanes would give
// them back up to rounding.
__device__ __forceinline__ void newg_fixed(const Par& p, const View<P64>& v, long long j, int q, bool use,
                                           long long dev, const long long (&xj)[3]) {
  const unsigned FULL = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  long long m[4] = {use ? dev : 0, use ? xj[0] : 0, use ? xj[1] : 0, use ? xj[2] : 0};
  const int c = __popc(__ballot_sync(FULL, use));
#pragma unroll
  for (int o = 16; o > 0; o >>= 1)
#pragma unroll
    for (int k = 0; k < 4; ++k) m[k] += __shfl_xor_sync(FULL, m[k], o);
  // (a mean a lane: one FP64 division and conversion for the four)
  const int l = lane & 3;
  const double mean = double_of_fix(l == 0 ? m[0] : (l == 1 ? m[1] : (l == 2 ? m[2] : m[3]))) / (double)c;
  const double rho = 1.0 + __shfl_sync(FULL, mean, 0);
  const double u0 = __shfl_sync(FULL, mean, 1) - 0.5 * p.g[0], u1 = __shfl_sync(FULL, mean, 2) - 0.5 * p.g[1],
               u2 = __shfl_sync(FULL, mean, 3) - 0.5 * p.g[2];
  const double w = q == 0 ? 1.0 / 3.0 : (q <= 6 ? 1.0 / 18.0 : 1.0 / 36.0);
  const double ax = cx(q), ay = cy(q), az = cz(q);
  const double cu = ax * u0 + ay * u1 + az * u2, usq = u0 * u0 + u1 * u1 + u2 * u2;
  const double fp = w * rho + (w * 1.5) * (3.0 * cu * cu - usq), fm = 3.0 * w * cu;  // even and odd part of f^eq
  // the collision moves them toward e^+(u + g/2) and e^-(u - g/lambda_-)
  const double cg = ax * p.g[0] + ay * p.g[1] + az * p.g[2];
  const double ug = u0 * p.g[0] + u1 * p.g[1] + u2 * p.g[2], gg = p.g[0] * p.g[0] + p.g[1] * p.g[1] + p.g[2] * p.g[2];
  const double np = w * 1.5 * ((ug + 0.25 * gg) - 3.0 * cg * (cu + 0.25 * cg));  // f^+ - e^+
  const double nm = 3.0 * w * cg * p.inv_lam_m;                                   // f^- - e^-
  if (lane < 19) v.fout[(size_t)q * (size_t)p.N + (size_t)j] = (fp + p.lam_p * np) + (fm + p.lam_m * nm);
  if (lane == 0) {
    v.m[j] = 0.0;
    v.phout[j] = 0.0;
  }
}

// new cell k by a warp: lane l (1..18) reads neighbour l's populations; the
// means are summed in neighbour order; lane q builds and collides population q
template <int P>
__device__ __forceinline__ void newg_cell(const Par& p, const View<P>& v, int k) {
  using R = typename Form<P>::R;
  const unsigned FULL = 0xffffffffu;
  const size_t N = (size_t)p.N;
  const int lane = threadIdx.x & 31;
  const int q = lane < 19 ? lane : 0;
  {
    const long long j = FSL_CK(p, v.nglist[k], p.N);
    int x, y, z;
    coords(p, j, x, y, z);
    bool use = false, range = true;
    R rr = R(0), ux = R(0), uy = R(0), uz = R(0);
    long long xr = 0, xj[3] = {0, 0, 0};  // the neighbour's rho - 1 and j in fixed point (FP64 form)
    if (lane >= 1 && lane < 19) {
      long long y2 = nbr(p, x, y, z, cx(q), cy(q), cz(q));
      if (y2 >= 0) {
        // the populations are loaded beside the flag (a gas cell's are read and dropped)
        R g[19];
#pragma unroll
        for (int r = 0; r < 19; ++r) g[r] = ldq<P>(v.fout, (size_t)r * N + (size_t)y2, r);
        use = is_fluid(v.flags[y2] & KIND);
        if (use) {
          if constexpr (P == P64) {
            range = p.fix_ok && moments_fixed(g, xr, xj);
            if (!range) moments_post<R, Form<P>::SH>(p, g, rr, ux, uy, uz);
          } else {
            moments_post<R, Form<P>::SH>(p, g, rr, ux, uy, uz);
          }
        }
      }
    }
    if constexpr (P == P64) {
      // every neighbour in range: the sums are exact in any order, and the FP64
      // pipe (which bounded the stage) sees four conversions
      if (__all_sync(FULL, range)) {
        newg_fixed(p, v, j, q, use, xr, xj);
        return;
      }
      if (use && range) {
        rr = 1.0 + double_of_fix(xr);
        ux = double_of_fix(xj[0]) - 0.5 * p.g[0];
        uy = double_of_fix(xj[1]) - 0.5 * p.g[1];
        uz = double_of_fix(xj[2]) - 0.5 * p.g[2];
      }
    }
    R rs = R(0), s0 = R(0), s1 = R(0), s2 = R(0);
    int c = 0;
#pragma unroll
    for (int l = 1; l < 19; ++l) {
      const bool ul = __shfl_sync(FULL, use, l);
      const R a = __shfl_sync(FULL, rr, l), b0 = __shfl_sync(FULL, ux, l);
      const R b1 = __shfl_sync(FULL, uy, l), b2 = __shfl_sync(FULL, uz, l);
      if (ul) { rs += a; s0 += b0; s1 += b1; s2 += b2; ++c; }
    }
    // (rbar is rho - 1 in the shifted forms: the mean of rho - 1)
    R rbar, u0, u1, u2;
    if constexpr (P == P64) {  // (one FP64 division for four: they bound the FP64 form's stage)
      const R dc = R(c), ic = R(1) / dc;
      rbar = quot_near(rs, dc, ic);
      u0 = quot_near(s0, dc, ic);
      u1 = quot_near(s1, dc, ic);
      u2 = quot_near(s2, dc, ic);
    } else {
      rbar = rs / R(c); u0 = s0 / R(c); u1 = s1 / R(c); u2 = s2 / R(c);
    }
    const R r0 = p.compressible ? rho_full_r<Form<P>::SH>(rbar) : R(1);
    const R usq = u0 * u0 + u1 * u1 + u2 * u2;
    const R wq_ = q == 0 ? R(1) / R(3) : (q <= 6 ? R(1) / R(18) : R(1) / R(36));
    // f^eq(rbar, ubar) with u^eq = ubar
    const R f = eplus_q<R>(p, q, rbar, r0, u0, u1, u2, usq) +
                R(3) * wq_ * r0 * (R(cx(q)) * u0 + R(cy(q)) * u1 + R(cz(q)) * u2);
    // collision (Eq. lbe2) of the new cell, lane q -> population q
    const R f19 = lane < 19 ? f : R(0);
    R rho = f19, jx = R(cx(q)) * f19, jy = R(cy(q)) * f19, jz = R(cz(q)) * f19;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      rho += __shfl_xor_sync(FULL, rho, o);
      jx += __shfl_xor_sync(FULL, jx, o);
      jy += __shfl_xor_sync(FULL, jy, o);
      jz += __shfl_xor_sync(FULL, jz, o);
    }
    const R rc = p.compressible ? rho_full_r<Form<P>::SH>(rho) : R(1);
    R Ux = jx, Uy = jy, Uz = jz;
    if (p.compressible) {
      Ux = jx / rc;
      Uy = jy / rc;
      Uz = jz / rc;
    }
    const R gx = R(p.g[0]), gy = R(p.g[1]), gz = R(p.g[2]);
    const R vx_ = Ux + R(0.5) * gx, vy_ = Uy + R(0.5) * gy, vz_ = Uz + R(0.5) * gz;
    const R ilm = P == P64 ? R(p.inv_lam_m) : R(1) / R(p.lam_m);
    const R ex = Ux - gx * ilm, ey = Uy - gy * ilm, ez = Uz - gz * ilm;
    const R usq2 = vx_ * vx_ + vy_ * vy_ + vz_ * vz_;
    const R fb = __shfl_sync(FULL, f, inv(q));
    const R ep = eplus_q<R>(p, q, rho, rc, vx_, vy_, vz_, usq2);
    const R em = R(3) * wq_ * rc * (R(cx(q)) * ex + R(cy(q)) * ey + R(cz(q)) * ez);
    const R out = f + R(p.lam_p) * (R(0.5) * (f + fb) - ep) + R(p.lam_m) * (R(0.5) * (f - fb) - em);
    if (lane < 19) stq<P>(v.fout, (size_t)q * N + (size_t)j, q, out);
    if (lane == 0) {
      v.m[j] = 0.0;
      v.phout[j] = R(0);
    }
  }
}

// empty cell k (still marked: only its own warp clears that) by a warp, lane q
// (1..18) takes link q
template <int P>
__device__ __forceinline__ void empty_cell(const Par& p, const View<P>& v, int k) {
  const int lane = threadIdx.x & 31;
  const int q = (lane >= 1 && lane < 19) ? lane : 0;
  {
    const long long i = FSL_CK(p, v.elist[k], p.N);
    int x, y, z;
    coords(p, i, x, y, z);
    long long j = -1;
    uint8_t kj = WALL, mj = 0;
    if (q) {
      j = nbr(p, x, y, z, cx(q), cy(q), cz(q));
      if (j >= 0) {
        kj = v.flags[j] & KIND;
        mj = v.mark[j];
      }
    }
    // an emptied cell next to a filled one stays interface
    if (__any_sync(0xffffffffu, (mj & MK_FILL) != 0)) {
      if (lane == 0) clear_u8(v.mark, i, MK_EMPTY);
      return;  // (warp-uniform)
    }
    bool won = false;
    if (kj == LIQ) {
      const uint8_t old = or_u8(v.mark, j, MK_NEWL);
      won = !(old & MK_NEWL);  // the first claimant lists it; newl sets m = rho
    }
    push(won, v.nllist, &v.cnt[4], v.cap, (int)j, v.err);
  }
}

// The calling warp's place among the grid's: the blocks' first warps, then their
// second ones, ..., so that a list shorter than the grid spreads over every SM
// (by blocks, 900 items of a 128x64x64 splash sat on a third of the SMs and
// its 5 k receivers, a thread each, on ten).
__device__ __forceinline__ int grid_warp() { return (int)((threadIdx.x >> 5) * gridDim.x + blockIdx.x); }
__device__ __forceinline__ int grid_warps() { return (int)((blockDim.x >> 5) * gridDim.x); }
// items of a thread each: few lanes of every warp where the list is short
struct LaneItems {
  int k, step, end;
  __device__ __forceinline__ explicit LaneItems(int n, int first_warp) {
    const int nw = grid_warps(), lane = threadIdx.x & 31;
    const int per = min(max((n + nw - 1) / nw, 1), 32);  // items per warp and round
    k = lane < per ? first_warp * per + lane : n;
    step = nw * per;
    end = n;
  }
};

// the first stage: a warp per fill or empty cell
template <int P>
__device__ __forceinline__ void do_fill_empty(const Par& p, const View<P>& v) {
  const int nf = min(load_count(&v.cnt[1]), v.cap), ne = min(load_count(&v.cnt[2]), v.cap);
  for (int k = grid_warp(); k < nf + ne; k += grid_warps()) {
    if (k < nf) fill_cell<P>(p, v, k);
    else empty_cell<P>(p, v, k - nf);
  }
}
// liquid cells turned interface next to an emptied cell: m = rho, phi = m/rho
// (by the grid's last warps first: its first ones take the other items of the
// stage)
template <int P>
__device__ __forceinline__ void do_newl(const Par& p, const View<P>& v) {
  using R = typename Form<P>::R;
  const LaneItems it(min(load_count(&v.cnt[4]), v.cap), grid_warps() - 1 - grid_warp());
  for (int k = it.k; k < it.end; k += it.step) {
    long long j = FSL_CK(p, v.nllist[k], p.N);
    const double r = rho_out<P>(p, v, j);
    v.m[j] = r;
    v.phout[j] = (R)(r / r);
  }
}

// Fill-level normal of a converting cell for the weighted excess split
// (Thuerey's distribution along the interface normal): n = -grad phi by
// central differences, n_a = (phi(x - e_a) - phi(x + e_a)) / 2, pointing into
// the gas, from the fill levels after the mass exchange (liquid 1, gas 0,
// interface m/rho as k_iface stored it, the cell's own value across a wall or
// a face).  The flags are those of time t until k_final.
template <int P>
__device__ __forceinline__ double phi_star(const Par& p, const View<P>& v, long long j, double own) {
  if (j < 0) return own;
  const uint8_t k = v.flags[j] & KIND;
  return k == LIQ ? 1.0 : (k == GAS ? 0.0 : (k == IFC ? (double)v.phout[j] : own));
}
template <int P>
__device__ __forceinline__ void fill_normal(const Par& p, const View<P>& v, long long i, double (&n)[3]) {
  int x, y, z;
  coords(p, i, x, y, z);
  const double own = (double)v.phout[i];
  n[0] = 0.5 * (phi_star<P>(p, v, nbr(p, x, y, z, -1, 0, 0), own) - phi_star<P>(p, v, nbr(p, x, y, z, 1, 0, 0), own));
  n[1] = 0.5 * (phi_star<P>(p, v, nbr(p, x, y, z, 0, -1, 0), own) - phi_star<P>(p, v, nbr(p, x, y, z, 0, 1, 0), own));
  n[2] = 0.5 * (phi_star<P>(p, v, nbr(p, x, y, z, 0, 0, -1), own) - phi_star<P>(p, v, nbr(p, x, y, z, 0, 0, 1), own));
}
// weight of the neighbour along c (components -1, 0, 1, so the products are
// exact and the sum is the same in any contraction): a filled cell pushes its
// excess toward the gas (n.c > 0), an emptied cell draws its deficit from the
// liquid side (n.c < 0)
__device__ __forceinline__ double split_weight(const double (&n)[3], int ax, int ay, int az, bool filled) {
  const double d = (double)ax * n[0] + (double)ay * n[1] + (double)az * n[2];
  return filled ? (d > 0.0 ? d : 0.0) : (d < 0.0 ? -d : 0.0);
}

template <int P>
__device__ __noinline__ double sender_weight(const Par& p, const View<P>& v, long long i, int ax, int ay, int az,
                                             bool filled) {
  double n[3];
  fill_normal<P>(p, v, i, n);
  return split_weight(n, ax, ay, az, filled);
}

// fill or empty cell k (of nf fills, then the empties) by a warp: lane q (1..18)
// tests neighbour q as a receiver; lane 0 computes the share (rho summed in q
// order, as a thread would)
template <int P>
__device__ __forceinline__ void share_cell(const Par& p, const View<P>& v, int k, int nf) {
  const unsigned FULL = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  const int q = (lane >= 1 && lane < 19) ? lane : 0;
  {
    const bool isF = k < nf;
    const long long i = FSL_CK(p, isF ? v.flist[k] : v.elist[k - nf], p.N);
    if (!isF && !(v.mark[i] & MK_EMPTY)) return;  // warp-uniform
    int x, y, z;
    coords(p, i, x, y, z);
    // lane 0: the cell's density and mass, loaded beside the neighbour tests
    double rho = 0.0, mi = 0.0;
    if (lane == 0) {
      rho = rho_out<P>(p, v, i);
      mi = v.m[i];
    }
    bool recv = false;
    long long j = -1;
    if (q) {
      j = nbr(p, x, y, z, cx(q), cy(q), cz(q));
      if (j >= 0) {
        const uint8_t mk = ((volatile uint8_t*)v.mark)[j];
        const uint8_t kj = v.flags[j] & KIND;
        recv = (mk & (MK_NEWG | MK_NEWL)) || (kj == IFC && !(mk & (MK_FILL | MK_EMPTY)));
      }
    }
    const unsigned rm = __ballot_sync(FULL, recv);
    // weighted split: the receivers' weights summed in q order on lane 0
    double V = 0.0;
    if (p.excess_split && rm) {
      const double w = recv ? sender_weight<P>(p, v, i, cx(q), cy(q), cz(q), isF) : 0.0;
      for (int s = 1; s < 19; ++s) V += __shfl_sync(FULL, w, s);
    }
    if (lane == 0) {
      const double ex = isF ? mi - rho : mi;
      const int nr = __popc(rm);
      if (nr == 0) {
        if (owned(p, x, y, z)) atomicAdd(v.lost, ex);  // (a ghost cell's owner books it)
        v.share[i] = 0.0;
      } else if (V > 1e-12) {
        v.share[i] = ex / V;
        v.mark[i] = (uint8_t)(v.mark[i] | MK_WSPLIT);
      } else {
        v.share[i] = ex / (double)nr;  // equal split (also where no receiver lies along the normal)
      }
      v.m[i] = isF ? rho : 0.0;
    }
    bool first = false;
    if (recv) {
      const uint8_t old = or_u8(v.mark, j, MK_RECV);
      first = !(old & MK_RECV);
    }
    push(first, v.rlist, &v.cnt[5], v.cap, (int)j, v.err);
  }
}

// new cells from gas, new cells from liquid and the excess shares are
// independent once the first stage has claimed the new cells and settled the
// empty list: their items follow one another over the grid's warps, so that a
// warp has one of them (not one of each) until every warp has one
template <int P>
__device__ __forceinline__ void do_new_share(const Par& p, const View<P>& v) {
  const int nf = min(load_count(&v.cnt[1]), v.cap), ne = min(load_count(&v.cnt[2]), v.cap);
  const int nn = min(load_count(&v.cnt[3]), v.cap);
  for (int k = grid_warp(); k < nn + nf + ne; k += grid_warps()) {
    if (k < nn) newg_cell<P>(p, v, k);
    else share_cell<P>(p, v, k - nn, nf);
  }
  do_newl<P>(p, v);
}
// a receiver's shares where some of them are split along the normal (out of
// line: an option, and with its normals inlined for every link it was most of
// the kernel's code)
template <int P>
__device__ __noinline__ double weighted_shares(const Par& p, const View<P>& v, int x, int y, int z) {
  double acc = 0.0;
#pragma unroll 1
  for (int q = 1; q < 19; ++q) {
    const long long j = nbr(p, x, y, z, cx(q), cy(q), cz(q));
    const uint8_t mk = j < 0 ? (uint8_t)0 : v.mark[j];
    if (!(mk & (MK_FILL | MK_EMPTY))) continue;
    if (mk & MK_WSPLIT) {  // the link from j to this receiver is -c_q
      double n[3];
      fill_normal<P>(p, v, j, n);
      acc += v.share[j] * split_weight(n, -cx(q), -cy(q), -cz(q), (mk & MK_FILL) != 0);
    } else {
      acc += v.share[j];
    }
  }
  return acc;
}

// one thread per receiver (the lists are long late in a run): gathers the
// shares of its converting neighbours in q order (deterministic)
template <int P>
__device__ __forceinline__ void do_recv(const Par& p, const View<P>& v) {
  using R = typename Form<P>::R;
  const LaneItems it(min(load_count(&v.cnt[5]), v.cap), grid_warp());
  for (int k = it.k; k < it.end; k += it.step) {
    const long long yj = FSL_CK(p, v.rlist[k], p.N);
    int x, y, z;
    coords(p, yj, x, y, z);
    int src[19];
    pull_sources(p, x, y, z, src);
    // the receiver's own mass and density first: their loads overlap the
    // neighbours' marks and shares
    const double m0 = v.m[yj];
    const double rho = p.excess_split ? 1.0 : rho_out<P>(p, v, yj);
    // the neighbours' marks, then the converting ones' shares, each as loads
    // in flight together (a load, a test and a dependent load per neighbour in
    // turn took 13 us of a 128x64x64 splash's 41 us conversions)
    unsigned conv = 0u, wsp = 0u;
#pragma unroll
    for (int q = 1; q < 19; ++q) {
      const int j = src[inv(q)];  // x + c_q
      const uint8_t mk = j < 0 ? (uint8_t)0 : v.mark[j];
      if (mk & (MK_FILL | MK_EMPTY)) conv |= 1u << q;
      if (mk & MK_WSPLIT) wsp |= 1u << q;
    }
    double acc = 0.0, sh[19];
#pragma unroll
    for (int q = 1; q < 19; ++q) sh[q] = (conv & (1u << q)) ? v.share[src[inv(q)]] : 0.0;
    if (!(conv & wsp)) {
#pragma unroll
      for (int q = 1; q < 19; ++q)
        if (conv & (1u << q)) acc += sh[q];
    } else {
      acc = weighted_shares<P>(p, v, x, y, z);
    }
    const double mm = m0 + acc;
    v.m[yj] = mm;
    // (the weighted split reads the fill levels of interface cells here, so
    // its receivers take their new fill level in k_final)
    if (!p.excess_split) {
      v.phout[yj] = (R)(mm / rho);
    }
  }
}

template <int P>
__device__ __forceinline__ void do_final(const Par& p, const View<P>& v) {
  using R = typename Form<P>::R;
  int nf = min(load_count(&v.cnt[1]), v.cap), ne = min(load_count(&v.cnt[2]), v.cap);
  int ng = min(load_count(&v.cnt[3]), v.cap), nl = min(load_count(&v.cnt[4]), v.cap);
  int nr = min(load_count(&v.cnt[5]), v.cap);
  int total = nf + ne + ng + nl + nr;
  // running total of conversions since the state was set (never reset per step)
  if (blockIdx.x == 0 && threadIdx.x == 0 && nf + ng + nl) atomicAdd(&v.cnt[8], nf + ng + nl);
  int emptied = 0;  // cells this thread turned to gas (counted once per warp below)
  const LaneItems it(total, grid_warp());
  for (int k = it.k; k < it.end; k += it.step) {
    int kk = k;
    if (kk < nf) {
      long long i = FSL_CK(p, v.flist[kk], p.N);
      v.flags[i] = (uint8_t)((v.flags[i] & STATIC_BITS) | LIQ);
      v.mark[i] = 0;
      continue;
    }
    kk -= nf;
    if (kk < ne) {
      long long i = FSL_CK(p, v.elist[kk], p.N);
      if (v.mark[i] & MK_EMPTY) {
        v.flags[i] = (uint8_t)((v.flags[i] & STATIC_BITS) | GAS);
        v.phout[i] = R(0);
        v.mark[i] = 0;
        ++emptied;
      }
      continue;
    }
    kk -= ne;
    if (kk < ng) {
      long long i = FSL_CK(p, v.nglist[kk], p.N);
      v.flags[i] = (uint8_t)((v.flags[i] & STATIC_BITS) | IFC);
      v.mark[i] = 0;
      continue;
    }
    kk -= ng;
    if (kk < nl) {
      long long i = FSL_CK(p, v.nllist[kk], p.N);
      v.flags[i] = (uint8_t)((v.flags[i] & STATIC_BITS) | IFC);
      v.mark[i] = 0;
      continue;
    }
    kk -= nl;
    const long long r = FSL_CK(p, v.rlist[kk], p.N);
    v.mark[r] = 0;
    if (p.excess_split) v.phout[r] = (R)(v.m[r] / rho_out<P>(p, v, r));
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) emptied += __shfl_down_sync(0xffffffffu, emptied, o);
  if ((threadIdx.x & 31) == 0 && emptied) {
    atomicAdd(&v.cnt[7], emptied);
    atomicAdd(&v.cnt[8], emptied);
  }
}

// removed E cells keep a zero mark; receivers, new cells and F/E cells are
// cleared above.  E cells that left E in k_fill carry no mark bits besides a
// possible RECV (cleared through the receiver list).

// Grid-wide barrier of the fused conversion kernel (a cooperative launch, so
// every block is resident): thread 0 of each block arrives on the per-step
// counter cnt[10] and waits until the blocks of this phase have arrived.  The
// wait is bounded (about a second); on expiry it records ERRB_SYNC and goes
// on, the step's result is then invalid and the host reports the error.
__device__ __forceinline__ void grid_arrive(unsigned* ctr) {
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    atomicAdd(ctr, 1u);
  }
}
// false (on every thread of the block) where the wait expired
__device__ __forceinline__ bool grid_wait(unsigned* ctr, unsigned target, int* err) {
  bool expired = false;
  if (threadIdx.x == 0) {
    unsigned spins = 0;
    while (*((volatile unsigned*)ctr) < target) {
      if (++spins > (1u << 20)) {
        atomicOr(err, ERRB_SYNC);
        expired = true;
        break;
      }
      __nanosleep(100);
    }
    __threadfence();
  }
  return __syncthreads_or(expired) == 0;
}

__device__ __forceinline__ void grid_sync(unsigned* ctr, unsigned target, int* err) {
  grid_arrive(ctr);
  grid_wait(ctr, target, err);
}

// The step's two-level mass reduction (the same chunks and order as the
// stand-alone pair of launches) on the grid's last blocks: a chunk each, and
// the last of them to finish adds up the chunks.  lost0: the lost ledger before
// any excess of this step (thread 0).
__device__ __forceinline__ void reduce_mass(const MassReduce& mr, int chunk, int* done, double lost0) {
  if (chunk < 0) return;  // (block-uniform)
  __shared__ bool last;
  const double t = block_chunk_sum(mr.in, mr.n, mr.chunk, chunk);
  if (threadIdx.x == 0) {
    mr.tmp[chunk] = t;
    __threadfence();
    last = atomicAdd(done, 1) == mr.nb - 1;
    __threadfence();
  }
  __syncthreads();
  if (last) {
    const double m = block_chunk_sum<true>(mr.tmp, mr.nb, mr.nb, 0);
    if (threadIdx.x == 0) *mr.out = m + lost0;
  }
}

}  // namespace fsl
