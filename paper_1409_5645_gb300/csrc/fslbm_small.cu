// fslbm_small.cu -- many time steps of a small lattice in one launch.
//
// A step of a lattice of a few thousand cells is a chain of six kernels whose
// work is a few us: most of its time goes to the launches' gaps and to
// fetching each kernel's code again (about 40 cycles an instruction that runs
// once).  k_steps stays on the chip for many steps, a block an SM, with one
// grid barrier a step while no cell converts and six more where one does:
//   interface cells   a warp each, geometry and interface cell in a row
//                     (coop_stencil, iface_warp64 / iface_warp32), from the
//                     grid's last warps on
//   liquid cells      a thread each, from the first warps on
//   barrier           then the conversion stages, where there are any, and a
//                     new list of the interface cells
// Every result of a step is the ordinary kernels' bit for bit; the last step of
// a call always runs through those, which leave the counters and the mass
// balance that a caller reads.  Loads of what the kernel itself has written
// are plain loads (no read-only path).
#include <cuda_runtime.h>

#include "fslbm_conv.cuh"
#include "fslbm_dev.cuh"
#include "fslbm_fixed.cuh"
#include "fslbm_kernels.h"
#include "fslbm_pull.cuh"
#include "fslbm_step.cuh"

namespace fsl {

// a liquid cell wherever it lies (out of line: apart from the interface cells'
// registers)
template <int P>
__device__ __noinline__ void liquid_cell(const Par& p, const View<P>& v, long long i) {
  using R = typename Form<P>::R;
  constexpr bool SH = Form<P>::SH;
  const size_t N = (size_t)p.N;
  int x, y, z;
  coords(p, i, x, y, z);
  R f[19];
  unsigned wallm, gasm, liqm;
  int srcs[19];
  f[0] = ldq<P>(v.fin, (size_t)i, 0);
  pull_table<P>(p, v, x, y, z, f, wallm, gasm, liqm, srcs);
  if (gasm) atomicOr(v.err, ERRB_STATE);  // liquid must not touch gas
  wallm |= gasm;
  if (wallm) {
    R own[19];
#pragma unroll
    for (int q = 0; q < 19; ++q) own[q] = ldq<P>(v.fin, (size_t)q * N + (size_t)i, q);
    wall_links<P>(p, v, i, wallm, 0u, own, f);
  }
  bool done = false;
  if constexpr (P == P64) {
    long long rf;
    bool over = false;
    done = collide_fixed(p, f, rf, over);
    if (done && over) atomicOr(v.err, ERRB_SPEED);
  }
  if (!done) {
    R rho, ux, uy, uz;
    collide<R, SH>(p, f, rho, ux, uy, uz);
    if (rho_bad<SH>(rho)) atomicOr(v.err, ERRB_UNSTABLE);
    if (speed_bad(p, ux, uy, uz)) atomicOr(v.err, ERRB_SPEED);
  }
#pragma unroll
  for (int q = 0; q < 19; ++q) stq<P>(v.fout, (size_t)q * N + (size_t)i, q, f[q]);
}

// CHAIN: the FP64 form without the fixed-point collision (the steps of a
// differentiation, whose operations stay those they have always been): the
// interface cell is the thread's general one.
// log: the state after every step is also copied there.
template <int P, bool SIG, bool CHAIN>
__global__ void __launch_bounds__(256, 1) k_steps(Par p, View<P> v, int steps, unsigned* ctr, StateLog log) {
  using R = typename Form<P>::R;
  using S = typename Form<P>::S;
  const int lane = threadIdx.x & 31, nw = grid_warps(), wid = grid_warp();
  const size_t cap = (size_t)v.cap;
  const bool geo = p.rule != 0 || p.sigma != 0.0;
  unsigned target = 0;
  auto barrier = [&]() {  // every block of the cooperative grid; false: the bounded wait expired
    target += gridDim.x;
    grid_arrive(ctr);
    return grid_wait(ctr, target, v.err);
  };
  // Two sets of the step counters in turn: a block that is already in the next
  // step appends to the other set while a slower one still reads this step's.
  // The count of the interface list and the running total stay in the first
  // counters (base).
  int* const base = v.cnt;
  if (blockIdx.x == 0 && threadIdx.x < 32) base[16 + threadIdx.x] = 0;
  bool relist = true;
  for (int s = 0; s < steps; ++s) {
    v.cnt = base + 16 * (1 + (s & 1));
    if (relist) {
      if (blockIdx.x == 0 && threadIdx.x == 0) base[0] = 0;
      if (!barrier()) return;
      for (long long b = 32LL * wid; b < p.N; b += 32LL * nw) {
        const long long i = b + lane;
        const bool on = i < p.N && (v.flags[i] & KIND) == IFC;
        warp_append(on, (int)i, v.ilist, &base[0], v.cap, v.err);
      }
      if (!barrier()) return;
      relist = false;
    }
    const int n = min(load_count(&base[0]), v.cap);
    for (int e = nw - 1 - wid; e < n; e += nw) {
      const long long i = FSL_CK(p, v.ilist[e], p.N);
      int x, y, z;
      coords(p, i, x, y, z);
      if (geo) {
        const bool in3 = x >= 3 && x < p.nx - 3 && y >= 3 && y < p.ny - 3 && z >= 3 && z < p.nz - 3;
        const R phic = v.phin[i];
        Geo<R> G;
        R nn, kopen;
        const bool ok = coop_stencil<R, SIG>(p, v.flags, v.phin, x, y, z, in3, (int)i, phic, nn, kopen, G);
        if (ok) coop_finish<R, SIG, false>(p, v.flags, v.phin, x, y, z, phic, nn, kopen, G);
        if (lane == 0) {
          v.geo[e] = ok ? G.n[0] : R(0);
          v.geo[cap + e] = ok ? G.n[1] : R(0);
          v.geo[2 * cap + e] = ok ? G.n[2] : R(0);
          v.geo[3 * cap + e] = G.d;
          v.geo[4 * cap + e] = G.kap;
        }
        __syncwarp();
      }
      bool fill = false, empty = false;
      if constexpr (CHAIN) {
        if (lane == 0) {
          if (x >= 3 && x < p.nx - 3 && y >= 3 && y < p.ny - 3 && z >= 3 && z < p.nz - 3)
            iface_cell<P, true, false>(p, v, e, i, x, y, z, fill, empty);
          else
            iface_cell<P, false, false>(p, v, e, i, x, y, z, fill, empty);
        }
        __syncwarp();
      } else if constexpr (P == P64) {
        iface_warp64(p, v, e, i, x, y, z, fill, empty);
      } else {
        iface_warp32<P>(p, v, e, i, x, y, z, fill, empty);
      }
      warp_append(lane == 0 && fill, (int)i, v.flist, &v.cnt[1], v.cap, v.err);
      warp_append(lane == 0 && empty, (int)i, v.elist, &v.cnt[2], v.cap, v.err);
    }
    for (long long i = 32LL * wid + lane; i < p.N; i += 32LL * nw)
      if ((v.flags[i] & KIND) == LIQ) liquid_cell<P>(p, v, i);
    if (!barrier()) return;
    if (!p.freeze) {
      if (load_count(&v.cnt[1]) + load_count(&v.cnt[2]) != 0) {
        do_fill_empty<P>(p, v);
        if (!barrier()) return;
        do_new_share<P>(p, v);
        if (!barrier()) return;
        do_recv<P>(p, v);
        if (!barrier()) return;
        do_final<P>(p, v);
        if (!barrier()) return;
        if (blockIdx.x == 0 && threadIdx.x == 0) {  // (the set is used again after two more barriers)
          base[8] += v.cnt[8];
          for (int k = 1; k < 9; ++k) v.cnt[k] = 0;
        }
        relist = true;
      }
      R* in = const_cast<R*>(v.phin);
      v.phin = v.phout;
      v.phout = in;
    }
    S* in = const_cast<S*>(v.fin);
    v.fin = v.fout;
    v.fout = in;
    if (log.f) {
      const long long n19 = 19 * p.N, at = (long long)(s + 1) * p.N;
      const int t = wid * 32 + lane, nt = nw * 32;
      S* lf = (S*)log.f + 19 * at;
      R* lp = (R*)log.phi + at;
      for (long long k = t; k < n19; k += nt) lf[k] = v.fin[k];
      for (long long k = t; k < p.N; k += nt) {
        log.m[at + k] = v.m[k];
        lp[k] = v.phin[k];
        log.flags[at + k] = v.flags[k];
      }
      if (!barrier()) return;  // the next step writes masses and kinds in place
    }
  }
}

// Lattices that k_steps takes: the default closures, and few enough cells for
// the chain of a step to outweigh its work: measured (us a step, kernels by
// graph -> k_steps) 4x4x32 FP64 film 33.9 -> 14.8, 64x1x68 FP64 inclined film
// 33.9 -> 16.2, 5x6x40 FP32 film 29.2 -> 9.4, 48x1x52 FP32 inclined film 30 ->
// 10.9; against the first version's kernels, a 57x20x25 FP32 splash 101 -> 45,
// a 70x28x31 FP64 one (60 760 cells, near the limit) 314 -> 87, a 240x1x244
// FP64 inclined film 89 -> 30.  Above, the interface cells by warps (see
// IFACE_WARP_MAX) would set the step.
bool small_ok(const Par& p, int prec) {
  if (p.stress || p.ub_extrap || p.recon_nc || p.elvira) return false;
  // (an FP64 lattice whose equilibria or forces rule the fixed point out takes the kernels)
  if (prec == P64 && !p.fix_ok) return false;
  return p.N <= SMALL_CELLS;
}

template <int P>
int small_blocks(const Par& p, int sms) {
  int nb = 0;
  auto fits = [&](auto k) {
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k, 256, 0) == cudaSuccess && nb >= 1;
  };
  if (!fits(k_steps<P, false, false>) || !fits(k_steps<P, true, false>)) return 0;
  if constexpr (P == P64) {
    if (!fits(k_steps<P, false, true>)) return 0;
  }
  const long long want = (p.N + 127) / 128;
  return (int)(want < 8 ? (sms < 8 ? sms : 8) : (want < sms ? want : sms));
}

template <int P>
int launch_small(const Par& p, const View<P>& v, cudaStream_t st, int blocks, int steps, unsigned* ctr,
                 const StateLog& log) {
  if (cudaMemsetAsync(ctr, 0, sizeof *ctr, st) != cudaSuccess) return 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(blocks);
  cfg.blockDim = dim3(256);
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeCooperative;
  at[0].val.cooperative = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  auto k = p.sigma != 0.0 ? k_steps<P, true, false> : k_steps<P, false, false>;
  if constexpr (P == P64) {
    if (!p.fix_ok) {
      if (p.sigma != 0.0) return 1;
      k = k_steps<P, false, true>;
    }
  }
  return (int)cudaLaunchKernelEx(&cfg, k, p, v, steps, ctr, log);
}

#define FSL_INST(P)                                                                                       \
  template int small_blocks<P>(const Par&, int);                                                         \
  template int launch_small<P>(const Par&, const View<P>&, cudaStream_t, int, int, unsigned*, const StateLog&);
FSL_INST(P64)
FSL_INST(P32)
FSL_INST(P16)
#undef FSL_INST

}  // namespace fsl
