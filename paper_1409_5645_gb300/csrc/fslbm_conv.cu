// fslbm_conv.cu -- cell conversions after the mass update (Sec. 2.3 / 4.4; the
// paper takes interface tracking from Koerner et al. and Thuerey).
//
// The step kernel appended interface cells with m > (1+eps) rho to the fill
// list F and those with m < -eps rho to the empty list E, and marked them.
// Then, all as list kernels (grid-stride; counts read on the device, no host
// synchronisation):
//   fill     gas neighbours of F become new interface (NEWG, listed once by an
//            atomic byte-OR)
//   empty    an E cell with an F neighbour leaves E (it stays interface);
//            liquid neighbours of the remaining E become interface (NEWL)
//   newg     NEWG cells get f = f^eq(mean rho, mean u) over their liquid /
//            interface neighbours (q order), collided, m = 0
//   newl     NEWL cells get m = rho
//   share    excess (F: m - rho, E: m) / number of receivers (interface after
//            the steps above, not converting); no receiver -> lost ledger
//   recv     each receiver gathers the shares of its converting neighbours in q
//            order (deterministic, no floating-point atomics)
//   final    F -> liquid, E -> gas, new cells -> interface, marks cleared
// fill and empty run together (each E cell tests its own neighbours for F
// marks, which the step kernel set), and so do newg, newl and share (share
// reads only the marks and claims of the first stage and the converting
// cells' own state).  The four stages run as one cooperative launch
// (k_convert, two resident blocks per SM, grid barriers between the stages)
// where the device allows it, else as four launches.  The result does not
// depend on list order.
#include "fslbm_conv.cuh"
#include "fslbm_dev.cuh"
#include "fslbm_kernels.h"

namespace fsl {

template <int P>
__global__ void __launch_bounds__(256) k_fill_empty(Par p, View<P> v) {
  pdl_begin();
  do_fill_empty<P>(p, v);
}

template <int P>
__global__ void __launch_bounds__(256) k_new_share(Par p, View<P> v) {
  pdl_begin();
  do_new_share<P>(p, v);
}

template <int P>
__global__ void __launch_bounds__(256) k_recv(Par p, View<P> v) {
  pdl_begin();
  do_recv<P>(p, v);
}

template <int P>
__global__ void __launch_bounds__(256) k_final(Par p, View<P> v) {
  pdl_begin();
  do_final<P>(p, v);
}

// the four conversion stages in one launch, separated by grid barriers, with
// the mass reduction between a block's arrival at the first barrier and its
// wait there.  A step without a fill or an empty cell has the mass only.
// Alone, with warm caches: a film's step 17.2 -> 6.8 us without the barriers;
// with conversions, a stage's items one to a warp over all SMs and a
// receiver's loads together, a 128x64x64 splash's 46.8 -> 35.9 us, a 256x128x128 FP64
// splash's 96 -> 60 us
template <int P>
__global__ void __launch_bounds__(256) k_convert(Par p, View<P> v, MassReduce mr) {
  pdl_begin();
  unsigned* ctr = (unsigned*)&v.cnt[10];
  const unsigned nb = gridDim.x;
  const int chunk = (int)blockIdx.x - ((int)gridDim.x - mr.nb);
  double lost0 = 0.0;
  if (chunk >= 0 && threadIdx.x == 0) lost0 = *((volatile const double*)mr.add);
  if (load_count(&v.cnt[1]) + load_count(&v.cnt[2]) == 0) {  // (settled before this kernel)
    reduce_mass(mr, chunk, &v.cnt[11], lost0);
    return;
  }
  do_fill_empty<P>(p, v);
  grid_arrive(ctr);
  reduce_mass(mr, chunk, &v.cnt[11], lost0);
  grid_wait(ctr, nb, v.err);
  do_new_share<P>(p, v);
  grid_sync(ctr, 2 * nb, v.err);
  do_recv<P>(p, v);
  grid_sync(ctr, 3 * nb, v.err);
  do_final<P>(p, v);
}

// self-check of the barrier: one grid_sync waiting for `extra` blocks more
// than the grid has (extra = 1: nothing completes it, the bounded wait runs out)
__global__ void __launch_bounds__(256) k_barrier_check(unsigned* ctr, unsigned extra, int* err) {
  grid_sync(ctr, gridDim.x + extra, err);
}

int launch_barrier_check(unsigned* ctr, int* err, int blocks, unsigned extra, cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(blocks);
  cfg.blockDim = dim3(256);
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeCooperative;
  at[0].val.cooperative = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return (int)cudaLaunchKernelEx(&cfg, k_barrier_check, ctr, extra, err);
}

// resident blocks of k_convert per SM (0: the fused kernel cannot be used)
template <int P>
int convert_blocks_per_sm() {
  int nb = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_convert<P>, 256, 0) != cudaSuccess) return 0;
  return nb;
}

// coop_blocks > 0: the fused cooperative kernel on that many blocks (all
// resident); else four launches of list_blocks
template <int P>
int launch_conversions(const Par& p, const View<P>& v, cudaStream_t st, int list_blocks, int coop_blocks,
                       const MassReduce& mr) {
  if (coop_blocks > 0) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(coop_blocks);
    cfg.blockDim = dim3(256);
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    if (mr.nb > coop_blocks) return (int)cudaErrorInvalidValue;
    return (int)cudaLaunchKernelEx(&cfg, k_convert<P>, p, v, mr);
  }
  void (*ks[4])(Par, View<P>) = {k_fill_empty<P>, k_new_share<P>, k_recv<P>, k_final<P>};
  for (auto k : ks)
    if (launch_k(k, list_blocks, 256, 0, st, p, v)) return 1;
  return 0;
}

template int launch_conversions<P64>(const Par&, const View<P64>&, cudaStream_t, int, int, const MassReduce&);
template int launch_conversions<P32>(const Par&, const View<P32>&, cudaStream_t, int, int, const MassReduce&);
template int launch_conversions<P16>(const Par&, const View<P16>&, cudaStream_t, int, int, const MassReduce&);
template int convert_blocks_per_sm<P64>();
template int convert_blocks_per_sm<P32>();
template int convert_blocks_per_sm<P16>();

}  // namespace fsl
