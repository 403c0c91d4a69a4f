// fslbm_bulk64.cu -- bulk stream-collide of the FP64 form.
//
// One lane per cell of a 32-cell segment, one warp per segment (as k_bulk),
// the kinds taken from the segment's masks and the next segment's record and
// masks loaded one round ahead (as k_bulk_pairs), the collision in fixed point
// (fslbm_fixed.cuh).  Algorithmic bytes 304 per liquid cell.
#include <cuda_runtime.h>

#include "fslbm_dev.cuh"
#include "fslbm_fixed.cuh"
#include "fslbm_kernels.h"
#include "fslbm_pull.cuh"
#include "fslbm_slow.cuh"

namespace fsl {

constexpr int BULK64_BLOCKS = 4;  // resident blocks of 128 threads per SM

__global__ void __launch_bounds__(128, BULK64_BLOCKS) k_bulk_fixed(Par p, View<P64> v,
                                                                   const int* __restrict__ seglist,
                                                                   const int* __restrict__ segcount) {
  pdl_begin();
  const int nseg = *((volatile const int*)segcount);
  const int lane = threadIdx.x & 31;
  const int gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int nw = (gridDim.x * blockDim.x) >> 5;
  const size_t N = (size_t)p.N;
  const long long sy = p.nx, sz = (long long)p.nx * p.ny;
  const int nsx = (p.nx + 31) >> 5;
  const uint4* masks = reinterpret_cast<const uint4*>(seglist) + (long long)nsx * p.ny * p.nz;
  double msum = 0.0;
  // the densities of the fast cells, summed exactly: low and high words of their fixed-point values
  long long slo = 0, shi = 0;
  int4 sd_n = make_int4(0, 0, 0, 0);
  uint4 sm_n = make_uint4(0u, 0u, 0u, 0u);
  if (gw < nseg) {
    sd_n = reinterpret_cast<const int4*>(seglist)[gw];
    sm_n = masks[gw];
  }
  for (int si = gw; si < nseg; si += nw) {
    const int4 sd = sd_n;  // x0, y, z, first cell
    const uint4 sm = sm_n;  // liquid, interface, liquid needing the general pull
    if (si + nw < nseg) {
      sd_n = reinterpret_cast<const int4*>(seglist)[si + nw];
      sm_n = masks[si + nw];
    }
    const bool on = (sm.x >> lane) & 1u;
    if (!on) continue;
    const int x = sd.x + lane, y = sd.y, z = sd.z;
    const unsigned i = (unsigned)FSL_CK_IF(p, on, (long long)sd.w + lane, p.N);
    if ((sm.z >> lane) & 1u) {
      msum += slow_cell<P64>(p, v, (long long)i, x, y, z, v.flags[i]);
      continue;
    }
    double f[19];
    const bool ax0 = x == 0, ax1 = x == p.nx - 1, ay0 = y == 0, ay1 = y == p.ny - 1, az0 = z == 0,
               az1 = z == p.nz - 1;
    // (each population's base pointer, shifted by its link, is the same for the whole grid)
    if (!(ax0 || ax1 || ay0 || ay1 || az0 || az1)) {
#pragma unroll
      for (int q = 0; q < 19; ++q) {
        const long long off = cx(q) + sy * cy(q) + sz * cz(q);
        const double* base = v.fin + ((long long)(q * N) - off);
        f[q] = __ldg(base + (size_t)(FSL_CK(p, (long long)i - off, p.N) + off));
      }
    } else {  // a source beyond a non-periodic face: half-way bounce-back from the cell's own slot
      f[0] = __ldg(v.fin + i);
#pragma unroll
      for (int q = 1; q < 19; ++q) {
        const bool bb = (cx(q) == 1 && ax0) || (cx(q) == -1 && ax1) || (cy(q) == 1 && ay0) || (cy(q) == -1 && ay1) ||
                        (cz(q) == 1 && az0) || (cz(q) == -1 && az1);
        const long long off = bb ? 0 : cx(q) + sy * cy(q) + sz * cz(q);
        f[q] = __ldg(v.fin + (bb ? inv(q) : q) * N + (size_t)FSL_CK(p, (long long)i - off, p.N));
      }
    }
    long long rf;
    bool over;
    if (collide_fixed(p, f, rf, over)) {
      if (over) atomicOr(v.err, ERRB_SPEED);
      if (owned(p, x, y, z)) {
        slo += (long long)(unsigned)rf;
        shi += rf >> 32;
      }
    } else {
      double rho, ux, uy, uz;
      collide<double>(p, f, rho, ux, uy, uz);
      if (rho_bad<false>(rho)) atomicOr(v.err, ERRB_UNSTABLE);
      if (speed_bad(p, ux, uy, uz)) atomicOr(v.err, ERRB_SPEED);
      if (owned(p, x, y, z)) msum += rho;
    }
#pragma unroll
    for (int q = 0; q < 19; ++q) (v.fout + q * N)[i] = f[q];
  }
  msum += (double)shi * 0x1p-28 + (double)slo * 0x1p-60;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) msum += __shfl_down_sync(0xffffffffu, msum, o);
  if (lane == 0) v.partials[gw] = msum;
}

int launch_bulk_fixed(const Par& p, const View<P64>& v, cudaStream_t st, int bulk_blocks, const int* seglist,
                      const int* segcount) {
  return launch_k(k_bulk_fixed, bulk_blocks, 128, 0, st, p, v, seglist, segcount);
}

}  // namespace fsl
