// fslbm_state.cu -- state set-up, field read-back and the full mass balance.
#include "fslbm_dev.cuh"
#include "fslbm_fixed.cuh"
#include "fslbm_kernels.h"

namespace fsl {

// Populations from the caller (pre-collision f, or f^eq(rho,u) + noise) ->
// collide -> stored f~(t); m = phi rho, phi = m/rho on interface cells.
template <int P>
__global__ void __launch_bounds__(128, P == P64 ? 4 : 6)
    k_init_pre(Par p, View<P> v, const double* __restrict__ fin, const double* __restrict__ phi,
               const double* __restrict__ rho_in, const double* __restrict__ u_in, const double* __restrict__ noise,
               double* __restrict__ keep_f0) {
  using R = typename Form<P>::R;
  const size_t N = (size_t)p.N;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < p.N;
       i += (long long)gridDim.x * blockDim.x) {
    uint8_t k = v.flags[i] & KIND;
    R* phA = const_cast<R*>(v.phin);
    if (!is_fluid(k)) {
      v.m[i] = 0.0;
      phA[i] = (k == GAS && p.freeze && phi) ? (R)phi[i] : R(0);
      continue;
    }
    double fd[19];
    if (fin) {
#pragma unroll
      for (int q = 0; q < 19; ++q) fd[q] = fin[(size_t)q * N + i];
    } else {
      // equilibrium at (rho, u), u^eq = u (Eq. eqEven / eqOdd): both
      // directions of a link share e^+ and take e^- with opposite signs (the
      // FP64 pipe bounds this kernel, so each is formed once; the roundings are
      // those of the expressions of eplus and eminus; 512x256x256, FP32 form:
      // 2.73 -> 1.67 ms, 1.45 with the conversions below in integers)
      const double r = rho_in[i];
      const double u[3] = {u_in[3 * i], u_in[3 * i + 1], u_in[3 * i + 2]};
      const double r0 = p.compressible ? r : 1.0, nl = p.linear_eq ? 0.0 : 1.0;
      const double usq = fma(u[2], u[2], fma(u[0], u[0], u[1] * u[1]));
      fd[0] = fma(wq<double>(0), r, -(((wq<double>(0) * 1.5) * r0 * nl) * usq));
      const double wr1 = wq<double>(1) * r, wr7 = wq<double>(7) * r;
      const double k1 = (wq<double>(1) * 1.5) * r0 * nl, k7 = (wq<double>(7) * 1.5) * r0 * nl;
      const double o1 = (3.0 * wq<double>(1)) * r0, o7 = (3.0 * wq<double>(7)) * r0;
#pragma unroll
      for (int q = 1; q < 19; q += 2) {
        double cu = 0.0;
        if (cx(q)) cu = cx(q) > 0 ? u[0] : -u[0];
        if (cy(q)) cu = cy(q) > 0 ? cu + u[1] : cu - u[1];
        if (cz(q)) cu = cz(q) > 0 ? cu + u[2] : cu - u[2];
        const double ep = fma(q <= 6 ? k1 : k7, fma(3.0 * cu, cu, -usq), q <= 6 ? wr1 : wr7);
        fd[q] = fma(q <= 6 ? o1 : o7, cu, ep);
        fd[q + 1] = fma(-(q <= 6 ? o1 : o7), cu, ep);
      }
      if (noise) {
#pragma unroll
        for (int q = 0; q < 19; ++q) fd[q] += noise[(size_t)q * N + i];
      }
    }
    double rs = 0.0;
    if (k == IFC || fin || noise) {
#pragma unroll
      for (int q = 0; q < 19; ++q) rs += fd[q];
    } else {
      rs = rho_in[i];  // (the equilibrium's sum; a liquid cell's m is read by nothing)
    }
    if (keep_f0) {
#pragma unroll
      for (int q = 0; q < 19; ++q) keep_f0[(size_t)q * N + i] = fd[q];
    }
    if (k == IFC) {
      double mm = (phi ? phi[i] : 1.0) * rs;
      v.m[i] = mm;
      phA[i] = (R)(mm / rs);
    } else {
      v.m[i] = rs;
      phA[i] = R(1);
    }
    R f[19];
    bool ints = false;
    if constexpr (Form<P>::SH) {
      // f - w_q exactly, then one rounding to float, in integers where the
      // populations are in the fixed-point range and above 2^-8 (no bit below
      // 2^-60): the subtractions and conversions were a third of the FP64
      // pipe's operations
      unsigned top = 0u, low = 0xffffffffu;
#pragma unroll
      for (int q = 0; q < 19; ++q) {
        const unsigned hi = (unsigned)(bits_of_double(fd[q]) >> 32);
        top = hi > top ? hi : top;
        low = hi < low ? hi : low;
      }
      ints = top < 0x3ff00000u && low >= 0x3f700000u;
      if (ints) {
#pragma unroll
        for (int q = 0; q < 19; ++q) {
          const long long w = q == 0 ? 0x0555555555555540LL : (q <= 6 ? 0x00e38e38e38e38e0LL : 0x0071c71c71c71c70LL);
          f[q] = (R)((float)(fix_of(bits_of_double(fd[q])) - w) * 0x1p-60f);
        }
      }
    }
    if (!ints) {
#pragma unroll
      for (int q = 0; q < 19; ++q) f[q] = to_arith<P>(fd[q], q);
    }
    R rho, ux, uy, uz;
    collide<R, Form<P>::SH>(p, f, rho, ux, uy, uz);
#pragma unroll
    for (int q = 0; q < 19; ++q) stq<P>(const_cast<typename Form<P>::S*>(v.fin), (size_t)q * N + i, q, f[q]);
  }
}

template <int P>
__global__ void k_init_post(Par p, View<P> v, const double* __restrict__ fpost, const double* __restrict__ m,
                            const double* __restrict__ phi) {
  using R = typename Form<P>::R;
  const size_t N = (size_t)p.N;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < p.N;
       i += (long long)gridDim.x * blockDim.x) {
    uint8_t k = v.flags[i] & KIND;
    R* phA = const_cast<R*>(v.phin);
    if (!is_fluid(k)) {
      v.m[i] = 0.0;
      phA[i] = (k == GAS && p.freeze && phi) ? (R)phi[i] : R(0);
      continue;
    }
#pragma unroll
    for (int q = 0; q < 19; ++q)
      stq<P>(const_cast<typename Form<P>::S*>(v.fin), (size_t)q * N + i, q, to_arith<P>(fpost[(size_t)q * N + i], q));
    v.m[i] = (k == IFC) ? m[i] : 0.0;
    phA[i] = (k == IFC) ? (R)phi[i] : R(1);
  }
}

// NEARB bit (a link ends in a wall or past a face) and invariant checks.
__device__ __forceinline__ void prepare_cell(const Par& p, uint8_t* flags, int* err, long long i, int x, int y, int z) {
  const uint8_t k = flags[i] & KIND;
  if (k != LIQ && k != IFC && k != GAS && k != WALL) {
    atomicOr(err, ERRB_STATE);
    return;
  }
  bool nearb = false, nearw = false, gas = false;
#pragma unroll
  for (int q = 1; q < 19; ++q) {
    long long j = nbr(p, x, y, z, cx(q), cy(q), cz(q));
    uint8_t kj = kind_at(flags, j);
    nearb |= (kj == WALL);
    nearw |= (j >= 0 && kj == WALL);
    gas |= (kj == GAS);
  }
  if (k == LIQ && gas) atomicOr(err, ERRB_STATE);
  flags[i] = (uint8_t)(k | (nearb ? NEARB : 0) | (nearw ? NEARW : 0));
}
__global__ void k_prepare_flags(Par p, uint8_t* flags, int* err) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < p.N;
       i += (long long)gridDim.x * blockDim.x) {
    int x, y, z;
    coords(p, i, x, y, z);
    prepare_cell(p, flags, err, i, x, y, z);
  }
}
// The same with 16 cells of a row per thread (nx a multiple of 16): the kinds
// are one-hot, so the OR of the neighbours' bytes holds their kinds; nine
// 16-byte loads and ten single bytes instead of 18 bytes a cell (512x256x256:
// 953 -> 90 us; its faces cell by cell took longer than the rest
// of a small lattice).  A row's first and last group on a periodic
// x axis take the cell path.  The bits written beside
// the kinds are masked from every load, so cells may be rewritten while their
// neighbours read them.
__global__ void __launch_bounds__(256) k_prepare_flags16(Par p, uint8_t* flags, int* err) {
  const long long total = p.N >> 4;
  const long long sy = p.nx, sz = (long long)p.nx * p.ny;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < total;
       t += (long long)gridDim.x * blockDim.x) {
    const long long i = t << 4;
    int x, y, z;
    coords(p, i, x, y, z);
    const bool xlo = x == 0, xhi = x + 16 == p.nx;
    if ((xlo || xhi) && p.px) {
      for (int k = 0; k < 16; ++k) prepare_cell(p, flags, err, i + k, x + k, y, z);
      continue;
    }
    unsigned near[4] = {0u, 0u, 0u, 0u}, own[4] = {0u, 0u, 0u, 0u};
    bool face = false;  // a row of neighbours lies past a non-periodic face
#pragma unroll
    for (int dz = -1; dz <= 1; ++dz)
#pragma unroll
      for (int dy = -1; dy <= 1; ++dy) {
        int Y = y + dy, Z = z + dz;
        if (p.py) Y += Y < 0 ? p.ny : (Y >= p.ny ? -p.ny : 0);
        if (p.pz) Z += Z < 0 ? p.nz : (Z >= p.nz ? -p.nz : 0);
        if ((unsigned)Y >= (unsigned)p.ny || (unsigned)Z >= (unsigned)p.nz) {
          face = true;
          continue;
        }
        const uint8_t* row = flags + (x + sy * Y + sz * Z);
        const uint4 w4 = *reinterpret_cast<const uint4*>(row);
        const unsigned w[4] = {w4.x, w4.y, w4.z, w4.w};
        const bool centre = dy == 0 && dz == 0;
        if (!centre) {
#pragma unroll
          for (int k = 0; k < 4; ++k) near[k] |= w[k];
        }
        if (dy == 0 || dz == 0) {  // the links along x too
          const unsigned before = xlo ? 0u : row[-1], after = xhi ? 0u : row[16];
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            near[k] |= (w[k] << 8) | (k ? w[k - 1] >> 24 : before);
            near[k] |= (w[k] >> 8) | ((k < 3 ? w[k + 1] : after) << 24);
          }
        }
        if (centre) {
#pragma unroll
          for (int k = 0; k < 4; ++k) own[k] = w[k] & 0x0f0f0f0fu;
        }
      }
    bool bad = false;
    uint4 out;
    unsigned* o = &out.x;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const unsigned one = 0x01010101u, b0 = own[k] & one, b1 = (own[k] >> 1) & one, b2 = (own[k] >> 2) & one,
                     b3 = (own[k] >> 3) & one;
      bad = bad || b0 + b1 + b2 + b3 != one;                  // each byte one kind (no carry: at most 4)
      bad = bad || (b0 & ((near[k] >> 2) & one)) != 0u;       // a liquid cell next to gas
      const unsigned wall = (near[k] >> 3) & one;
      o[k] = own[k] | (wall * (unsigned)(NEARB | NEARW)) | (face ? one * (unsigned)NEARB : 0u);
    }
    if (xlo) o[0] |= NEARB;  // (beyond a non-periodic face: a wall)
    if (xhi) o[3] |= (unsigned)NEARB << 24;
    if (bad) atomicOr(err, ERRB_STATE);
    *reinterpret_cast<uint4*>(flags + i) = out;
  }
}

// one 8- or 16-byte store of VEC doubles
template <int VEC>
struct VecT;
template <>
struct VecT<1> {
  using T = double;
  static __device__ __forceinline__ T of(const double* a) { return a[0]; }
};
template <>
struct VecT<2> {
  using T = double2;
  static __device__ __forceinline__ T of(const double* a) { return make_double2(a[0], a[1]); }
};

// The fields of VEC x-adjacent cells per thread (VEC = 2 where N is even, so
// that every plane's pairs are 16-byte aligned).  The velocities, three per
// cell, go through shared memory so that a warp's stores are whole sectors.
// The 512x256x256 read-back (every field, FP32 form) writes 6.7 GB: 2.54 ms
// with a cell per thread and the velocities stored 24 bytes apart, 1.83 ms so
// (0.54 of the copy bandwidth).
template <int P, int VEC>
__global__ void __launch_bounds__(128) k_fields(Par p, View<P> v, unsigned mask, uint8_t* oflags, double* of,
                                                double* om, double* ophi, double* orho, double* ou) {
  using S = typename Form<P>::S;
  using R = typename Form<P>::R;
  constexpr bool SH = Form<P>::SH;
  struct alignas(8 * VEC) Vec { double a[VEC]; };
  struct alignas(sizeof(S) * VEC) SVec { S a[VEC]; };
  __shared__ double su[128 * 3 * VEC];
  const size_t N = (size_t)p.N;
  const long long n = p.N / VEC;
  for (long long b0 = (long long)blockIdx.x * 128; b0 < n; b0 += (long long)gridDim.x * 128) {
    const long long t = b0 + threadIdx.x;
    const bool in = t < n;
    const long long i = t * VEC;
    double ux[VEC][3];
    if (in) {
      uint8_t k[VEC];
      bool any = false, fl[VEC];
#pragma unroll
      for (int c = 0; c < VEC; ++c) {
        k[c] = v.flags[i + c] & KIND;
        fl[c] = is_fluid(k[c]);
        any = any || fl[c];
      }
      any = any && (of || om || orho || ou);  // (kinds and fill levels alone read no population)
      R f[VEC][19];
      if (any) {
#pragma unroll
        for (int q = 0; q < 19; ++q) {
          const SVec w = *reinterpret_cast<const SVec*>(v.fin + (size_t)q * N + i);
#pragma unroll
          for (int c = 0; c < VEC; ++c) {
            R val;
            if constexpr (P == P16) val = __half2float(w.a[c]);
            else val = w.a[c];
            f[c][q] = fl[c] ? val : R(0);
          }
        }
      } else {
#pragma unroll
        for (int q = 0; q < 19; ++q)
#pragma unroll
          for (int c = 0; c < VEC; ++c) f[c][q] = R(0);
      }
      if (of) {
#pragma unroll
        for (int q = 0; q < 19; ++q) {
          Vec w;
#pragma unroll
          for (int c = 0; c < VEC; ++c) {
            w.a[c] = (double)f[c][q];
            if constexpr (SH) {
              if (any) w.a[c] = fl[c] ? w.a[c] + wq<double>(q) : 0.0;
            }
          }
          __stcs(reinterpret_cast<typename VecT<VEC>::T*>(of + (size_t)q * N + i), VecT<VEC>::of(w.a));
        }
      }
      Vec wm, wp, wr;
#pragma unroll
      for (int c = 0; c < VEC; ++c) {
        R rho = R(0), vx = R(0), vy = R(0), vz = R(0);
        if (fl[c]) moments_post<R, SH>(p, f[c], rho, vx, vy, vz);
        const double rhof = fl[c] ? rho_full<SH>(rho) : 0.0;
        if (oflags) oflags[i + c] = k[c];
        wm.a[c] = !om ? 0.0 : (k[c] == IFC ? v.m[i + c] : (k[c] == LIQ ? rhof : 0.0));
        double ph = 0.0;
        if (k[c] == LIQ) ph = 1.0;
        else if (ophi && (k[c] == IFC || (k[c] == GAS && p.freeze))) ph = (double)v.phin[i + c];
        wp.a[c] = ph;
        wr.a[c] = rhof;
        ux[c][0] = (double)vx; ux[c][1] = (double)vy; ux[c][2] = (double)vz;
      }
      using T = typename VecT<VEC>::T;
      if (om) __stcs(reinterpret_cast<T*>(om + i), VecT<VEC>::of(wm.a));
      if (ophi) __stcs(reinterpret_cast<T*>(ophi + i), VecT<VEC>::of(wp.a));
      if (orho) __stcs(reinterpret_cast<T*>(orho + i), VecT<VEC>::of(wr.a));
    }
    if (ou) {
      if (in) {
#pragma unroll
        for (int c = 0; c < VEC; ++c)
#pragma unroll
          for (int a = 0; a < 3; ++a) su[(threadIdx.x * VEC + c) * 3 + a] = ux[c][a];
      }
      __syncthreads();
      const long long left = (n - b0 < 128 ? n - b0 : 128) * VEC * 3;
      double* dst = ou + b0 * VEC * 3;
      for (int e = threadIdx.x; e < left; e += 128) __stcs(dst + e, su[e]);
      __syncthreads();
    }
  }
}

// M = sum_liquid rho + sum_interface m: per-block partials in cell order.
template <int P>
__global__ void __launch_bounds__(256) k_mass_partials(Par p, View<P> v, double* __restrict__ partials,
                                                       long long per_block) {
  using R = typename Form<P>::R;
  __shared__ double red[8];
  const size_t N = (size_t)p.N;
  long long lo = (long long)blockIdx.x * per_block;
  long long hi = lo + per_block < p.N ? lo + per_block : p.N;
  double s = 0.0;
  for (long long i = lo + threadIdx.x; i < hi; i += blockDim.x) {
    uint8_t k = v.flags[i] & KIND;
    if (!p.owned_all) {
      int x, y, z;
      coords(p, i, x, y, z);
      if (!owned(p, x, y, z)) continue;
    }
    if (k == LIQ) {
      R r = R(0);
#pragma unroll
      for (int q = 0; q < 19; ++q) r += ldq<P>(v.fin, (size_t)q * N + i, q);
      s += rho_full<Form<P>::SH>(r);
    } else if (k == IFC) {
      s += v.m[i];
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0)
    partials[blockIdx.x] = ((red[0] + red[1]) + (red[2] + red[3])) + ((red[4] + red[5]) + (red[6] + red[7]));
}

static int grid_for(long long n, int block) {
  long long g = (n + block - 1) / block;
  if (g > 152LL * 32) g = 152LL * 32;
  if (g < 1) g = 1;
  return (int)g;
}

template <int P>
int launch_init_pre(const Par& p, const View<P>& v, const double* f, const double* phi, const double* rho_in,
                    const double* u_in, const double* noise, double* keep_f0, cudaStream_t st) {
  k_init_pre<P><<<grid_for(p.N, 128), 128, 0, st>>>(p, v, f, phi, rho_in, u_in, noise, keep_f0);
  return (int)cudaGetLastError();
}
template <int P>
int launch_init_post(const Par& p, const View<P>& v, const double* f, const double* m, const double* phi,
                     cudaStream_t st) {
  k_init_post<P><<<grid_for(p.N, 128), 128, 0, st>>>(p, v, f, m, phi);
  return (int)cudaGetLastError();
}
int launch_prepare_flags(const Par& p, uint8_t* flags, int* err, cudaStream_t st) {
  if ((p.nx & 15) == 0)
    k_prepare_flags16<<<grid_for(p.N / 16, 256), 256, 0, st>>>(p, flags, err);
  else
    k_prepare_flags<<<grid_for(p.N, 256), 256, 0, st>>>(p, flags, err);
  return (int)cudaGetLastError();
}
template <int P>
int launch_fields(const Par& p, const View<P>& v, unsigned mask, void* const* out, cudaStream_t st) {
  void* ptr[6] = {nullptr, nullptr, nullptr, nullptr, nullptr, nullptr};
  int k = 0;
  for (int b = 0; b < 6; ++b)
    if (mask & (1u << b)) ptr[b] = out[k++];
  // (the callers' buffers need not be 16-byte aligned)
  bool pairs = (p.N & 1) == 0;
  for (int b = 1; b < 6; ++b) pairs = pairs && ((uintptr_t)ptr[b] & 15) == 0;
  auto kernel = pairs ? k_fields<P, 2> : k_fields<P, 1>;
  kernel<<<grid_for(pairs ? p.N / 2 : p.N, 128), 128, 0, st>>>(p, v, mask, (uint8_t*)ptr[0], (double*)ptr[1],
                                                               (double*)ptr[2], (double*)ptr[3], (double*)ptr[4],
                                                               (double*)ptr[5]);
  return (int)cudaGetLastError();
}
template <int P>
int launch_total_mass(const Par& p, const View<P>& v, double* partials, long long nparts, double* tmp,
                      int tmp_blocks, double* out, cudaStream_t st) {
  long long per = (p.N + nparts - 1) / nparts;
  if (per < 1) per = 1;
  long long nb = (p.N + per - 1) / per;
  k_mass_partials<P><<<(int)nb, 256, 0, st>>>(p, v, partials, per);
  return launch_reduce(partials, nb, tmp, tmp_blocks, v.lost, out, st);
}

#define FSL_INST(P)                                                                                          \
  template int launch_init_pre<P>(const Par&, const View<P>&, const double*, const double*, const double*,  \
                                  const double*, const double*, double*, cudaStream_t);                     \
  template int launch_init_post<P>(const Par&, const View<P>&, const double*, const double*, const double*, \
                                   cudaStream_t);                                                           \
  template int launch_fields<P>(const Par&, const View<P>&, unsigned, void* const*, cudaStream_t);          \
  template int launch_total_mass<P>(const Par&, const View<P>&, double*, long long, double*, int, double*,  \
                                    cudaStream_t);
FSL_INST(P64)
FSL_INST(P32)
FSL_INST(P16)
#undef FSL_INST

}  // namespace fsl
