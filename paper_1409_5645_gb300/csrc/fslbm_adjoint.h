// fslbm_adjoint.h -- the state of a checkpointed reverse sweep and what the
// adjoint's translation units share: the host entry points (fslbm_adjoint.cu)
// and the reverse step's kernels, instantiated per precision form
// (fslbm_adjoint_p64/p32/p16.cu from fslbm_adjoint.cuh).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>
#include <initializer_list>

#include "fslbm.h"
#include "fslbm_dev.cuh"
#include "fslbm_handle.h"
#include "fslbm_kernels.h"


struct AdjointState {
  int nsteps = 0, K = 1, objective = 0, nck = 0;
  size_t fbytes = 0, rbytes = 0;
  void* ck_f = nullptr;
  double* ck_m = nullptr;
  void* ck_phi = nullptr;
  uint8_t* ck_flags = nullptr;
  void* seg_f = nullptr;  // K + 1 states of the segment being reversed
  double* seg_m = nullptr;
  void* seg_phi = nullptr;
  uint8_t* seg_flags = nullptr;
  int* flist = nullptr;  // [2][2N + 2]: liquid and interface cells of a flag field, their counts
                         // (double buffer: the fields before and after the step being reversed)
  double* Mh = nullptr;  // conversion reverse: final-mass and density adjoints, new-cell means
  double* rh = nullptr;
  double* ngb = nullptr;
  double* abar[2] = {nullptr, nullptr};
  double* P = nullptr;
  double* mbar[2] = {nullptr, nullptr};
  double* phibar[2] = {nullptr, nullptr};
  double* theta = nullptr;  // [0] lambda_+ [1] lambda_- [2..4] g
  double* red = nullptr;    // objective reductions
  double* dphi0 = nullptr;
  int conv0 = 0;
  long long conversions = 0;  // cell conversions inside the window
  double J = 0.0, gseed = 0.0;
  double fwd_ms = 0.0, adj_ms = 0.0;
  size_t bytes = 0;
  bool ready = false;
  bool reverse = false;  // every buffer of the reverse sweep is allocated (adj_alloc_reverse)
  bool live = false;  // belongs to the handle's current state (a new state ends it, its buffers may stay)
};

struct AdjBuffer {
  void** p;
  size_t bytes;
};
// All of the buffers (null before) or none: where one cannot be had, those
// before it are given back and null again.  (alloc: pointer to fill, bytes ->
// done, null where not; release: pointer)
template <class Alloc, class Release>
inline bool adj_alloc_all(AdjointState* A, std::initializer_list<AdjBuffer> bufs, Alloc alloc, Release release) {
  for (const AdjBuffer* b = bufs.begin(); b != bufs.end(); ++b) {
    if (alloc(b->p, b->bytes ? b->bytes : 16)) {
      A->bytes += b->bytes;
      continue;
    }
    while (b != bufs.begin()) {
      --b;
      release(*b->p);
      *b->p = nullptr;
      A->bytes -= b->bytes;
    }
    return false;
  }
  return true;
}
// the buffers of the reverse sweep, once per state
template <class Alloc, class Release>
inline bool adj_alloc_reverse(AdjointState* A, size_t N, Alloc alloc, Release release) {
  if (A->reverse) return true;
  const size_t K1 = (size_t)A->K + 1;
  A->reverse = adj_alloc_all(
      A,
      {{(void**)&A->abar[0], 19 * N * 8}, {(void**)&A->abar[1], 19 * N * 8}, {(void**)&A->P, 19 * N * 8},
       {(void**)&A->mbar[0], N * 8}, {(void**)&A->mbar[1], N * 8}, {(void**)&A->phibar[0], N * 8},
       {(void**)&A->phibar[1], N * 8}, {(void**)&A->theta, 64}, {(void**)&A->dphi0, N * 8},
       {&A->seg_f, A->fbytes * K1}, {(void**)&A->seg_m, N * 8 * K1}, {&A->seg_phi, A->rbytes * K1},
       {(void**)&A->seg_flags, N * K1}, {(void**)&A->Mh, N * 8}, {(void**)&A->flist, 2 * (2 * N + 2) * sizeof(int)},
       {(void**)&A->rh, N * 8}, {(void**)&A->ngb, N * 4 * 8}},
      alloc, release);
  return A->reverse;
}

// blocks of the objective's reduction, and the doubles of AdjointState::red:
// result, count, a block counter, then two partial sums per block
constexpr int ADJ_RED_BLOCKS = 152 * 2;
constexpr int ADJ_RED_DOUBLES = 8 + 2 * ADJ_RED_BLOCKS;

namespace fsl {

// the liquid and interface cells of a flag field (see k_adj_lists)
struct CellLists {
  int* liq;
  int* ifc;
  int* cnt;  // [0] liquid, [1] interface
};
void build_lists(const Par& p, const uint8_t* flags, const CellLists& L, cudaStream_t st);
}  // namespace fsl

// the handle's current populations and fill levels
inline void* cur_f(fslbm* h) { return h->cur ? h->fB : h->fA; }
inline void* cur_phi(fslbm* h) { return (h->par.freeze || !h->cur) ? h->phiA : h->phiB; }
// copies of the handle's state to and from a checkpoint (device to device, on the handle's stream)
int save_state(fslbm* h, void* f, double* m, void* phi, uint8_t* flags);
int restore_state(fslbm* h, const void* f, const double* m, const void* phi, const uint8_t* flags);
// the objective at the current state (J, its normalisation; sets the seed of dJ/dg_x)
template <int P>
int adj_objective(fslbm* h, double* J, double* norm);
// the reverse sweep over the recorded window (fslbm_adjoint_backward)
template <int P>
int adj_backward(fslbm* h);
