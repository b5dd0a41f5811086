// pair_common.cuh -- what the passes over unordered pairs share: the early exit
// of a relaxation chunk, the pair record, the four-double record.
#pragma once

#include "mxe_internal.cuh"

namespace mxe {

__device__ __forceinline__ bool skin_violated(const Ctrl* c) {
  double disp = sqrt(__longlong_as_double((long long)c->disp2_bits));
  double smax = __longlong_as_double((long long)c->smax_bits);
  return 2.0 * disp + kSqrt6 * (smax - c->sigma_max_build) > c->skin;
}

// Uniform early exit of the relaxation chunk.  Returns true if the kernel must
// stop.  The skin test runs once per launch, on thread 0 of block 0 (on the
// 1:64 FP64 pipe a test per block kept the FP64 pipe a quarter busy and held
// every block at the barrier behind it); each block reads the halt flag
// through one thread.  Blocks that start before block 0 sets the flag run the
// pass on the old lists (valid arrays, so every access stays in bounds); a
// halted pass is always evaluated again after the rebuild, so that output is
// never used.  Every thread of the block must call this before any early
// return.
__device__ __forceinline__ bool chunk_halted(const PassArgs& A) {
  if (A.ctrl == nullptr) return false;
  __shared__ int halt;
  if (threadIdx.x == 0) {
    int h = A.ctrl->halted ? 1 : 0;
    if (!h && blockIdx.x == 0 && A.check_skin && skin_violated(A.ctrl)) {
      A.ctrl->reason = kReasonRebuild;
      A.ctrl->halted = 1;
      h = 1;
    }
    halt = h;
  }
  __syncthreads();
  return halt != 0;
}

// The record of unordered pair p: owner site i, the entry of j in row i (j with
// its image code), that entry's index tp and the index tr of the reverse
// entry (i in row j).  The records are built from the current lists, so they
// are consistent with them by construction; every index is still bounded
// (a bad record sets the overflow flag and the pair is skipped).  Building
// with MXE_DEBUG_CHECKS also checks that tp and tr lie in their rows.
struct PairRef {
  int64_t i, j;
  uint32_t code;
  int tp, tr;
};
template <typename Args>
__device__ __forceinline__ bool load_pair(const Args& A, const int4* __restrict__ rec, int64_t p, PairRef& r) {
  const int4 v = __ldg(&rec[p]);
  r.i = v.x;
  r.j = (uint32_t)v.y & kIdxMask;
  r.code = (uint32_t)v.y >> kCodeShift;
  r.tp = v.z;
  r.tr = v.w;
  bool ok = (uint64_t)(uint32_t)v.x < (uint64_t)A.n && (uint64_t)r.j < (uint64_t)A.n &&
            (uint64_t)(uint32_t)v.z < (uint64_t)A.n_ent && (uint64_t)(uint32_t)v.w < (uint64_t)A.n_ent;
#ifdef MXE_DEBUG_CHECKS
  ok = ok && r.tp >= A.nb_off[r.i] && r.tp < A.nb_off[r.i + 1] && A.nb_ent[r.tp] == (uint32_t)v.y &&
       r.tr >= A.nb_off[r.j] && r.tr < A.nb_off[r.j + 1] && (A.nb_ent[r.tr] & kIdxMask) == (uint32_t)r.i;
#endif
  if (!ok) atomicOr(A.flags, kFlagOverflow);
  return ok;
}

// float -> double on bits (no FP64 instruction; subnormals give zero)
__device__ __forceinline__ double widen(float x) {
  const unsigned u = __float_as_uint(x), e = (u >> 23) & 0xffu;
  const unsigned hi = (u & 0x80000000u) | ((e == 255u ? 0x7ffu : e + 896u) << 20) | ((u >> 3) & 0xfffffu);
  return e == 0 ? 0.0 : __hiloint2double((int)hi, (int)(u << 29));
}

struct alignas(32) Dbl4 {
  double x, y, z, w;
};

// ---------------------------------------------------------------- geometry of a pair
// separation and node offsets (sqrt(6) sigma) of a pair from the FP64 state
struct PairGeom {
  double d[3], D2, s_i, s_j;
};
// minimum image of q_j - q_i; the division by the box only where a component
// reaches half the box (pairs of the list are nearer than that elsewhere)
template <typename Args>
__device__ __forceinline__ void pair_geometry(const DevGrid& g0, const Args& A, int64_t i, int64_t j, PairGeom& G) {
  const int64_t n = A.n;
  const DevGrid* gp = A.batch.nsys ? &A.batch.grids[A.batch.sys_of[i]] : nullptr;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    double da = __ldg(&A.q[a * n + j]) - __ldg(&A.q[a * n + i]);
    const double L = gp ? gp->L[a] : g0.L[a];
    // high words of positive doubles order as the doubles do
    if ((__double2hiint(da) & 0x7fffffff) >= __double2hiint(L) - (1 << 20)) {
      const double invL = gp ? gp->invL[a] : g0.invL[a];
      da -= L * rint(da * invL);
    }
    G.d[a] = da;
  }
  G.D2 = G.d[0] * G.d[0] + G.d[1] * G.d[1] + G.d[2] * G.d[2];
  G.s_i = kSqrt6 * __ldg(&A.sigma[i]);
  G.s_j = kSqrt6 * __ldg(&A.sigma[j]);
}

}  // namespace mxe
