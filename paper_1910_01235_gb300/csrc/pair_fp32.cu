// pair_fp32.cu -- the relaxation's pair passes of the FP32 modes (MIXED and
// float-float contexts: FP32 node arithmetic, float4 records), two nodes at a
// time in packed FP32 instructions.
//
// What bounds them: instruction issue.  One node at a time the force pass
// issued 771 instructions per pair (89 % of the issue slots, FMA pipe 61 %,
// XU 35 %).  The two nodes +-s of an axis run through the same operations, so
// everything but the reciprocal square roots, the exponentials and the
// saturation is one fma.rn.f32x2 (or add, mul) for both.  With a geometric-mean
// cross pair the like terms are squares of exp2 halves a, b and the cross term
// is a b: two exponentials per node instead of three on the XU pipe.
// Their error is that of three exponentials: the rounding of the argument is half
// as large in a half, and the larger part (34 alloys of 256 to 256,000 sites,
// geometric mean rms against FP64: forces 4.20e-7 eV/A and 4.19e-7, width
// derivatives 3.96e-7 and 4.03e-7, halves first).
// Measured: 522 instructions per pair; forces at 256,000 sites (6.9 M pairs of the
// binary alloy) 150 -> 136 us, densities 90 -> 80 us, slab forces (241 M pairs)
// 6.96 -> 5.32 ms.  Issue 67 %; the rest is the FMA pipe, which a packed
// instruction holds twice as long, and the latency of the first loads.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>

#include "pair_common.cuh"

namespace mxe {
namespace {

// ---------------------------------------------------------------- packed FP32
using f2 = unsigned long long;
__device__ __forceinline__ f2 pk(float a, float b) {
  f2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ f2 dup(float a) { return pk(a, a); }
__device__ __forceinline__ void unpk(f2 v, float& a, float& b) { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v)); }
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) {
  f2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ f2 mul2(f2 a, f2 b) {
  f2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f2 add2(f2 a, f2 b) {
  f2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ float sum2(f2 v) {
  float a, b;
  unpk(v, a, b);
  return a + b;
}
__device__ __forceinline__ float ex2f(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float rsqf(float x) {
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ f2 ex2p(f2 v) {
  float a, b;
  unpk(v, a, b);
  return pk(ex2f(a), ex2f(b));
}
__device__ __forceinline__ f2 sat2(f2 v, float w) {
  float a, b;
  unpk(v, a, b);
  return pk(__saturatef(a * w), __saturatef(b * w));
}

// The potential as these kernels read it, constants doubled for packed
// operands: exp2(c0 + c1 r) per term (c1 negative), density terms first.  half:
// the like pair terms' halves (c0 / 2, c1 / 2) of a geometric-mean alloy.
struct Pot32 {
  float2 c0[5], c1[5], half0[2], half1[2];
  float lam_n[5];  // minus the decay rate
  float rs, inv_w, dS_scale;
  float2 rs_n2, scale2;
  int n_f, n_phi;
  int8_t phi_of[2][2], f_of[2][2];
};
__device__ __forceinline__ f2 ld(const float2& v) { return pk(v.x, v.y); }

template <int S>
struct Site32 {
  float p[3], sig, x[S];
};
template <int S>
__device__ __forceinline__ void load32(const PassArgs& A, int64_t j, Site32<S>& d) {
  const float4 P = __ldg(&A.pos32[j]), X = __ldg(&A.x32[j]);
  d.p[0] = P.x;
  d.p[1] = P.y;
  d.p[2] = P.z;
  d.sig = P.w;
  d.x[0] = X.x;
  if (S > 1) d.x[S > 1 ? 1 : 0] = X.y;
}
// q_j - q_i from the cell-relative positions and the image code
__device__ __forceinline__ void separation32(const DevGrid& g, const float* pi, const float* pj, uint32_t code, float* d) {
  const int c = (int)code;
  const int s[3] = {c / 9 - 1, (c / 3) % 3 - 1, c % 3 - 1};
#pragma unroll
  for (int a = 0; a < 3; ++a) d[a] = (pj[a] - pi[a]) + (float)s[a] * g.h_f[a];
}
__device__ __forceinline__ DevGrid grid_of(const DevGrid& g, const Batch& B, int64_t i) {
  return B.nsys ? B.grids[B.sys_of[i]] : g;
}

// two nodes: r, 1/r, S(r) and dS/dr
__device__ __forceinline__ void nodes2(const Pot32& P, f2 r2, f2& r, f2& rinv, f2& t, f2& t2, f2& Sw) {
  float a, b;
  unpk(r2, a, b);
  rinv = pk(rsqf(a), rsqf(b));
  r = mul2(r2, rinv);
  t = sat2(add2(r, ld(P.rs_n2)), P.inv_w);
  t2 = mul2(t, t);
  Sw = fma2(mul2(t2, t), fma2(t, fma2(dup(-6.f), t, dup(15.f)), dup(-10.f)), dup(1.f));
}
__device__ __forceinline__ f2 dswitch2(const Pot32& P, f2 t, f2 t2) {
  const f2 u = fma2(t, dup(-1.f), dup(1.f));
  return mul2(mul2(t2, mul2(u, u)), ld(P.scale2));
}
// one point (the mean separation)
__device__ __forceinline__ void point(const Pot32& P, float r2, float& r, float& rinv, float& S, float& dS) {
  rinv = rsqf(r2);
  r = r2 * rinv;
  const float t = __saturatef((r - P.rs) * P.inv_w), t2 = t * t, u = 1.f - t;
  S = fmaf(t2 * t, fmaf(t, fmaf(-6.f, t, 15.f), -10.f), 1.f);
  dS = (t2 * (u * u)) * P.dS_scale;
}

template <int S, int TAB>
__device__ __forceinline__ int phi_id(const Pot32& P, int k, int l) {
  return TAB ? k + l : (int)P.phi_of[k][l];
}
template <int S, int TAB>
__device__ __forceinline__ int f_id(const Pot32& P, int k, int l) {
  return TAB ? l : (int)P.f_of[k][l];
}

// ---------------------------------------------------------------- densities
// TAB 1 or 2: the binary pattern (Tables<1>); 0: tables read at run time.
// Grid-stride (a resident grid, see resident_grid).
template <int S, int TAB>
__global__ void __launch_bounds__(256) k_rdensity32(const __grid_constant__ Pot32 P, const __grid_constant__ DevGrid g0,
                                                    const __grid_constant__ PassArgs A,
                                                    const int4* __restrict__ pair_rec, int64_t npair,
                                                    float4* __restrict__ dens) {
  constexpr int NF = S;
  pdl_wait();
  pdl_trigger();
  if (chunk_halted(A)) return;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < npair; p += stride) {
    PairRef pr;
    if (!load_pair(A, pair_rec, p, pr)) continue;
    const DevGrid g = grid_of(g0, A.batch, pr.i);
    Site32<S> si, sj;
    load32<S>(A, pr.i, si);
    load32<S>(A, pr.j, sj);
    float d[3];
    separation32(g, si.p, sj.p, pr.code, d);
    const float s_i = 2.44948974f * si.sig, s_j = 2.44948974f * sj.sig;
    const float D2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2];
    float fst[NF];
    {
      float r, rinv, Sw, dS;
      point(P, D2, r, rinv, Sw, dS);
#pragma unroll
      for (int v = 0; v < NF; ++v) fst[v] = TAB || v < P.n_f ? ex2f(fmaf(P.c1[v].x, r, P.c0[v].x)) * Sw : 0.f;
    }
    f2 fav[NF];
#pragma unroll
    for (int v = 0; v < NF; ++v) fav[v] = dup(0.f);
#pragma unroll
    for (int site = 0; site < 2; ++site) {
      const float s = site == 0 ? s_i : s_j;
      const f2 base = dup(fmaf(s, s, D2)), s2 = pk(s + s, -(s + s));
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        f2 r, rinv, t, t2, Sw;
        nodes2(P, fma2(dup(d[a]), s2, base), r, rinv, t, t2, Sw);
#pragma unroll
        for (int v = 0; v < NF; ++v)
          if (TAB || v < P.n_f) fav[v] = fma2(ex2p(fma2(ld(P.c1[v]), r, ld(P.c0[v]))), Sw, fav[v]);
      }
    }
    int bad = D2 < (float)(kRMin * kRMin);
    const float near = (float)kRMin + fmaxf(s_i, s_j);
    if (D2 < near * near) {  // rare: the exact node distances
      for (int site = 0; site < 2; ++site) {
        const float s = site == 0 ? s_i : s_j;
        for (int a = 0; a < 3; ++a) {
          const float base = D2 + s * s, tw = 2.f * s * d[a];
          bad |= (base + tw) < (float)(kRMin * kRMin);
          bad |= (base - tw) < (float)(kRMin * kRMin);
        }
      }
    }
    // each entry receives its own site's contributions from the other site
    float ci[4] = {0.f, 0.f, 0.f, 0.f}, cj[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int k = 0; k < S; ++k)
#pragma unroll
      for (int l = 0; l < S; ++l) {
        const int fo = f_id<S, TAB>(P, k, l);
#pragma unroll
        for (int v = 0; v < NF; ++v)
          if (fo == v) {
            const float fa = sum2(fav[v]);
            ci[k] += sj.x[l] * fst[v];
            ci[2 + k] += sj.x[l] * fa;
            cj[k] += si.x[l] * fst[v];
            cj[2 + k] += si.x[l] * fa;
          }
      }
    if constexpr (S == 1 || TAB != 0) {  // one density for every species
      float2* d2 = reinterpret_cast<float2*>(dens);
      d2[pr.tp] = make_float2(ci[0], ci[2]);
      d2[pr.tr] = make_float2(cj[0], cj[2]);
    } else {
      dens[pr.tp] = make_float4(ci[0], ci[1], ci[2], ci[3]);
      dens[pr.tr] = make_float4(cj[0], cj[1], cj[2], cj[3]);
    }
    if (bad) atomicOr(A.flags, kFlagGeometry);
  }
}

// ---------------------------------------------------------------- forces
// One thread per pair.  TAB 2: the binary pattern with a geometric-mean cross
// term.
template <int S, int TAB>
__global__ void __launch_bounds__(256) k_rforce32(const __grid_constant__ Pot32 P, const __grid_constant__ DevGrid g0,
                                                  const __grid_constant__ PassArgs A,
                                                  const int4* __restrict__ pair_rec, int64_t npair,
                                                  float4* __restrict__ frc) {
  constexpr int NF = S, NP = S * (S + 1) / 2, NT = NF + NP;
  pdl_wait();
  pdl_trigger();
  if (A.ctrl != nullptr && A.ctrl->halted) return;
  const int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (p >= npair) return;
  PairRef pr;
  if (!load_pair(A, pair_rec, p, pr)) return;
  const DevGrid g = grid_of(g0, A.batch, pr.i);
  Site32<S> si, sj;
  load32<S>(A, pr.i, si);
  load32<S>(A, pr.j, sj);
  const float4 abi = __ldg(&A.ab32[2 * pr.i]), abj = __ldg(&A.ab32[2 * pr.j]);
  const float ai[2] = {abi.x, abi.z}, bi[2] = {abi.y, abi.w}, aj[2] = {abj.x, abj.z}, bj[2] = {abj.y, abj.w};
  float d[3];
  separation32(g, si.p, sj.p, pr.code, d);
  const float s_i = 2.44948974f * si.sig, s_j = 2.44948974f * sj.sig;
  const float D2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2];
  // weights of the terms at the nodes and at the static point
  float C[NT], cfs[NF];
#pragma unroll
  for (int u = 0; u < NT; ++u) C[u] = 0.f;
#pragma unroll
  for (int v = 0; v < NF; ++v) cfs[v] = 0.f;
#pragma unroll
  for (int k = 0; k < S; ++k)
#pragma unroll
    for (int l = 0; l < S; ++l) {
      const int po = phi_id<S, TAB>(P, k, l), fo = f_id<S, TAB>(P, k, l);
#pragma unroll
      for (int u = 0; u < NP; ++u)
        if (po == u) C[NF + u] += si.x[k] * sj.x[l];
#pragma unroll
      for (int v = 0; v < NF; ++v)
        if (fo == v) {
          C[v] += bi[k] * sj.x[l] + bj[k] * si.x[l];
          cfs[v] += ai[k] * sj.x[l] + aj[k] * si.x[l];
        }
    }
  float Gs = 0.f;
  {
    float r, rinv, Sw, dS;
    point(P, D2, r, rinv, Sw, dS);
#pragma unroll
    for (int v = 0; v < NF; ++v)
      if (TAB || v < P.n_f) {
        const float e = ex2f(fmaf(P.c1[v].x, r, P.c0[v].x));
        Gs += cfs[v] * (e * fmaf(P.lam_n[v], Sw, dS));
      }
    Gs *= rinv;
  }
  f2 W1[NT], W2[NT];  // weights, and times minus the decay rates
#pragma unroll
  for (int u = 0; u < NT; ++u) {
    W1[u] = dup(C[u]);
    W2[u] = dup(C[u] * P.lam_n[u]);
  }
  f2 T = dup(0.f), U[3] = {dup(0.f), dup(0.f), dup(0.f)};
  float Vs[2];
#pragma unroll
  for (int site = 0; site < 2; ++site) {
    const float s = site == 0 ? s_i : s_j;
    const f2 base = dup(fmaf(s, s, D2)), s1 = pk(s, -s), s2 = pk(s + s, -(s + s));
    f2 V = dup(0.f);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const f2 dd = dup(d[a]);
      f2 r, rinv, t, t2, Sw;
      nodes2(P, fma2(dd, s2, base), r, rinv, t, t2, Sw);
      const f2 dS = dswitch2(P, t, t2);
      f2 A1, A2;
      {
        const f2 e = ex2p(fma2(ld(P.c1[0]), r, ld(P.c0[0])));
        A1 = mul2(W1[0], e);
        A2 = mul2(W2[0], e);
      }
      auto add_term = [&](int u, f2 e) {
        A1 = fma2(W1[u], e, A1);
        A2 = fma2(W2[u], e, A2);
      };
#pragma unroll
      for (int v = 1; v < NF; ++v)
        if (TAB || v < P.n_f) add_term(v, ex2p(fma2(ld(P.c1[v]), r, ld(P.c0[v]))));
      if constexpr (TAB == 2) {
        const f2 ha = ex2p(fma2(ld(P.half1[0]), r, ld(P.half0[0])));
        const f2 hb = ex2p(fma2(ld(P.half1[1]), r, ld(P.half0[1])));
        add_term(NF + 0, mul2(ha, ha));
        add_term(NF + 1, mul2(ha, hb));
        add_term(NF + 2, mul2(hb, hb));
      } else {
#pragma unroll
        for (int u = 0; u < NP; ++u)
          if (TAB || u < P.n_phi) add_term(NF + u, ex2p(fma2(ld(P.c1[NF + u]), r, ld(P.c0[NF + u]))));
      }
      const f2 w = mul2(fma2(A1, dS, mul2(A2, Sw)), rinv);
      T = add2(T, w);
      U[a] = fma2(w, s1, U[a]);
      // (d_a + s) w_+ - (d_a - s) w_-
      V = fma2(w, add2(pk(d[a], -d[a]), dup(s)), V);
    }
    Vs[site] = 2.44948974f * sum2(V);
  }
  const float inv12 = 1.0f / 12.0f;
  const float Tt = sum2(T) * inv12 + Gs;
  const float fx = -(d[0] * Tt + sum2(U[0]) * inv12), fy = -(d[1] * Tt + sum2(U[1]) * inv12),
              fz = -(d[2] * Tt + sum2(U[2]) * inv12);
  frc[pr.tp] = make_float4(fx, fy, fz, Vs[0] * inv12);
  frc[pr.tr] = make_float4(-fx, -fy, -fz, Vs[1] * inv12);
}

Pot32 make_pot32(const DevPot& P) {
  Pot32 Q = {};
  const int NF = P.S;
  auto put = [&](int u, const RadialFn& F) {
    Q.c0[u] = make_float2(F.c0, F.c0);
    Q.c1[u] = make_float2(-F.c1, -F.c1);
    Q.lam_n[u] = -F.lam_f;
  };
  for (int v = 0; v < P.n_f && v < NF; ++v) put(v, P.f[v]);
  for (int u = 0; u < P.n_phi && NF + u < 5; ++u) put(NF + u, P.phi[u]);
  if (P.tab == 1)
    for (int s = 0; s < 2; ++s) {
      const RadialFn& F = P.phi[2 * s];
      const double log2e = 1.4426950408889634;
      const float h0 = (float)(0.5 * (std::log2(F.A) + F.kappa * log2e)), h1 = (float)(-0.5 * F.lambda * log2e);
      Q.half0[s] = make_float2(h0, h0);
      Q.half1[s] = make_float2(h1, h1);
    }
  Q.rs = P.rs_f;
  Q.inv_w = P.inv_w_f;
  Q.dS_scale = P.dS_scale_f;
  Q.rs_n2 = make_float2(-P.rs_f, -P.rs_f);
  Q.scale2 = make_float2(P.dS_scale_f, P.dS_scale_f);
  Q.n_f = P.n_f;
  Q.n_phi = P.n_phi;
  for (int k = 0; k < 2; ++k)
    for (int l = 0; l < 2; ++l) {
      Q.phi_of[k][l] = P.phi_of[k][l];
      Q.f_of[k][l] = P.f_of[k][l];
    }
  return Q;
}

}  // namespace

cudaError_t launch_relax_pair32(bool force, const DevPot& P, const DevGrid& g, const PassArgs& A, const int4* pair_rec,
                                int64_t npair, void* out, cudaStream_t s) {
  if (A.n == 0 || npair == 0) return cudaSuccess;
  if (!pair_kernels_supported(P) || P.lj) return cudaErrorInvalidValue;
  const Pot32 Q = make_pot32(P);
  const int pt = pair_threads(A);
  // the density pass strides over a resident grid in a single system; the force
  // pass, and every pass of a batch, take one thread per pair
  auto run = [&](auto kernel, bool resident) {
    const int64_t blocks = resident ? resident_grid((const void*)kernel, pt, npair) : (npair + pt - 1) / pt;
    if (blocks < 0 || blocks > 0x7fffffff) return cudaErrorInvalidValue;
    return launch_pdl(kernel, dim3((unsigned)blocks), dim3(pt), 0, s, Q, g, A, pair_rec, npair, (float4*)out);
  };
  if (force) {
    if (P.S == 1) return run(k_rforce32<1, 0>, false);
    if (P.tab == 1) return P.cross_geo ? run(k_rforce32<2, 2>, false) : run(k_rforce32<2, 1>, false);
    return run(k_rforce32<2, 0>, false);
  }
  if (P.S == 1) return run(k_rdensity32<1, 0>, A.batch.nsys == 0);
  return P.tab == 1 ? run(k_rdensity32<2, 1>, A.batch.nsys == 0) : run(k_rdensity32<2, 0>, A.batch.nsys == 0);
}

}  // namespace mxe
