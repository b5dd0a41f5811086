// pair_table.cu -- the passes over unordered pairs with tabulated radial terms
// (radial_table.cuh): the geometry records of the accurate pass (every
// precision) and the relaxation's density and force passes of FP64 contexts.
//
// What bounds them: the direct FP64 kernels sit on the FP64 pipe (2 lanes per
// SM), the direct float-float kernel on instruction issue (two exponentials, a
// square root and a switch in float-float per node).  Here a node costs a
// 64-bit integer addition, a table row from shared memory (two or three
// 16-byte loads per term) and 20 to 36 FP32 operations per term.
//
// Measured (event time per launch, direct -> tabulated).  FP64, 19,652-site
// binary alloy (531 k pairs): forces 1127 -> 160 us, densities 709 -> 71 us,
// geometry 911 -> 140 us.  Float-float geometry: 6.9 M pairs of the binary
// alloy (which had the power form) 1.35 -> 0.92 ms, 23.3 M pairs of one species
// 3.54 -> 1.77 ms, 241 M pairs of the interstitial slab 52.6 -> 26.5 ms.  What
// bounds them now (ncu): the geometry kernels the shared-memory wavefronts
// (86 % float-float, 93 % FP64; 32 lanes reading random rows take about 12
// wavefronts per 16-byte load, 4 without bank conflicts), the force kernel those
// (82 %), instruction issue (65 %) and the FP64 pipe (48 %) together, the density
// kernel the wavefronts (86 %) and the FP64 pipe (64 %).  With the constant terms and the
// sums of the nodes in FP64 (207 FP64 instructions a pair and lane) the force
// kernel took 210 us, the FP64 pipe 84 % busy; with the direct evaluation
// called inside the table loop 9 us more; with 640 threads a block (96
// registers) 171 us, with 384 (160 registers) as with 512.
//
// Layout: one block per SM holds the whole table in shared memory (up to
// 224 KB) and strides over the pairs; the table is copied before the kernel
// waits for the previous one.
#include <cuda_runtime.h>

#include <algorithm>
#include <type_traits>

#include "pair_common.cuh"
#include "radial_table.cuh"

namespace mxe {
namespace {

// squared node distances in units of 2^-55: the static point, the common part
// of each site's nodes and the shifts 2 s |d_a|
struct PairNodes {
  long long w0, base[2], tw[2][3];
};
__device__ __forceinline__ int pair_nodes(const PairGeom& G, PairNodes& N) {
  int big = 0;
  N.w0 = tab_fixed(G.D2, big);
#pragma unroll
  for (int site = 0; site < 2; ++site) {
    const double s = site ? G.s_j : G.s_i;
    N.base[site] = tab_fixed(fma(s, s, G.D2), big);
    const double s2 = s + s;
#pragma unroll
    for (int a = 0; a < 3; ++a) N.tw[site][a] = tab_fixed(fabs(s2 * G.d[a]), big);
  }
  return big;
}

// the smallest of a pair's twelve squared node distances
__device__ __forceinline__ long long nearest_node(const PairNodes& N) {
  return min(N.base[0] - max(N.tw[0][0], max(N.tw[0][1], N.tw[0][2])),
             N.base[1] - max(N.tw[1][0], max(N.tw[1][1], N.tw[1][2])));
}

// float pair of x from its bits (no FP64 instruction): 24 bits, then the other
// 29; magnitudes below 2^-74 (a biased exponent of kNoFloatPair or less) give zero
constexpr int kNoFloatPair = 948;
__device__ __forceinline__ ff ff_bits(double x) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const int e = (int)((hi >> 20) & 0x7ff);
  if (e <= kNoFloatPair) return ff{0.f, 0.f};
  const unsigned sign = hi & 0x80000000u;
  const float h = __uint_as_float(sign | ((unsigned)(e - 896) << 23) | ((hi & 0xfffffu) << 3) | (lo >> 29));
  const float sc = __uint_as_float(sign | ((unsigned)(e - 948) << 23));
  return ff{h, (float)(lo & 0x1fffffffu) * sc};
}

// ---------------------------------------------------------------- direct evaluation
// Pairs the table does not cover (radial_table.cuh): FP64, one term at a time.
__device__ __noinline__ int direct_values(const DevPot& P, const PairGeom& G, double* __restrict__ st,
                                          double* __restrict__ av, double* __restrict__ ph) {
  int bad = G.D2 < kRMin * kRMin;
  for (int v = 0; v < P.n_f; ++v) st[v] = av[v] = 0.0;
  for (int u = 0; u < P.n_phi; ++u) ph[u] = 0.0;
#pragma unroll 1
  for (int k = 0; k < 13; ++k) {
    double r2 = G.D2;
    if (k < 12) {
      const double s = k < 6 ? G.s_i : G.s_j, d = G.d[(k / 2) % 3];
      r2 = fma(s, s, G.D2) + (k & 1 ? -2.0 : 2.0) * s * d;
      bad |= r2 < kRMin * kRMin;
    }
    const double r = sqrt(r2);
    const double t = fmin(fmax((r - P.rs) * P.inv_w, 0.0), 1.0);
    const double S = fma(t * t * t, fma(t, fma(-6.0, t, 15.0), -10.0), 1.0);
    for (int v = 0; v < P.n_f; ++v) {
      const double e = P.f[v].A * exp(P.f[v].kappa - P.f[v].lambda * r) * S;
      if (k == 12) st[v] = e;
      else av[v] += e;
    }
    for (int u = 0; u < P.n_phi && k < 12; ++u) ph[u] += P.phi[u].A * exp(P.phi[u].kappa - P.phi[u].lambda * r) * S;
  }
  return bad;
}

// T, U[3], V[2] (force sums of the 12 nodes) and Gs (static point) of one pair
__device__ __noinline__ void direct_forces(const DevPot& P, const PairGeom& G, const double* __restrict__ cfa,
                                           const double* __restrict__ cfs, const double* __restrict__ cphi,
                                           double* __restrict__ out) {
  for (int c = 0; c < 7; ++c) out[c] = 0.0;
#pragma unroll 1
  for (int k = 0; k < 13; ++k) {
    const int site = k / 6, a = (k / 2) % 3;
    const double s = (site == 0 ? G.s_i : G.s_j) * (k & 1 ? -1.0 : 1.0);
    const double r2 = k < 12 ? fma(s, s, G.D2) + 2.0 * s * G.d[a] : G.D2;
    const double r = sqrt(r2);
    const double t = fmin(fmax((r - P.rs) * P.inv_w, 0.0), 1.0), t2 = t * t, u1 = 1.0 - t;
    const double S = fma(t2 * t, fma(t, fma(-6.0, t, 15.0), -10.0), 1.0);
    const double dS = t2 * (u1 * u1) * (-30.0 * P.inv_w);
    double w = 0.0;
    for (int v = 0; v < P.n_f; ++v) {
      const RadialFn& F = P.f[v];
      w += (k < 12 ? cfa[v] : cfs[v]) * (F.A * exp(F.kappa - F.lambda * r) * (dS - F.lambda * S));
    }
    for (int u = 0; u < P.n_phi && k < 12; ++u) {
      const RadialFn& F = P.phi[u];
      w += cphi[u] * (F.A * exp(F.kappa - F.lambda * r) * (dS - F.lambda * S));
    }
    w /= r;
    if (k == 12) {
      out[6] = w;
    } else {
      out[0] += w;
      out[1 + a] += s * w;
      out[4 + site] += kSqrt6 * (k & 1 ? -1.0 : 1.0) * (G.d[a] + s) * w;
    }
  }
}

// ---------------------------------------------------------------- geometry records
// a sum of nodes: integer constant terms in units of 2^(k - kTabValueBias) and
// the float pair of the rest
struct NodeSum {
  long long c;
  ff p;
  int k;
};
constexpr int kSumHead = 5;  // bits above the nearest node's constant term: 12 nodes sum below 2^62
__device__ __forceinline__ double sum_value(const NodeSum& v, double*) {
  return fixed_double(v.c, v.k - kTabValueBias) + (widen(v.p.hi) + widen(v.p.lo));
}
__device__ __forceinline__ ff sum_value(const NodeSum& v, ff*) {
  // |c| < 2^62: the high word as a float, then what it left
  const int h = (int)(v.c >> 32);
  const float fh = (float)h;
  const long long rest = v.c - ((long long)(int)fh << 32);  // below 2^39
  const float fl = (float)(int)((rest + 128) >> 8);
  const float s = exp2f_bits(v.k - 128);  // k from 6 on; the units are below the floats' range
  return ff{fh * 0x1p-30f * s, fl * 0x1p-54f * s} + v.p;
}

template <typename R>
struct GeoOut;
template <>
struct GeoOut<ff> {
  using T = float2;
  static constexpr bool kFF = true;
  static __device__ __forceinline__ T put(ff v) { return make_float2(v.hi, v.lo); }
  static __device__ __forceinline__ uint4 two(ff a, ff b) {
    return make_uint4(__float_as_uint(a.hi), __float_as_uint(a.lo), __float_as_uint(b.hi), __float_as_uint(b.lo));
  }
  static __device__ __forceinline__ ff from(double v) { return ff_from_double(v); }
};
template <>
struct GeoOut<double> {
  using T = double;
  static constexpr bool kFF = false;
  static __device__ __forceinline__ T put(double v) { return v; }
  static __device__ __forceinline__ uint4 two(double a, double b) {
    return make_uint4((unsigned)__double2loint(a), (unsigned)__double2hiint(a), (unsigned)__double2loint(b),
                      (unsigned)__double2hiint(b));
  }
  static __device__ __forceinline__ double from(double v) { return v; }
};

__device__ __forceinline__ long long row_integer(uint4 a) {
  return (long long)(((unsigned long long)a.y << 32) | (a.x & 0xffffff00u));
}
template <int W, bool FFQ>
__device__ __forceinline__ ff row_rest(uint4 a, const uint4* t, float th, float tl) {
  if constexpr (FFQ) return tab_polyff(__uint_as_float(a.z), __uint_as_float(a.w), t[1], th, tl);
  else return tab_poly64(__uint_as_float(a.z), __uint_as_float(a.w), t[1], t[2], th, tl);
}
// the terms at one point, each on its own row's grid
template <int N, int W, bool FFQ, bool LOWS>
__device__ __forceinline__ void one_node(const RadialTab& Tb, const uint4* sm, long long w, int& low, NodeSum* s) {
  float th, tl;
  const uint4* row = tab_row<FFQ, LOWS>(Tb, sm, w, th, tl, low);
#pragma unroll
  for (int u = 0; u < N; ++u) {
    const uint4 a = row[u * W];
    s[u] = NodeSum{row_integer(a) >> kSumHead, row_rest<W, FFQ>(a, row + u * W, th, tl), (int)(a.x & 0xffu) + kSumHead};
  }
}
// empty sums on the grid of the pair's nearest node, where the terms are largest
template <int N, int W, bool FFQ, bool LOWS>
__device__ __forceinline__ void start_sums(const RadialTab& Tb, const uint4* sm, const PairNodes& D, int& low,
                                           NodeSum* s) {
  float th, tl;
  const uint4* row = tab_row<FFQ, LOWS>(Tb, sm, nearest_node(D), th, tl, low);
#pragma unroll
  for (int u = 0; u < N; ++u) s[u] = NodeSum{0, ff{0.f, 0.f}, (int)(row[u * W].x & 0xffu) + kSumHead};
}
template <int N, int W, bool FFQ, bool LOWS>
__device__ __forceinline__ void add_node(const RadialTab& Tb, const uint4* sm, long long w, int& low, NodeSum* s) {
  float th, tl;
  const uint4* row = tab_row<FFQ, LOWS>(Tb, sm, w, th, tl, low);
#pragma unroll
  for (int u = 0; u < N; ++u) {
    const uint4 a = row[u * W];
    const int sh = s[u].k - (int)(a.x & 0xffu);
    low |= sh;  // negative: over 2^5 times the nearest node's (no table has that)
    s[u].c += shift_right(row_integer(a), sh);
    tab_acc(s[u].p, row_rest<W, FFQ>(a, row + u * W, th, tl));
  }
}

constexpr int kTabThreads = 512;

// The record of every unordered pair (eam.cu: f_v static, 12 <f_v>, 12 <phi_u>)
// written to both of its entries.  R ff: float-float quality rows and records
// of float pairs (FP32 modes); R double: FP64 quality.
template <int S, int NP, typename R>
__global__ void __launch_bounds__(kTabThreads, 1) k_geo_tab(
    const __grid_constant__ DevPot P, const __grid_constant__ DevGrid g0, const __grid_constant__ PassArgs A,
    const __grid_constant__ RadialTab Tb, const int4* __restrict__ pair_rec, int64_t npair,
    typename GeoOut<R>::T* __restrict__ buf, GeoLayout L) {
  using O = GeoOut<R>;
  constexpr int NF = S, NT = NF + NP, W = O::kFF ? kTabWordsFF : kTabWords64;
  extern __shared__ uint4 sm[];
  tab_stage(Tb, sm);
  pdl_wait();
  pdl_trigger();
  __syncthreads();
  if (chunk_halted(A)) return;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < npair; p += stride) {
    PairRef pr;
    if (!load_pair(A, pair_rec, p, pr)) continue;
    PairGeom G;
    pair_geometry(g0, A, pr.i, pr.j, G);
    PairNodes N;
    const int big = pair_nodes(G, N);
    int low = 0;
    R val[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) val[c] = (R)0;
    auto evaluate = [&](auto lows) {
      constexpr bool kLows = decltype(lows)::value;
      NodeSum s[NT];
      one_node<NF, W, O::kFF, kLows>(Tb, sm, N.w0, low, s);
#pragma unroll
      for (int v = 0; v < NF; ++v) val[v] = sum_value(s[v], (R*)nullptr);
      start_sums<NT, W, O::kFF, kLows>(Tb, sm, N, low, s);
#pragma unroll 1
      for (int site = 0; site < 2; ++site) {
#pragma unroll 1
        for (int a = 0; a < 3; ++a) {
          add_node<NT, W, O::kFF, kLows>(Tb, sm, N.base[0] + N.tw[0][0], low, s);
          add_node<NT, W, O::kFF, kLows>(Tb, sm, N.base[0] - N.tw[0][0], low, s);
          // the next axis (registers rotate: one copy of the node code)
          const long long t = N.tw[0][0];
          N.tw[0][0] = N.tw[0][1];
          N.tw[0][1] = N.tw[0][2];
          N.tw[0][2] = t;
        }
        N.base[0] = N.base[1];
#pragma unroll
        for (int a = 0; a < 3; ++a) N.tw[0][a] = N.tw[1][a];
      }
#pragma unroll
      for (int v = 0; v < NF; ++v) val[NF + v] = sum_value(s[v], (R*)nullptr);
#pragma unroll
      for (int u = 0; u < NP; ++u) val[2 * NF + u] = sum_value(s[NF + u], (R*)nullptr);
    };
    // one branch per warp, not one per node: few warps have a pair this close
    bool below = false;
    if constexpr (O::kFF) {
      const long long w = min(nearest_node(N), N.w0);
      below = __any_sync(__activemask(), (unsigned)((unsigned long long)w >> 32) < Tb.main_hi);
    }
    if (below) evaluate(std::bool_constant<O::kFF>{});
    else evaluate(std::false_type{});
    if (big || low < 0) {
      double st[2], av[2], ph[3];
      const PairGeom H = G;
      if (direct_values(P, H, st, av, ph)) atomicOr(A.flags, kFlagGeometry);
#pragma unroll
      for (int v = 0; v < NF; ++v)
        if (v < P.n_f) {
          val[v] = O::from(st[v]);
          val[NF + v] = O::from(av[v]);
        }
#pragma unroll
      for (int u = 0; u < NP; ++u)
        if (u < P.n_phi) val[2 * NF + u] = O::from(ph[u]);
    }
    if (P.n_f == NF && P.n_phi == NP) {
      // 16-byte stores to plane A of each entry, then plane B
      uint4* oa = reinterpret_cast<uint4*>(buf + (int64_t)pr.tp * L.ca);
      uint4* oa2 = reinterpret_cast<uint4*>(buf + (int64_t)pr.tr * L.ca);
      typename O::T *ob = buf + L.b_off + (int64_t)pr.tp * L.cb, *ob2 = buf + L.b_off + (int64_t)pr.tr * L.cb;
#pragma unroll
      for (int v = 0; v < NF; ++v) oa[v] = oa2[v] = O::two(val[2 * v], val[2 * v + 1]);
      if constexpr (NP == 1) {
        *ob = *ob2 = O::put(val[2 * NF]);
      } else {
#pragma unroll
        for (int u = 0; u < (NP + 1) / 2; ++u)
          reinterpret_cast<uint4*>(ob)[u] = reinterpret_cast<uint4*>(ob2)[u] =
              O::two(val[2 * NF + 2 * u], val[2 * NF + 2 * u + 1]);
      }
    } else {
      typename O::T *oa = buf + (int64_t)pr.tp * L.ca, *oa2 = buf + (int64_t)pr.tr * L.ca;
      typename O::T *ob = buf + L.b_off + (int64_t)pr.tp * L.cb, *ob2 = buf + L.b_off + (int64_t)pr.tr * L.cb;
#pragma unroll
      for (int v = 0; v < NF; ++v)
        if (v < P.n_f) {
          oa[v] = oa2[v] = O::put(val[v]);
          oa[P.n_f + v] = oa2[P.n_f + v] = O::put(val[NF + v]);
        }
#pragma unroll
      for (int u = 0; u < NP; ++u)
        if (u < P.n_phi) ob[u] = ob2[u] = O::put(val[2 * NF + u]);
    }
  }
}

// ---------------------------------------------------------------- relaxation densities, FP64
template <int S, int TAB>
__global__ void __launch_bounds__(kTabThreads, 1) k_rdensity_tab(
    const __grid_constant__ DevPot P, const __grid_constant__ DevGrid g0, const __grid_constant__ PassArgs A,
    const __grid_constant__ RadialTab Tb, const int4* __restrict__ pair_rec, int64_t npair, Dbl4* __restrict__ dens) {
  using TB = Tables<TAB>;
  constexpr int NF = S, W = kTabWords64;
  extern __shared__ uint4 sm[];
  tab_stage(Tb, sm);
  pdl_wait();
  pdl_trigger();
  __syncthreads();
  if (chunk_halted(A)) return;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < npair; p += stride) {
    PairRef pr;
    if (!load_pair(A, pair_rec, p, pr)) continue;
    PairGeom G;
    pair_geometry(g0, A, pr.i, pr.j, G);
    PairNodes N;
    const int big = pair_nodes(G, N);
    int low = 0;
    NodeSum s[NF];
    double fst[NF], fav[NF];
    one_node<NF, W, false, false>(Tb, sm, N.w0, low, s);
#pragma unroll
    for (int v = 0; v < NF; ++v) fst[v] = sum_value(s[v], (double*)nullptr);
    start_sums<NF, W, false, false>(Tb, sm, N, low, s);
#pragma unroll 1
    for (int site = 0; site < 2; ++site) {
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        add_node<NF, W, false, false>(Tb, sm, N.base[0] + N.tw[0][a], low, s);
        add_node<NF, W, false, false>(Tb, sm, N.base[0] - N.tw[0][a], low, s);
      }
      N.base[0] = N.base[1];
#pragma unroll
      for (int a = 0; a < 3; ++a) N.tw[0][a] = N.tw[1][a];
    }
#pragma unroll
    for (int v = 0; v < NF; ++v) fav[v] = sum_value(s[v], (double*)nullptr);
    if (big || low < 0) {
      double st[2], av[2], ph[3];
      const PairGeom H = G;
      if (direct_values(P, H, st, av, ph)) atomicOr(A.flags, kFlagGeometry);
#pragma unroll
      for (int v = 0; v < NF; ++v)
        if (v < P.n_f) {
          fst[v] = st[v];
          fav[v] = av[v];
        }
    }
    double ci[4] = {0.0, 0.0, 0.0, 0.0}, cj[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
    for (int l = 0; l < S; ++l) {
      const double xi = __ldg(&A.x[l * A.n + pr.i]), xj = __ldg(&A.x[l * A.n + pr.j]);
#pragma unroll
      for (int k = 0; k < S; ++k) {
        const int fo = TB::f(P, k, l);
#pragma unroll
        for (int v = 0; v < NF; ++v)
          if (fo == v) {
            ci[k] += xj * fst[v];
            ci[2 + k] += xj * fav[v];
            cj[k] += xi * fst[v];
            cj[2 + k] += xi * fav[v];
          }
      }
    }
    if constexpr (S == 1 || TAB == 1) {  // one density for every species
      double2* d2 = reinterpret_cast<double2*>(dens);
      d2[pr.tp] = make_double2(ci[0], ci[2]);
      d2[pr.tr] = make_double2(cj[0], cj[2]);
    } else {
      dens[pr.tp] = Dbl4{ci[0], ci[1], ci[2], ci[3]};
      dens[pr.tr] = Dbl4{cj[0], cj[1], cj[2], cj[3]};
    }
  }
}

// ---------------------------------------------------------------- relaxation forces, FP64
// The weights of a pair's terms: C_u = (hi 2^31 + lo) 2^(e - 1082) with |hi| <=
// 2^29, 0 <= lo < 2^31 (all 53 bits), and as float pairs.  The constant terms
// of the rows are multiplied by them in integers on one grid per pair: a
// product of 60-bit halves is three 32-bit multiplications and a few additions,
// some 11 issue slots where an FP64 instruction holds a 2-lane pipe for 64.
// The grid leaves 55 bits (one or two terms: 56) below the largest term at the
// pair's nearest node, where the terms, which decrease, are largest, and eight
// (seven) above, for the sum of 12 nodes: a product that is more than four
// times larger somewhere sends the pair to the direct evaluation.
template <int NT>
struct FixedWeights {
  static constexpr int kHead = NT <= 2 ? 4 : 5;  // shift of the largest term
  int hi[NT], lo[NT], k[NT];
  int terms;  // that are not zero
  ff f[NT];
};
// The integers' unit is 2^(the result); row: the row of the nearest node.  A
// weight below 2^-74 has no float pair (ff_bits gives zero): the linear and
// higher terms of its rows would be lost, at most 2^-6 of the term, so unless
// the pair's largest term is over 2^50 times it the pair is evaluated directly.
template <int NT>
__device__ __forceinline__ int fixed_weights(const double* C, const uint4* row, FixedWeights<NT>& F, int& big) {
  int top = 0, faint = -1000;  // largest exponents of all terms and of those without a float pair
  F.terms = 0;
#pragma unroll
  for (int u = 0; u < NT; ++u) {
    const int h = __double2hiint(C[u]), e = (h >> 20) & 0x7ff;
    big |= e == 0x7ff;
    const long long m = ((long long)((h & 0xfffff) | 0x100000) << 32) | (unsigned)__double2loint(C[u]);
    const long long v = e == 0 ? 0ll : (h < 0 ? -m : m) << 7;
    F.hi[u] = (int)(v >> 31);
    F.lo[u] = (int)((unsigned)v & 0x7fffffffu);
    F.k[u] = e;
    F.f[u] = ff_bits(C[u]);
    // the constant term, or next to the cutoff, where it vanishes, 2^5 times
    // the linear and quadratic terms at |tau| = 1/2 (elsewhere below 2^-6 of it)
    const uint4 a = row[u * kTabWords64];
    const int e1 = (int)((a.z >> 23) & 0xffu), e2 = (int)((row[u * kTabWords64 + 1].x >> 23) & 0xffu);
    const int e8 = max((int)(a.x & 0xffu), max(e1 ? e1 + 5 : 0, e2 ? e2 + 4 : 0));
    if (e != 0 && e8 != 0) {
      top = max(top, e + e8);
      F.terms += 1;
      if (e <= kNoFloatPair) faint = max(faint, e + e8);
    }
  }
  big |= faint > top - 50;
#pragma unroll
  for (int u = 0; u < NT; ++u) F.k[u] = top == 0 ? 1000 : top + F.kHead - F.k[u];  // top 0: every node beyond the cutoff
  // hi m_hi is a product shifted by 62: exponents e - 1082, e8 - kTabExpBias
  const int unit = top == 0 ? 0 : top + F.kHead - 1082 - kTabExpBias + 62;
  // 2^(-24 - unit) has to be a float
  big |= unit > 90 || unit < -140;
  return unit;
}

// dV/dr / r of the pair's weighted terms at one node, in units of the pair's
// grid: the constant terms as above, the rest (below 2^-6 of them) as a float
// pair, added in two pieces of 24 bits.  sc: 2^-24 units.
template <int NT>
__device__ __forceinline__ long long force_node(const RadialTab& Tb, const uint4* sm, long long w,
                                                const FixedWeights<NT>& F, float sc, int& low) {
  float th, tl;
  const uint4* row = tab_row<false, false>(Tb, sm, w, th, tl, low);
  long long h = 0;
  ff p{0.f, 0.f};
#pragma unroll
  for (int u = 0; u < NT; ++u) {
    const uint4 a = row[u * kTabWords64];
    const ff q = tab_poly64(__uint_as_float(a.z), __uint_as_float(a.w), row[u * kTabWords64 + 1],
                            row[u * kTabWords64 + 2], th, tl);
    const int mh = (int)a.y, ml = (int)(a.x & 0x7fffff00u), sh = F.k[u] - (int)(a.x & 0xffu);
    const long long cross = (long long)F.hi[u] * ml + (long long)F.lo[u] * mh;
    low |= sh - (F.kHead - 2);  // negative: over four times the expected largest term
    h += shift_right((long long)F.hi[u] * mh + (cross >> 31), sh);
    ff m = two_prod(F.f[u].hi, q.hi);
    m.lo = fmaf(F.f[u].hi, q.lo, fmaf(F.f[u].lo, q.hi, m.lo));
    tab_acc(p, m);
  }
  const float x = p.hi * sc;
  const int i1 = __float2int_rn(x);
  low |= (1 << 30) - abs(i1);
  const int i2 = __float2int_rn(fmaf(p.lo, sc, x - (float)i1) * 16777216.0f);
  return h + (long long)i1 * 16777216ll + i2;
}

// Marks (in a thread's own record) a pair left for the direct evaluation, which
// runs after the table loop: a call inside it costs registers in every pair.
constexpr long long kTabLater = 0x7ff8a5a5c3c31e1ell;

// weights of the terms: nodes (C) and the static point (cfs)
template <int S, int NP, int TAB>
__device__ __forceinline__ void force_weights(const DevPot& P, const PassArgs& A, const PairRef& pr, double* C,
                                              double* cfs) {
  using TB = Tables<TAB>;
  constexpr int NF = S, NT = NF + NP;
  const int64_t n = A.n;
#pragma unroll
  for (int u = 0; u < NT; ++u) C[u] = 0.0;
#pragma unroll
  for (int v = 0; v < NF; ++v) cfs[v] = 0.0;
  double xi[S], xj[S], bi[S], bj[S], ai[S], aj[S];
#pragma unroll
  for (int k = 0; k < S; ++k) {
    xi[k] = __ldg(&A.x[k * n + pr.i]), xj[k] = __ldg(&A.x[k * n + pr.j]);
    ai[k] = __ldg(&A.a[k * n + pr.i]), aj[k] = __ldg(&A.a[k * n + pr.j]);
    bi[k] = __ldg(&A.b[k * n + pr.i]), bj[k] = __ldg(&A.b[k * n + pr.j]);
  }
#pragma unroll
  for (int k = 0; k < S; ++k)
#pragma unroll
    for (int l = 0; l < S; ++l) {
      const int po = TB::phi(P, k, l);
#pragma unroll
      for (int u = 0; u < NP; ++u)
        if (po == u) C[NF + u] += xi[k] * xj[l];
    }
  if constexpr (TAB == 1) {
    // the density term is that of the neighbour's species
    const double sbi = bi[0] + bi[1], sbj = bj[0] + bj[1], sai = ai[0] + ai[1], saj = aj[0] + aj[1];
#pragma unroll
    for (int v = 0; v < NF; ++v) {
      C[v] = sbi * xj[v] + sbj * xi[v];
      cfs[v] = sai * xj[v] + saj * xi[v];
    }
  } else {
#pragma unroll
    for (int k = 0; k < S; ++k)
#pragma unroll
      for (int l = 0; l < S; ++l) {
        const int fo = TB::f(P, k, l);
#pragma unroll
        for (int v = 0; v < NF; ++v)
          if (fo == v) {
            C[v] += bi[k] * xj[l] + bj[k] * xi[l];
            cfs[v] += ai[k] * xj[l] + aj[k] * xi[l];
          }
      }
  }
}

// both entries' records from T, U, V and Gs
__device__ __forceinline__ void store_force(const PairGeom& G, const double* out, const PairRef& pr,
                                            Dbl4* __restrict__ frc) {
  const double inv12 = 1.0 / 12.0;
  const double Tt = out[0] * inv12 + out[6];
  const double fx = -(G.d[0] * Tt + out[1] * inv12), fy = -(G.d[1] * Tt + out[2] * inv12),
               fz = -(G.d[2] * Tt + out[3] * inv12);
  frc[pr.tp] = Dbl4{fx, fy, fz, out[4] * inv12};
  frc[pr.tr] = Dbl4{-fx, -fy, -fz, out[5] * inv12};
}

template <int S, int NP, int TAB>
__global__ void __launch_bounds__(kTabThreads, 1) k_rforce_tab(
    const __grid_constant__ DevPot P, const __grid_constant__ DevGrid g0, const __grid_constant__ PassArgs A,
    const __grid_constant__ RadialTab Tb, const int4* __restrict__ pair_rec, int64_t npair, Dbl4* __restrict__ frc) {
  using TB = Tables<TAB>;
  constexpr int NF = S, NT = NF + NP;
  extern __shared__ uint4 sm[];
  tab_stage(Tb, sm);
  pdl_wait();
  pdl_trigger();
  __syncthreads();
  if (A.ctrl != nullptr && A.ctrl->halted) return;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  bool later = false;
  for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < npair; p += stride) {
    PairRef pr;
    if (!load_pair(A, pair_rec, p, pr)) continue;
    PairGeom G;
    pair_geometry(g0, A, pr.i, pr.j, G);
    PairNodes N;
    int big = pair_nodes(G, N);
    int low = 0;
    double C[NT], cfs[NF];
    force_weights<S, NP, TAB>(P, A, pr, C, cfs);
    double out[7];  // T, U[3], V[2], Gs
    float th, tl;
    {
      FixedWeights<NF> F;
      const int unit = fixed_weights<NF>(cfs, tab_row<false, false>(Tb, sm, N.w0, th, tl, low), F, big);
      const long long h = force_node<NF>(Tb, sm, N.w0, F, exp2f_bits(-24 - unit), low);
      out[6] = fixed_double(h != 0 ? h + (F.terms >> 1) : 0, unit);
    }
    const long long near = nearest_node(N);
    FixedWeights<NT> F;
    const int unit = fixed_weights<NT>(C, tab_row<false, false>(Tb, sm, near, th, tl, low), F, big);
    const float sc = exp2f_bits(-24 - unit);
    long long T = 0;
    double U[3] = {0.0, 0.0, 0.0}, V0 = 0.0, ad[3] = {fabs(G.d[0]), fabs(G.d[1]), fabs(G.d[2])};
    double s = G.s_i;
#pragma unroll 1
    for (int site = 0; site < 2; ++site) {
      long long E = 0;
      double V = 0.0;
#pragma unroll 1
      for (int a = 0; a < 3; ++a) {
        const long long h1 = force_node<NT>(Tb, sm, N.base[0] + N.tw[0][0], F, sc, low);
        const long long h2 = force_node<NT>(Tb, sm, N.base[0] - N.tw[0][0], F, sc, low);
        E += h1 + h2 + ((h1 | h2) != 0 ? F.terms : 0);  // the shifts round down, half a unit each
        const double D = fixed_double(h1 - h2, unit), Ua = fma(s, D, U[0]), da = ad[0];
        V = fma(da, D, V);
        // the next axis (registers rotate: one copy of the node code)
        const long long t = N.tw[0][0];
        N.tw[0][0] = N.tw[0][1];
        N.tw[0][1] = N.tw[0][2];
        N.tw[0][2] = t;
        U[0] = U[1];
        U[1] = U[2];
        U[2] = Ua;
        ad[0] = ad[1];
        ad[1] = ad[2];
        ad[2] = da;
      }
      T += E;
      V = kSqrt6 * fma(s, fixed_double(E, unit), V);
      out[4] = V0;
      out[5] = V0 = V;
      s = G.s_j;
      N.base[0] = N.base[1];
#pragma unroll
      for (int a = 0; a < 3; ++a) N.tw[0][a] = N.tw[1][a];
    }
    out[0] = fixed_double(T, unit);
#pragma unroll
    for (int a = 0; a < 3; ++a) out[1 + a] = __double2hiint(G.d[a]) < 0 ? -U[a] : U[a];
    store_force(G, out, pr, frc);
    if (big || low < 0) {
      frc[pr.tp].x = __longlong_as_double(kTabLater);
      later = true;
    }
  }
  if (!later) return;
  for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < npair; p += stride) {
    PairRef pr;
    if (!load_pair(A, pair_rec, p, pr) || __double_as_longlong(frc[pr.tp].x) != kTabLater) continue;
    PairGeom G;
    pair_geometry(g0, A, pr.i, pr.j, G);
    double C[NT], cfs[NF], ca[2] = {0.0, 0.0}, cs[2] = {0.0, 0.0}, cp[3] = {0.0, 0.0, 0.0}, out[7];
    force_weights<S, NP, TAB>(P, A, pr, C, cfs);
#pragma unroll
    for (int v = 0; v < NF; ++v) {
      ca[v] = C[v];
      cs[v] = cfs[v];
    }
#pragma unroll
    for (int u = 0; u < NP; ++u) cp[u] = C[NF + u];
    direct_forces(P, G, ca, cs, cp, out);
    store_force(G, out, pr, frc);
  }
}

// one block per SM; few pairs: enough smaller blocks to use every SM
template <typename... KArgs, typename... Args>
cudaError_t launch_table_kernel(void (*kernel)(KArgs...), const RadialTab& Tb, int64_t npair, cudaStream_t s,
                                Args... args) {
  const size_t shm = (size_t)Tb.nrow * Tb.stride * 16;
  cudaError_t e = cudaFuncSetAttribute((const void*)kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kTabMaxBytes);
  if (e != cudaSuccess) return e;
  int dev = 0, sms = 0;
  e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  int threads = kTabThreads;
  while (threads > 128 && (npair + threads - 1) / threads < sms) threads /= 2;
  const int64_t blocks = std::min<int64_t>((npair + threads - 1) / threads, sms);
  return launch_pdl(kernel, dim3((unsigned)std::max<int64_t>(blocks, 1)), dim3(threads), shm, s, args...);
}

}  // namespace

cudaError_t launch_geo_tab(int precision, const DevPot& P, const DevGrid& g, const PassArgs& A, const RadialTab& Tb,
                           const int4* pair_rec, int64_t npair, void* buf, int64_t cap, cudaStream_t s) {
  if (npair == 0) return cudaSuccess;
  const GeoLayout L = geo_layout(P, cap);
  auto run = [&](auto kernel, auto* out) {
    return launch_table_kernel(kernel, Tb, npair, s, P, g, A, Tb, pair_rec, npair, out, L);
  };
  if (precision == 0) {
    if (P.S == 1) return run(k_geo_tab<1, 1, double>, (double*)buf);
    if (Tb.np_slots == 2) return run(k_geo_tab<2, 2, double>, (double*)buf);
    return run(k_geo_tab<2, 3, double>, (double*)buf);
  }
  if (P.S == 1) return run(k_geo_tab<1, 1, ff>, (float2*)buf);
  if (Tb.np_slots == 2) return run(k_geo_tab<2, 2, ff>, (float2*)buf);
  return run(k_geo_tab<2, 3, ff>, (float2*)buf);
}

cudaError_t launch_relax_tab(bool force, const DevPot& P, const DevGrid& g, const PassArgs& A, const RadialTab& Tb,
                             const int4* pair_rec, int64_t npair, void* out, cudaStream_t s) {
  if (A.n == 0 || npair == 0) return cudaSuccess;
  auto run = [&](auto kernel) {
    return launch_table_kernel(kernel, Tb, npair, s, P, g, A, Tb, pair_rec, npair, (Dbl4*)out);
  };
  if (!force) {
    if (P.S == 1) return run(k_rdensity_tab<1, 0>);
    return P.tab == 1 ? run(k_rdensity_tab<2, 1>) : run(k_rdensity_tab<2, 0>);
  }
  if (P.S == 1) return run(k_rforce_tab<1, 1, 0>);
  if (Tb.np_slots == 2) return run(k_rforce_tab<2, 2, 0>);
  return P.tab == 1 ? run(k_rforce_tab<2, 3, 1>) : run(k_rforce_tab<2, 3, 0>);
}

}  // namespace mxe
