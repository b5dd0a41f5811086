// gathers.cu -- per-site sums of the pair passes' records over each site's own
// row (rows in order), and the per-site arithmetic that follows them.
//
//  k_geo_density / k_geo_mu      geometry records of the accurate pass (eam.cu,
//                                pair_table.cu): densities and embedding terms,
//                                then chemical potentials and energies
//  k_relax_density / k_relax_force   records of the relaxation passes
//
// A team of NL lanes owns a site and strides over its row.  What bounded the
// kernels, besides the record stream, was the per-site arithmetic in FP64: with
// NL = 8 a warp ran a square root, two divisions or four logarithms for four
// sites at a time on the 2-lane FP64 pipe (79 % of it in the float-float
// density gather, 55 % in the chemical-potential gather).  The sums now go
// through shared memory to as many threads as the block has sites, so a warp
// finishes 32 sites; conversions between FP32 pairs and FP64 are done on bits.
//
// One density (ND = 1): with one species, or with a density that does not
// depend on the site's own species (tab 1), every species of a site has the
// same density: half the density records, one square root, and the neighbour's
// embedding coefficients enter only as their sums over species.
//
// Measured before -> after: accurate gathers (density, mu) at 256,000 sites
// float-float 239 -> 115 and 384 -> 216 us, 864,000 sites of one species 672 -> 233
// and 790 -> 379 us, 19,652 sites FP64 57 -> 21 and 116 -> 45 us; relaxation
// densities at 256,000 sites 54 -> 38 us, 19,652 sites FP64 42 -> 16 us.
#include <cuda_runtime.h>

#include <type_traits>

#include "accum.cuh"
#include "pair_common.cuh"

namespace mxe {
namespace {

// ---------------------------------------------------------------- values
// two consecutive values of a record or site record (16 bytes)
__device__ __forceinline__ void load2(const ff* p, int64_t k, ff& a, ff& b) {
  const float4 v = __ldg(reinterpret_cast<const float4*>(p) + k);
  a = ff(v.x, v.y);
  b = ff(v.z, v.w);
}
__device__ __forceinline__ void load2(const double* p, int64_t k, double& a, double& b) {
  const double2 v = __ldg(reinterpret_cast<const double2*>(p) + k);
  a = v.x;
  b = v.y;
}
__device__ __forceinline__ ff load1(const ff* p) {
  const float2 v = __ldg(reinterpret_cast<const float2*>(p));
  return ff(v.x, v.y);
}
__device__ __forceinline__ double load1(const double* p) { return __ldg(p); }
__device__ __forceinline__ void store2(ff* p, int64_t k, double a, double b) {
  const ff x = ff_from_double(a), y = ff_from_double(b);
  reinterpret_cast<float4*>(p)[k] = make_float4(x.hi, x.lo, y.hi, y.lo);
}
__device__ __forceinline__ void store2(double* p, int64_t k, double a, double b) {
  reinterpret_cast<double2*>(p)[k] = make_double2(a, b);
}

template <typename Acc>
__device__ __forceinline__ void madd(Acc& s, ff a, ff b, ff c, ff d) { s.add(a * b + c * d); }  // s += a b + c d
template <typename Acc>
__device__ __forceinline__ void madd(Acc& s, ff a, ff b) { s.add(a * b); }
__device__ __forceinline__ void madd(AccD& s, double a, double b, double c, double d) { s.v = fma(a, b, fma(c, d, s.v)); }
__device__ __forceinline__ void madd(AccD& s, double a, double b) { s.v = fma(a, b, s.v); }

// sqrt(x) and 1 / sqrt(x), each with one Newton correction of CUDA's rsqrt (both
// to about half an ulp; no division)
__device__ __forceinline__ double inv_sqrt(double x, double& sq) {
  const double y = rsqrt(x);
  sq = x * y;
  sq = fma(0.5 * y, fma(-sq, sq, x), sq);
  return fma(y, fma(-sq, y, 1.0), y);
}

template <int S, int TAB>
constexpr int one_density() { return S == 1 || TAB == 1 ? 1 : S; }

// ---------------------------------------------------------------- densities
// Site record srec (site_record_len values): x of both species, then per
// density a and b / 12, FP64: 12 a and b (ND = 1: their sums over the species).
// The FP32 modes' pack kernel has written x, this kernel the rest.
template <int S, int TAB, int NL, typename R, typename Acc>
__global__ void __launch_bounds__(256) k_geo_density(const __grid_constant__ DevPot P,
                                                     const __grid_constant__ PassArgs A, const R* __restrict__ buf,
                                                     GeoLayout L) {
  constexpr int ND = one_density<S, TAB>(), NR = 2 + 2 * ND;
  constexpr bool kFP64 = std::is_same<R, double>::value;
  if (A.ctrl != nullptr && A.ctrl->halted) return;
  const int nsite = blockDim.x / NL;
  const int64_t i0 = (int64_t)blockIdx.x * nsite, n = A.n;
  const int64_t i = i0 + threadIdx.x / NL;
  const int lane = threadIdx.x % NL;
  Acc rb[ND], ra[ND];
#pragma unroll
  for (int k = 0; k < ND; ++k) {
    rb[k].zero();
    ra[k].zero();
  }
  R* srec = reinterpret_cast<R*>(A.srec);
  if (i < n) {
    const int beg = A.nb_off[i], end = A.nb_off[i + 1];
#pragma unroll 4
    for (int t = beg + lane; t < end; t += NL) {
      const int64_t j = __ldg(&A.nb_ent[t]) & kIdxMask;
      R x[2];
      if constexpr (kFP64) {
        x[0] = __ldg(&A.x[j]);
        if (S > 1) x[1] = __ldg(&A.x[n + j]);
      } else {
        load2(srec, j * (NR / 2), x[0], x[1]);
      }
      if constexpr (S == 1) {
        if (P.n_f == 1) {
          R st, av;
          load2(buf, t, st, av);
          madd(rb[0], x[0], st);
          madd(ra[0], x[0], av);
        }
      } else if constexpr (TAB == 1) {
        R s0, s1, v0, v1;
        load2(buf, 2 * (int64_t)t, s0, s1);
        load2(buf, 2 * (int64_t)t + 1, v0, v1);
        madd(rb[0], x[0], s0, x[1], s1);
        madd(ra[0], x[0], v0, x[1], v1);
      } else {
        const R* rec = buf + (int64_t)t * L.ca;
#pragma unroll
        for (int k = 0; k < S; ++k)
#pragma unroll
          for (int l = 0; l < S; ++l) {
            const int v = P.f_of[k][l];
            if (v < 0) continue;
            madd(rb[k], x[l], load1(rec + v));
            madd(ra[k], x[l], load1(rec + P.n_f + v));
          }
      }
    }
  }
  __shared__ Acc s_acc[64 * 2 * ND];
#pragma unroll
  for (int k = 0; k < ND; ++k) {
    rb[k].team_reduce(NL);
    ra[k].team_reduce(NL);
    if (lane == 0) {
      s_acc[(threadIdx.x / NL) * 2 * ND + 2 * k] = rb[k];
      s_acc[(threadIdx.x / NL) * 2 * ND + 2 * k + 1] = ra[k];
    }
  }
  __syncthreads();
  const int64_t m = i0 + threadIdx.x;
  if ((int)threadIdx.x >= nsite || m >= n) return;
  double a[S], b[S];
#pragma unroll
  for (int d = 0; d < ND; ++d) {
    const double rbar = s_acc[threadIdx.x * 2 * ND + 2 * d].get();
    const double dr = s_acc[threadIdx.x * 2 * ND + 2 * d + 1].get() * (1.0 / 12.0) - rbar;
    const bool ok = rbar > kRhoMin;
    double sq;
    const double y = ok ? inv_sqrt(rbar, sq) : (sq = 0.0);
#pragma unroll
    for (int k = d; k < (ND == 1 ? S : d + 1); ++k) {
      const double E = P.E[k], x = A.x[k * n + m];
      double e = 0.0;
      a[k] = b[k] = 0.0;
      if (E == 0.0) {
        // no embedding energy for this element
      } else if (ok) {
        const double F1 = -0.5 * E * y, F2 = -0.5 * F1 * (y * y);
        e = fma(F1, dr, -E * sq);
        a[k] = x * F2 * dr;
        b[k] = x * F1;
      } else {
        atomicOr(A.flags, kFlagGeometry);
      }
      A.e[k * n + m] = e;
    }
  }
  if constexpr (kFP64) {
#pragma unroll
    for (int k = 0; k < S; ++k) {
      A.a[k * n + m] = a[k];
      A.b[k * n + m] = b[k];
    }
    store2(srec, m * (NR / 2), A.x[m], S > 1 ? A.x[(S > 1 ? 1 : 0) * n + m] : 0.0);
  } else {
    A.ab32[2 * m] = make_float4((float)a[0], (float)b[0], S > 1 ? (float)a[S - 1] : 0.f, S > 1 ? (float)b[S - 1] : 0.f);
  }
  const double ka = kFP64 ? 12.0 : 1.0, kb = kFP64 ? 1.0 : 1.0 / 12.0;
  if constexpr (ND == 1) {
    store2(srec, m * 2 + 1, (S > 1 ? a[0] + a[S - 1] : a[0]) * ka, (S > 1 ? b[0] + b[S - 1] : b[0]) * kb);
  } else {
#pragma unroll
    for (int k = 0; k < S; ++k) store2(srec, m * 3 + 1 + k, a[k] * ka, b[k] * kb);
  }
}

// ---------------------------------------------------------------- chemical potentials and energies
// Float pairs: the pair part (x 12; also the site's pair energy) and the
// embedding part are summed apart.  FP64: they are added entry by entry, x 12,
// since they cancel to a tenth (the sums apart cost 1.2 times the error of mu),
// with one division per site; the pair energy has its own sum.
template <int S, int TAB, int NL, typename R, typename Acc>
__global__ void __launch_bounds__(256) k_geo_mu(const __grid_constant__ DevPot P, const __grid_constant__ PassArgs A,
                                                const R* __restrict__ buf, GeoLayout L) {
  constexpr int ND = one_density<S, TAB>(), NR = 2 + 2 * ND;
  constexpr bool kFP64 = std::is_same<R, double>::value;
  if (A.ctrl != nullptr && A.ctrl->halted) return;
  const int nsite = blockDim.x / NL;
  const int64_t i0 = (int64_t)blockIdx.x * nsite, n = A.n;
  const int64_t i = i0 + threadIdx.x / NL;
  const int lane = threadIdx.x % NL;
  Acc pr[S], em[S];  // FP64: pr[0] the pair energy, em[k] the chemical potentials, both x 12
  R xi[S];
#pragma unroll
  for (int k = 0; k < S; ++k) {
    pr[k].zero();
    em[k].zero();
    if constexpr (kFP64) xi[k] = i < n ? __ldg(&A.x[k * n + i]) : 0.0;
  }
  const R* srec = reinterpret_cast<const R*>(A.srec);
  const R* bufp = buf + L.b_off;
  // the pair part m of species k
  auto pair_part = [&](int k, R m) {
    if constexpr (kFP64) {
      em[k].v += m;
      pr[0].v = fma(xi[k], m, pr[0].v);
    } else {
      pr[k].add(m);
    }
  };
  if (i < n) {
    const int beg = A.nb_off[i], end = A.nb_off[i + 1];
#pragma unroll 2
    for (int t = beg + lane; t < end; t += NL) {
      const int64_t j = __ldg(&A.nb_ent[t]) & kIdxMask;
      R x[2];
      load2(srec, j * (NR / 2), x[0], x[1]);
      if constexpr (ND == 1) {
        R sa, sb;
        load2(srec, j * (NR / 2) + 1, sa, sb);
        if constexpr (S == 1) {
          if (P.n_phi == 1) pair_part(0, x[0] * load1(bufp + t));
          if (P.n_f == 1) {
            R st, av;
            load2(buf, t, st, av);
            madd(em[0], sa, st, sb, av);
          }
        } else {
          R s0, s1, v0, v1, p0, p1, p2, pad;
          load2(buf, 2 * (int64_t)t, s0, s1);
          load2(buf, 2 * (int64_t)t + 1, v0, v1);
          load2(bufp, 2 * (int64_t)t, p0, p1);
          load2(bufp, 2 * (int64_t)t + 1, p2, pad);
          pair_part(0, x[0] * p0 + x[1] * p1);
          pair_part(S - 1, x[0] * p1 + x[1] * p2);
          madd(em[0], sa, s0, sb, v0);
          madd(em[S - 1], sa, s1, sb, v1);
        }
      } else {
        const R *rec = buf + (int64_t)t * L.ca, *recp = bufp + (int64_t)t * L.cb;
        R a[S], b[S];
#pragma unroll
        for (int l = 0; l < S; ++l) load2(srec, j * (NR / 2) + 1 + l, a[l], b[l]);
#pragma unroll
        for (int k = 0; k < S; ++k)
#pragma unroll
          for (int l = 0; l < S; ++l) {
            const int u = P.phi_of[k][l];
            if (u >= 0) pair_part(k, x[l] * load1(recp + u));
            // density at j of species l from this site holding species k: f_lk
            const int v = P.f_of[l][k];
            if (v >= 0) madd(em[k], a[l], load1(rec + v), b[l], load1(rec + P.n_f + v));
          }
      }
    }
  }
  __shared__ Acc s_acc[64 * 2 * S];
  __shared__ double s_log[64 * (S + 2)];
#pragma unroll
  for (int k = 0; k < S; ++k) {
    pr[k].team_reduce(NL);
    em[k].team_reduce(NL);
    if (lane == 0) {
      s_acc[(threadIdx.x / NL) * 2 * S + 2 * k] = pr[k];
      s_acc[(threadIdx.x / NL) * 2 * S + 2 * k + 1] = em[k];
    }
  }
  // one logarithm per thread: ln x_k, ln x_v (with the floor of the chemical
  // potential), ln sigma (energies only)
  const bool logs = A.mu != nullptr || A.site_E != nullptr;
  if (logs) {
    for (int c = threadIdx.x; c < nsite * (S + 2); c += blockDim.x) {
      const int w = c / nsite;
      const int64_t m = i0 + c % nsite;
      double arg = 1.0;
      if (m < n) {
        if (w < S) {
          arg = fmax(A.x[w * n + m], kLogFloor);
        } else if (w == S) {
          arg = 1.0;
#pragma unroll
          for (int k = 0; k < S; ++k) arg -= A.x[k * n + m];
          arg = fmax(arg, kLogFloor);
        } else if (A.site_E) {
          arg = A.sigma[m];
        }
      }
      s_log[c] = log(arg);
    }
  }
  __syncthreads();
  const int site = threadIdx.x;
  const int64_t m = i0 + site;
  if (site >= nsite || m >= n) return;
  bool finite = true;
  double ep = 0.0, emb = 0.0, xs[S], xv = 1.0;
  const double kT = logs ? kKB * A.T[m] : 0.0;
#pragma unroll
  for (int k = 0; k < S; ++k) {
    const double pk = s_acc[site * 2 * S + 2 * k].get(), ek = s_acc[site * 2 * S + 2 * k + 1].get();
    const double e = A.e[k * n + m];
    xs[k] = A.x[k * n + m];
    xv -= xs[k];
    const double mu = kFP64 ? ek / 12.0 + e : fma(pk, 1.0 / 12.0, ek) + e;
    finite = finite && isfinite(mu);
    if (A.mu_ex) A.mu_ex[k * n + m] = mu;
    if (A.mu) A.mu[k * n + m] = mu + kT * (s_log[k * nsite + site] - s_log[S * nsite + site]);
    if (kFP64) ep = k == 0 ? pk : ep;
    else ep = fma(xs[k], pk, ep);
    emb = fma(xs[k], e, emb);
  }
  if (A.site_E) {
    // x ln x reuses the logarithms (its own only for 0 < x below the floor)
    double mix = 0.0;
#pragma unroll
    for (int k = 0; k <= S; ++k) {
      const double x = k < S ? xs[k < S ? k : 0] : xv;
      if (x > 0.0) mix += x * (x >= kLogFloor ? s_log[k * nsite + site] : log(x));
    }
    const double EV = fma(0.5 / 12.0, ep, emb);
    const double Fv = -3.0 * kT * s_log[(S + 1) * nsite + site];
    const double Fm = kT * mix;
    A.site_E[m] = EV;
    A.site_E[n + m] = Fv;
    A.site_E[2 * n + m] = Fm;
    finite = finite && isfinite(EV) && isfinite(Fv) && isfinite(Fm);
  }
  if (!finite) atomicOr(A.flags, kFlagNonfinite);
}

// ---------------------------------------------------------------- relaxation
template <int PREC>
struct Relax;  // record value and per-site sum
template <>
struct Relax<0> {
  using V = double;
  using Acc = AccD;
};
template <>
struct Relax<1> {
  using V = float;
  using Acc = AccT;
};
template <>
struct Relax<2> {
  using V = float;
  using Acc = AccFF;
};

template <int C>
__device__ __forceinline__ void load_rec(const float* rec, int64_t t, float* v) {
  if constexpr (C == 2) {
    const float2 r = __ldg(reinterpret_cast<const float2*>(rec) + t);
    v[0] = r.x;
    v[1] = r.y;
  } else {
    const float4 r = __ldg(reinterpret_cast<const float4*>(rec) + t);
    v[0] = r.x;
    v[1] = r.y;
    v[2] = r.z;
    v[3] = r.w;
  }
}
template <int C>
__device__ __forceinline__ void load_rec(const double* rec, int64_t t, double* v) {
#pragma unroll
  for (int c = 0; c < C / 2; ++c) {
    const double2 r = __ldg(reinterpret_cast<const double2*>(rec) + t * (C / 2) + c);
    v[2 * c] = r.x;
    v[2 * c + 1] = r.y;
  }
}

struct EmbedE {
  double d[2];
  float f[2];
};

// Record of an entry: rho_bar then 12 <rho> of every distinct density.
template <int PREC, int S, int ND, int NL>
__global__ void __launch_bounds__(256) k_relax_density(EmbedE E, const __grid_constant__ PassArgs A,
                                                       const typename Relax<PREC>::V* __restrict__ dens) {
  using V = typename Relax<PREC>::V;
  using Acc = typename Relax<PREC>::Acc;
  pdl_wait();
  pdl_trigger();
  if (A.ctrl != nullptr && A.ctrl->halted) return;
  const int nsite = blockDim.x / NL;
  const int64_t i0 = (int64_t)blockIdx.x * nsite, n = A.n;
  const int64_t i = i0 + threadIdx.x / NL;
  const int lane = threadIdx.x % NL;
  Acc s[2 * ND];
#pragma unroll
  for (int c = 0; c < 2 * ND; ++c) s[c].zero();
  if (i < n) {
    const int beg = A.nb_off[i], end = A.nb_off[i + 1];
#pragma unroll 4
    for (int t = beg + lane; t < end; t += NL) {
      V r[2 * ND];
      load_rec<2 * ND>(dens, t, r);
#pragma unroll
      for (int c = 0; c < 2 * ND; ++c) s[c].add(r[c]);
    }
  }
#pragma unroll
  for (int c = 0; c < 2 * ND; ++c) s[c].team_reduce(NL);
  if constexpr (PREC == 0) {
    // FP64: one thread per site
    __shared__ double s_acc[64 * 2 * ND];
    if (lane == 0) {
#pragma unroll
      for (int c = 0; c < 2 * ND; ++c) s_acc[(threadIdx.x / NL) * 2 * ND + c] = s[c].get();
    }
    __syncthreads();
    const int64_t m = i0 + threadIdx.x;
    if ((int)threadIdx.x >= nsite || m >= n) return;
#pragma unroll
    for (int d = 0; d < ND; ++d) {
      const double rbar = s_acc[threadIdx.x * 2 * ND + d];
      const double dr = s_acc[threadIdx.x * 2 * ND + ND + d] * (1.0 / 12.0) - rbar;
      const bool ok = rbar > kRhoMin;
      double sq;
      const double y = ok ? inv_sqrt(rbar, sq) : 0.0;
#pragma unroll
      for (int k = d; k < (ND == 1 ? S : d + 1); ++k) {
        const double x = A.x[k * n + m];
        double a = 0.0, b = 0.0;
        if (E.d[k] == 0.0) {
          // no embedding energy for this element
        } else if (ok) {
          const double F1 = -0.5 * E.d[k] * y, F2 = -0.5 * F1 * (y * y);
          a = x * F2 * dr;
          b = x * F1;
        } else {
          atomicOr(A.flags, kFlagGeometry);
        }
        A.a[k * n + m] = a;
        A.b[k * n + m] = b;
      }
    }
  } else {
    if (i >= n || lane != 0) return;
    float ab[4] = {0.f, 0.f, 0.f, 0.f};
    const float4 X = __ldg(&A.x32[i]);
    const float xs[2] = {X.x, X.y};
    int flag = 0;
#pragma unroll
    for (int d = 0; d < ND; ++d) {
      const float2 b2 = s[d].get_pair(), a2 = s[ND + d].get_pair();
      const float rf = b2.x + b2.y;
      const float df = fmaf(a2.x, 1.0f / 12.0f, -b2.x) + fmaf(a2.y, 1.0f / 12.0f, -b2.y);
      float isq;
      asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(isq) : "f"(rf));
#pragma unroll
      for (int k = d; k < (ND == 1 ? S : d + 1); ++k) {
        if (E.f[k] == 0.f) {
          // no embedding energy for this element
        } else if (rf > (float)kRhoMin) {
          const float dF = -0.5f * E.f[k] * isq;
          const float d2F = 0.25f * E.f[k] * isq * isq * isq;
          ab[2 * k] = xs[k] * d2F * df;
          ab[2 * k + 1] = xs[k] * dF;
        } else {
          flag |= kFlagGeometry;
        }
      }
    }
    A.ab32[2 * i] = make_float4(ab[0], ab[1], ab[2], ab[3]);
    if (flag) atomicOr(A.flags, flag);
  }
}

template <int PREC, int NL>
__global__ void __launch_bounds__(256) k_relax_force(const __grid_constant__ PassArgs A,
                                                     const typename Relax<PREC>::V* __restrict__ frc) {
  using V = typename Relax<PREC>::V;
  using Acc = typename Relax<PREC>::Acc;
  pdl_wait();
  pdl_trigger();
  if (A.ctrl != nullptr && A.ctrl->halted) return;
  const int64_t tid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, n = A.n;
  const int64_t i = tid / NL;
  const int lane = (int)(tid % NL);
  Acc g[4];
#pragma unroll
  for (int c = 0; c < 4; ++c) g[c].zero();
  if (i < n) {
    const int beg = A.nb_off[i], end = A.nb_off[i + 1];
#pragma unroll 4
    for (int t = beg + lane; t < end; t += NL) {
      V f[4];
      load_rec<4>(frc, t, f);
#pragma unroll
      for (int c = 0; c < 4; ++c) g[c].add(f[c]);
    }
  }
#pragma unroll
  for (int c = 0; c < 4; ++c) g[c].team_reduce(NL);
  // team lanes 0-2 the force components, lane 3 the width derivative with its
  // thermal term; after the butterfly every lane holds the whole sum
  static_assert(NL >= 4, "one team lane per output");
  if (i >= n || lane > 3) return;
  double v;
  if constexpr (PREC == 0) {
    v = lane == 0 ? g[0].get() : lane == 1 ? g[1].get() : lane == 2 ? g[2].get()
                  : g[3].get() - 3.0 * kKB * A.T[i] / A.sigma[i];
  } else {
    float2 h = g[0].get_pair();
    if (lane == 1) h = g[1].get_pair();
    else if (lane == 2) h = g[2].get_pair();
    else if (lane == 3) {
      // FP32 modes: the thermal term in FP32 (sigma as packed, T rounded)
      const float2 gp = g[3].get_pair();
      const float th = 3.0f * (float)kKB * (float)A.T[i] / __ldg(&A.pos32[i]).w;
      h = make_float2((gp.x - th) + gp.y, 0.f);
    }
    v = widen(h.x) + widen(h.y);
  }
  if (lane < 3) {
    if (A.gq) A.gq[lane * n + i] = v;
  } else if (A.gs) {
    A.gs[i] = v;
  }
  if (!isfinite(v)) atomicOr(A.flags, kFlagNonfinite);
}

// ---------------------------------------------------------------- dispatch
template <int S, int TAB, int NL>
cudaError_t geo_gather_p(int precision, bool mu, const DevPot& P, const PassArgs& A, const void* buf, GeoLayout L,
                         cudaStream_t s) {
  const int threads = A.tpb > 0 ? A.tpb : 256;
  const unsigned blocks = (unsigned)((A.n * NL + threads - 1) / threads);
  auto run = [&](auto dens, auto chem, auto* b) {
    if (mu) chem<<<blocks, threads, 0, s>>>(P, A, b, L);
    else dens<<<blocks, threads, 0, s>>>(P, A, b, L);
    return cudaGetLastError();
  };
  switch (precision) {
    case 0:
      return run(k_geo_density<S, TAB, NL, double, AccD>, k_geo_mu<S, TAB, NL, double, AccD>, (const double*)buf);
    case 1: return run(k_geo_density<S, TAB, NL, ff, AccT>, k_geo_mu<S, TAB, NL, ff, AccT>, (const ff*)buf);
    case 2: return run(k_geo_density<S, TAB, NL, ff, AccF2>, k_geo_mu<S, TAB, NL, ff, AccF2>, (const ff*)buf);
    default: return cudaErrorInvalidValue;
  }
}
template <int S, int TAB>
cudaError_t geo_gather_nl(int precision, bool mu, int nl, const DevPot& P, const PassArgs& A, const void* buf,
                          GeoLayout L, cudaStream_t s) {
  switch (nl) {
    case 4: return geo_gather_p<S, TAB, 4>(precision, mu, P, A, buf, L, s);
    case 8: return geo_gather_p<S, TAB, 8>(precision, mu, P, A, buf, L, s);
    case 16: return geo_gather_p<S, TAB, 16>(precision, mu, P, A, buf, L, s);
    default: return cudaErrorInvalidValue;
  }
}

template <int PREC, int S, int ND, int NL>
cudaError_t relax_gather_t(bool force, const DevPot& P, const PassArgs& A, const void* dens, const void* frc,
                           cudaStream_t s) {
  using V = typename Relax<PREC>::V;
  const int threads = A.tpb > 0 ? A.tpb : 256;
  const dim3 blocks((unsigned)((A.n * NL + threads - 1) / threads));
  if (force) return launch_pdl(k_relax_force<PREC, NL>, blocks, dim3(threads), 0, s, A, (const V*)frc);
  EmbedE E = {};
  for (int k = 0; k < S; ++k) {
    E.d[k] = P.E[k];
    E.f[k] = (float)P.E[k];
  }
  return launch_pdl(k_relax_density<PREC, S, ND, NL>, blocks, dim3(threads), 0, s, E, A, (const V*)dens);
}
template <int PREC, int S, int ND>
cudaError_t relax_gather_nl(bool force, int nl, const DevPot& P, const PassArgs& A, const void* dens, const void* frc,
                            cudaStream_t s) {
  switch (nl) {
    case 4: return relax_gather_t<PREC, S, ND, 4>(force, P, A, dens, frc, s);
    case 8: return relax_gather_t<PREC, S, ND, 8>(force, P, A, dens, frc, s);
    case 16: return relax_gather_t<PREC, S, ND, 16>(force, P, A, dens, frc, s);
    default: return cudaErrorInvalidValue;
  }
}
template <int PREC>
cudaError_t relax_gather_p(bool force, int nl, const DevPot& P, const PassArgs& A, const void* dens, const void* frc,
                           cudaStream_t s) {
  if (P.S == 1) return relax_gather_nl<PREC, 1, 1>(force, nl, P, A, dens, frc, s);
  if (P.tab == 1) return relax_gather_nl<PREC, 2, 1>(force, nl, P, A, dens, frc, s);
  return relax_gather_nl<PREC, 2, 2>(force, nl, P, A, dens, frc, s);
}

}  // namespace

int site_record_len(const DevPot& P) { return P.S == 1 || P.tab == 1 ? 4 : 6; }

cudaError_t launch_pair_gather(int precision, bool mu, int nl, const DevPot& P, const PassArgs& A, const void* buf,
                               int64_t cap, cudaStream_t s) {
  if (A.n == 0) return cudaSuccess;
  const GeoLayout L = geo_layout(P, cap);
  if (P.S == 1) return geo_gather_nl<1, 0>(precision, mu, nl, P, A, buf, L, s);
  if (P.tab == 1) return geo_gather_nl<2, 1>(precision, mu, nl, P, A, buf, L, s);
  return geo_gather_nl<2, 0>(precision, mu, nl, P, A, buf, L, s);
}

cudaError_t launch_relax_gather(int precision, bool force, int nl, const DevPot& P, const PassArgs& A,
                                const void* dens, const void* frc, cudaStream_t s) {
  if (A.n == 0) return cudaSuccess;
  if (!pair_kernels_supported(P)) return cudaErrorInvalidValue;
  switch (precision) {
    case 0: return relax_gather_p<0>(force, nl, P, A, dens, frc, s);
    case 1: return relax_gather_p<1>(force, nl, P, A, dens, frc, s);
    case 2: return relax_gather_p<2>(force, nl, P, A, dens, frc, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace mxe
