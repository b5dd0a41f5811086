// radial_table.cu -- fills the radial tables of a context (radial_table.cuh):
// one thread per interval and term forms the Taylor series of the term about
// the interval's centre, the constant terms in double-double arithmetic
// (error-free TwoSum and TwoProduct; about 100 bits).  One launch per context.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>

#include "radial_table.cuh"

namespace mxe {
namespace {

constexpr int kDeg = 9;  // series order (coefficients 0..9)

struct dd {
  double h, l;
};
__device__ __forceinline__ dd dd_two_sum(double a, double b) {
  const double s = __dadd_rn(a, b), bp = __dsub_rn(s, a);
  return dd{s, __dadd_rn(__dsub_rn(a, __dsub_rn(s, bp)), __dsub_rn(b, bp))};
}
__device__ __forceinline__ dd dd_fast(double a, double b) {
  const double s = __dadd_rn(a, b);
  return dd{s, __dsub_rn(b, __dsub_rn(s, a))};
}
__device__ __forceinline__ dd operator+(dd a, dd b) {
  const dd s = dd_two_sum(a.h, b.h), t = dd_two_sum(a.l, b.l);
  const dd u = dd_fast(s.h, __dadd_rn(s.l, t.h));
  return dd_fast(u.h, __dadd_rn(u.l, t.l));
}
__device__ __forceinline__ dd operator-(dd a) { return dd{-a.h, -a.l}; }
__device__ __forceinline__ dd operator-(dd a, dd b) { return a + (-b); }
__device__ __forceinline__ dd operator*(dd a, dd b) {
  const double p = __dmul_rn(a.h, b.h);
  const double e = __fma_rn(a.h, b.h, -p);
  return dd_fast(p, __fma_rn(a.h, b.l, __fma_rn(a.l, b.h, e)));
}
__device__ __forceinline__ dd dd_of(double v) { return dd{v, 0.0}; }
__device__ __forceinline__ dd operator*(double a, dd b) { return dd_of(a) * b; }
// 1/a: the double reciprocal and one Newton correction
__device__ __forceinline__ dd dd_recip(dd a) {
  const double y = 1.0 / a.h;
  const dd r = dd_of(1.0) - y * a;
  return dd_of(y) + y * r;
}
__device__ __forceinline__ dd dd_sqrt(double a) {
  const double y = sqrt(a);
  const double r = __fma_rn(-y, y, a);  // exact
  return dd_fast(y, r / (2.0 * y));
}
// exp by argument reduction, a Taylor series of (exp - 1) at x / 512 (Horner)
// and nine doublings e <- 2 e + e^2
__device__ dd dd_exp(dd x) {
  const dd ln2{0.6931471805599453, 2.3190468138462996e-17};
  const double n = rint(x.h / ln2.h);
  dd r = x - n * ln2;
  r = dd{r.h * (1.0 / 512.0), r.l * (1.0 / 512.0)};
  dd sum = dd_of(1.0);
#pragma unroll 1
  for (int k = 8; k >= 2; --k) sum = dd_of(1.0) + (r * sum) * dd_recip(dd_of((double)k));
  sum = r * sum;
#pragma unroll 1
  for (int k = 0; k < 9; ++k) sum = 2.0 * sum + sum * sum;
  sum = sum + dd_of(1.0);
  const double sc = exp2(n);
  return dd{sum.h * sc, sum.l * sc};
}

__device__ __forceinline__ void mul(const double* a, const double* b, double* o) {
#pragma unroll
  for (int n = 0; n <= kDeg; ++n) {
    double s = 0.0;
#pragma unroll
    for (int i = 0; i <= n; ++i) s = fma(a[i], b[n - i], s);
    o[n] = s;
  }
}

// Taylor coefficients of a term with its switch about w = wc in units of h.
// The first three carry the constant terms of the value and derivative tables:
// double-double (V0..V2); the others weigh at most 2^-7 of them: FP64.
__device__ void term_series(const RadialFn& F, double wc, double h, bool beyond_rs, double rs, double rc, dd& V0,
                            dd& V1, dd& V2, double* V) {
  const dd r0 = dd_sqrt(wc);
  const dd r1 = (0.5 * h) * dd_recip(r0);
  const dd r2 = (-0.25 * h) * (r1 * dd_recip(dd_of(wc)));
  // r = sqrt(wc + h tau), binomial series
  double r[kDeg + 1];
  r[0] = r0.h;
  const double q = h / wc;
#pragma unroll
  for (int n = 1; n <= kDeg; ++n) r[n] = r[n - 1] * q * ((1.5 - n) / n);
  // E = A exp(kappa - lambda r): n E_n = -lambda sum_i i r_i E_{n-i}
  const dd e0 = F.A * dd_exp(dd_of(F.kappa) - F.lambda * r0);
  const dd e1 = -(F.lambda * (r1 * e0));
  const dd e2 = -((0.5 * F.lambda) * (r1 * e1 + 2.0 * (r2 * e0)));
  double E[kDeg + 1];
  E[0] = e0.h;
#pragma unroll
  for (int n = 1; n <= kDeg; ++n) {
    double s = 0.0;
#pragma unroll
    for (int i = 1; i <= n; ++i) s = fma((double)i * r[i], E[n - i], s);
    E[n] = -F.lambda * s / n;
  }
  V0 = e0;
  V1 = e1;
  V2 = e2;
  if (!beyond_rs) {
#pragma unroll
    for (int n = 0; n <= kDeg; ++n) V[n] = E[n];
    return;
  }
  // S = 1 - z^3 (10 - z (15 - 6 z)), S' = -30 z^2 (1 - z)^2, z = (r - rs) / (rc - rs)
  const dd iw = dd_recip(dd_of(rc) - dd_of(rs));
  const dd z0 = (r0 - dd_of(rs)) * iw, z02 = z0 * z0, u = dd_of(1.0) - z0;
  const dd S0 = dd_of(1.0) - (z02 * z0) * (dd_of(10.0) - z0 * (dd_of(15.0) - 6.0 * z0));
  const dd dS = (-30.0) * (z02 * (u * u));                              // dS/dz
  const dd d2S = (-60.0) * ((z0 * u) * (dd_of(1.0) - 2.0 * z0));        // d2S/dz2
  const dd z1 = r1 * iw;
  const dd S1 = dS * z1;
  const dd S2 = 0.5 * (d2S * (z1 * z1)) + dS * (r2 * iw);
  V0 = e0 * S0;
  V1 = e1 * S0 + e0 * S1;
  V2 = e2 * S0 + e1 * S1 + e0 * S2;
  double z[kDeg + 1], z2[kDeg + 1], z3[kDeg + 1], p[kDeg + 1], t[kDeg + 1];
#pragma unroll
  for (int n = 0; n <= kDeg; ++n) z[n] = n == 0 ? z0.h : r[n] * iw.h;
#pragma unroll
  for (int n = 0; n <= kDeg; ++n) p[n] = (n == 0 ? 15.0 : 0.0) - 6.0 * z[n];
  mul(p, z, t);
#pragma unroll
  for (int n = 0; n <= kDeg; ++n) t[n] = (n == 0 ? 10.0 : 0.0) - t[n];
  mul(z, z, z2);
  mul(z2, z, z3);
  mul(z3, t, p);
#pragma unroll
  for (int n = 0; n <= kDeg; ++n) p[n] = -p[n];
  p[0] = S0.h;
  mul(E, p, V);
}

__device__ __forceinline__ uint32_t bits(float v) { return __float_as_uint(v); }
__device__ __forceinline__ void split(double v, float& h, float& l) {
  h = (float)v;
  l = (float)(v - (double)h);
}

struct TabJobs {
  RadialTab tab[3];
  int kind[3];
};

// rows [nrow][stride] 16-byte words of every table of a context in one launch;
// blockIdx.y: the term (density terms first, then pair terms; slots beyond the
// potential's terms stay zero), blockIdx.z: the table
__global__ void __launch_bounds__(32) k_radial_table(const __grid_constant__ DevPot P,
                                                     const __grid_constant__ TabJobs J) {
  const RadialTab& Tb = J.tab[blockIdx.z];
  const int kind = J.kind[blockIdx.z];
  const int row = blockIdx.x * blockDim.x + threadIdx.x, u = blockIdx.y, nterm = Tb.nf_slots + Tb.np_slots;
  if (row >= Tb.nrow || u >= nterm) return;
  uint4* line = const_cast<uint4*>(Tb.rows) + (int64_t)row * Tb.stride;
  uint4* out = line + u * Tb.words;
  if (u == 0)
    for (int t = nterm * Tb.words; t < Tb.stride; ++t) line[t] = make_uint4(0, 0, 0, 0);  // padding
  const RadialFn* F = nullptr;
  if (u < Tb.nf_slots) {
    if (u < P.n_f) F = &P.f[u];
  } else if (u - Tb.nf_slots < P.n_phi) {
    F = &P.phi[u - Tb.nf_slots];
  }
  if (F == nullptr || row == Tb.nrow - 1) {
    for (int t = 0; t < Tb.words; ++t) out[t] = make_uint4(0, 0, 0, 0);
    return;
  }
  // rows step by one at r_switch^2: its interval has a row for each side
  const int mid = row - Tb.n_low, ks = (int)(Tb.rs_hi >> Tb.shift) - Tb.k_lo;
  const bool beyond = mid > ks;
  double h = Tb.h;
  int k = mid - (beyond ? 1 : 0) + Tb.k_lo;
  if (mid < 0) {
    const int oct = min(row >> 6, 2);  // [1/4, 1/2), [1/2, 1), from 1 on
    h = 1.0 / (256 >> oct);
    k = row - 64 * (oct - 1);
  } else if (row >= Tb.n_main) {
    h *= 1.0 / (1 << kTabNarrow);
    k = row - Tb.n_main + (int)(Tb.near_hi >> (Tb.shift - kTabNarrow));
  }
  const double wc = ((double)k + 0.5) * h;
  dd V0, V1, V2;
  double V[kDeg + 1];
  term_series(*F, wc, h, beyond, P.rs, P.rc, V0, V1, V2, V);
  if (kind == kTabTaylor64) {
    double2* o = reinterpret_cast<double2*>(out);
    o[0] = make_double2(V0.h, V1.h);
    o[1] = make_double2(V2.h, V[3]);
    o[2] = make_double2(V[4], V[5]);
    o[3] = make_double2(V[6], V[7]);
    o[4] = make_double2(V[8], V[9]);
    return;
  }
  dd c0 = V0;
  double c[8] = {0.0, V1.h, V2.h, V[3], V[4], V[5], V[6], V[7]};
  double c1l = V1.l;
  if (kind == kTabDeriv64) {  // dV/dr / r = 2 dV/dw
    c0 = (2.0 / h) * V1;
    c[1] = (4.0 / h) * V2.h;
    c1l = (4.0 / h) * V2.l;
#pragma unroll
    for (int n = 2; n < 8; ++n) c[n] = (2.0 / h) * (n + 1) * V[n + 1];
  } else if (kind == kTabValueFF) {
    // Chebyshev economisation of tau^6 on |tau| <= 1/2 (a = 1/2):
    // x^6 -> 3/2 a^2 x^4 - 9/16 a^4 x^2 + a^6/32
    c[4] += (1.5 / 4.0) * c[6];
    c[2] -= (9.0 / 256.0) * c[6];
    c0 = c0 + dd_of((1.0 / 2048.0) * c[6]);
  }
  float c1h, c1lf, c2h, c2l, c3h, c3l;
  c1h = (float)c[1];
  c1lf = (float)((c[1] - (double)c1h) + c1l);
  split(c[2], c2h, c2l);
  split(c[3], c3h, c3l);
  // the leading bits (derivatives 54, values 55) and the exponent
  unsigned long long w0 = 0ull;
  const int top = kind == kTabDeriv64 ? 53 : 54;
  if (c0.h != 0.0) {
    int x = ilogb(c0.h);
    long long m = __double2ll_rn(scalbn(c0.h, top - x)) + __double2ll_rn(scalbn(c0.l, top - x));
    if (m >= (2ll << top) || m <= -(2ll << top)) {
      m /= 2;
      x += 1;
    }
    const int e8 = x + 128;  // above 255: excluded by plan_radial_tab
    if (e8 > 0) {
      if (kind == kTabDeriv64) w0 = ((unsigned long long)(m >> 23) << 32) | ((unsigned long long)(m & 0x7fffff) << 8);
      else w0 = (unsigned long long)m << 8;
      w0 |= (unsigned)min(e8, 255);
    }
  }
  out[0] = make_uint4((unsigned)w0, (unsigned)(w0 >> 32), bits(c1h), bits(c1lf));
  if (kind == kTabValueFF) {
    // the nearest 16-bit heads of c2's low part and of c5
    const uint32_t pack = ((bits(c2l) + 0x8000u) & 0xffff0000u) | ((bits((float)c[5]) + 0x8000u) >> 16);
    out[1] = make_uint4(bits(c2h), pack, bits(c3h), bits((float)c[4]));
  } else {
    out[1] = make_uint4(bits(c2h), bits(c2l), bits(c3h), bits(c3l));
    out[2] = make_uint4(bits((float)c[4]), bits((float)c[5]), bits((float)c[6]), bits((float)c[7]));
  }
}

}  // namespace

// Whether the potential's terms may be tabulated, and the table's shape.  The
// Taylor terms fall as x^n / n! with x = lambda h / (4 r) for the exponential
// and as y^n with y = h / (4 r_switch (r_cut - r_switch)) for the switch (z is
// a polynomial of degree 5 in r): x <= 0.016 and y <= 0.004 keep the first
// dropped term (n = 8) below 2^-60 and the FP32 terms (n >= 4) below 2^-53 of
// the value, provided r = sqrt(w) itself converges: its terms fall as (h / 2w)^n,
// 1/100 at kTabRMin (at r = 0.7, for a cut-off of 2.8 A, 1/31 left 4e-14 of the
// value in FP64).  At lambda = 2.5, r near 1.5 every output's error against
// extended precision was at most the direct kernels'.  The table has to
// leave room in the 227 KB of shared memory of one block.  Lennard-Jones terms
// (r^-12 varies faster than any of the exponentials) keep the direct kernels.
bool plan_radial_tab(const DevPot& P, int kind, bool with_pairs, RadialTab& Tb) {
  Tb = RadialTab{};
  if (P.lj || P.S > 2 || P.n_f > 2 || P.n_phi + P.n_f == 0) return false;
  const double rc2 = P.rc * P.rc;
  if (!(rc2 < 60.0)) return false;
  double lam = 0.0, grow = 0.0;
  auto rate = [&](const RadialFn& F) {
    lam = std::max(lam, F.lambda);
    grow = std::min(grow, F.lambda);
  };
  for (int u = 0; u < P.n_phi; ++u) rate(P.phi[u]);
  for (int v = 0; v < P.n_f; ++v) rate(P.f[v]);
  if (!(lam < 1e3) || grow < 0.0) return false;
  // all-FP64 rows of degree 9 afford intervals twice as wide
  const bool taylor = kind == kTabTaylor64;
  const int bits_h = taylor ? 4 : 5;
  const double h = std::ldexp(1.0, -bits_h), r_lo = std::max(kTabRLow * P.rc, kTabRMin), wide = taylor ? 2.0 : 1.0;
  if (!(lam * h <= 0.016 * wide * 4.0 * r_lo)) return false;
  if (!(h <= 0.004 * wide * 4.0 * P.rs * (P.rc - P.rs))) return false;
  Tb.words = taylor ? kTabWordsTaylor : kind == kTabValueFF ? kTabWordsFF : kTabWords64;
  Tb.nf_slots = P.S;
  Tb.np_slots = !with_pairs ? 0 : P.S == 1 ? 1 : (P.n_phi <= 2 ? 2 : 3);
  Tb.stride = tab_stride(Tb.nf_slots + Tb.np_slots, Tb.words);
  Tb.h = h;
  Tb.shift = kTabFixedBits - 32 - bits_h;
  const bool graded = kind == kTabValueFF;
  Tb.k_lo = (int)std::floor((graded ? std::max(r_lo * r_lo, kTabMainW) : r_lo * r_lo) / h);
  Tb.main_hi = (unsigned)Tb.k_lo << Tb.shift;
  Tb.n_low = graded ? 64 + 2 * Tb.k_lo : 0;  // 64, 64 and 64 per unit of w from 1 on
  const double unit = std::ldexp(1.0, kTabFixedBits - 32);
  Tb.rs_hi = (unsigned)std::floor(P.rs * P.rs * unit);
  Tb.rc_hi = (unsigned)std::ceil(rc2 * unit);
  if ((int)(Tb.rs_hi >> Tb.shift) < Tb.k_lo) return false;
  Tb.n_main = Tb.n_low + (int)((Tb.rc_hi - 1) >> Tb.shift) - Tb.k_lo + 2;  // both sides of r_switch
  Tb.nrow = Tb.n_main + 1;                                                   // and the zeros
  Tb.near_hi = 0xffffffffu;
  if (graded) {
    const double rn = P.rc - kTabNearU * (P.rc - P.rs);
    const unsigned kn = std::max((unsigned)std::floor(rn * rn / h), (Tb.rs_hi >> Tb.shift) + 1u);
    if (kn <= (Tb.rc_hi - 1) >> Tb.shift) {
      Tb.near_hi = kn << Tb.shift;
      Tb.n_main = Tb.n_low + (int)kn - Tb.k_lo + 1;
      const int sh = Tb.shift - kTabNarrow;
      Tb.nrow = Tb.n_main + (int)((Tb.rc_hi - 1) >> sh) - (int)(Tb.near_hi >> sh) + 2;
    }
  }
  Tb.first = Tb.n_low - Tb.k_lo;
  Tb.first_near = Tb.n_main - 1 - (int)(Tb.near_hi >> (Tb.shift - kTabNarrow));  // one less: beyond r_switch
  if ((int64_t)Tb.nrow * Tb.stride * 16 > kTabMaxBytes) return false;
  for (int u = 0; u < Tb.nf_slots + Tb.np_slots; ++u) {
    const int f = u, p = u - Tb.nf_slots;
    const RadialFn* F = u < Tb.nf_slots ? (f < P.n_f ? &P.f[f] : nullptr) : (p < P.n_phi ? &P.phi[p] : nullptr);
    // largest value: at the first row's lower end (the terms decrease)
    const double wl = graded ? 0.25 : Tb.k_lo * h;
    const double vmax = F ? F->A * std::exp(F->kappa - F->lambda * std::sqrt(wl)) : 1.0;
    if (!std::isfinite(vmax) || vmax > 1e30) return false;
    if (F && vmax < 1e-30) return false;
    // the other rows have 8 bits of exponent, 2^-127 .. 2^127; from the first row
    // to the last a term falls by less than 2^55 (float-float 2^70) within the
    // limits above
    if (!taylor && F && vmax < (graded ? 1e-15 : 1e-20)) return false;
    if (kind == kTabDeriv64 && F && vmax > 1e20) return false;
  }
  return true;
}

cudaError_t launch_radial_tables(const DevPot& P, const int* kinds, const RadialTab* const* tabs, int count,
                                 cudaStream_t s) {
  if (count < 1 || count > 3) return cudaErrorInvalidValue;
  TabJobs J;
  int rows = 0, terms = 0;
  for (int t = 0; t < 3; ++t) {
    J.tab[t] = *tabs[t < count ? t : 0];
    J.kind[t] = kinds[t < count ? t : 0];
    rows = std::max(rows, J.tab[t].nrow);
    terms = std::max(terms, J.tab[t].nf_slots + J.tab[t].np_slots);
  }
  k_radial_table<<<dim3((rows + 31) / 32, terms, count), 32, 0, s>>>(P, J);
  return cudaGetLastError();
}

}  // namespace mxe
