// taylor_rows.cuh -- terms from FP64 Taylor rows (kind kTabTaylor64 of
// radial_table.cuh): value and derivatives in w = r^2, with the formula itself
// where the table does not reach.
#pragma once

#include "radial_table.cuh"

namespace mxe {

struct V3 {  // a term and its derivatives in tau = (w - w_k) / h: V, dV/dtau, 1/2 d2V/dtau2
  double v, d1, h2;
};

// the term at w from its formula (w below the first row, or not finite)
static __device__ __noinline__ V3 direct_term(const RadialFn& F, double rs, double rc, double w, double h) {
  const double r = sqrt(w), iw = 1.0 / (rc - rs);
  const double z = fmin(fmax((r - rs) * iw, 0.0), 1.0), u = 1.0 - z;
  const double S = 1.0 - z * z * z * (10.0 - z * (15.0 - 6.0 * z));
  const double S1 = -30.0 * z * z * u * u * iw, S2 = -60.0 * z * u * (1.0 - 2.0 * z) * iw * iw;
  const double E = F.A * exp(F.kappa - F.lambda * r), lam = F.lambda;
  const double Vr = E * (S1 - lam * S), Vrr = E * (S2 - 2.0 * lam * S1 + lam * lam * S);
  return V3{E * S, h * Vr / (2.0 * r), 0.5 * h * h * (Vrr - Vr / r) / (4.0 * w)};
}

struct TaylorTab {
  RadialTab t;
  double rs2, rc2, w_lo, ih;
};

// row of w; null: direct evaluation
__device__ __forceinline__ const double2* taylor_row(const TaylorTab& Tb, const uint4* sm, double w, double& tau) {
  const double y = w * Tb.ih, f = floor(y);
  tau = (y - f) - 0.5;
  if (!(w >= Tb.w_lo)) return nullptr;
  int k = w < Tb.rc2 ? (int)f - Tb.t.k_lo + (w >= Tb.rs2 ? 1 : 0) : Tb.t.nrow - 1;
  k = min(max(k, 0), Tb.t.nrow - 1);
  return reinterpret_cast<const double2*>(sm + k * Tb.t.stride);
}

__device__ __forceinline__ V3 taylor_eval(const double2* __restrict__ row, double t) {
  const double2 a = row[0], b = row[1], c = row[2], d = row[3], e = row[4];
  const double k[9] = {e.x, d.y, d.x, c.y, c.x, b.y, b.x, a.y, a.x};  // c8 .. c0
  double v = fma(e.y, t, k[0]), d1 = e.y, h2 = e.y;
  d1 = fma(d1, t, v);
  v = fma(v, t, k[1]);
#pragma unroll
  for (int n = 2; n < 9; ++n) {
    h2 = fma(h2, t, d1);
    d1 = fma(d1, t, v);
    v = fma(v, t, k[n]);
  }
  return V3{v, d1, h2};
}

// slot u of a row: density terms, then pair terms
__device__ __forceinline__ const RadialFn* slot_fn(const DevPot& P, const RadialTab& T, int u) {
  if (u < T.nf_slots) return u < P.n_f ? &P.f[u] : nullptr;
  return u - T.nf_slots < P.n_phi ? &P.phi[u - T.nf_slots] : nullptr;
}
__device__ __forceinline__ V3 term_at(const DevPot& P, const TaylorTab& Tb, const double2* row, int u, double w,
                                      double tau) {
  if (row) return taylor_eval(row + u * kTabWordsTaylor, tau);
  const RadialFn* F = slot_fn(P, Tb.t, u);
  return F ? direct_term(*F, P.rs, P.rc, w, Tb.t.h) : V3{0.0, 0.0, 0.0};
}

inline TaylorTab taylor_tab(const DevPot& P, const RadialTab& T) {
  return TaylorTab{T, P.rs * P.rs, P.rc * P.rc, T.k_lo * T.h, 1.0 / T.h};
}

}  // namespace mxe
