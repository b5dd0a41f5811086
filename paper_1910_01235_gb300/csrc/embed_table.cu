// embed_table.cu -- the exact phase average of the embedding term (App. B.2,
// eam.cu) in FP64 with the density terms from Taylor rows in r^2.
//
// Same two passes over every site's row as eam.cu's: k_emb_nodes_tab the rule
// data of each site, k_emb_grad_tab the derivatives.  The direct kernels sit on
// the FP64 pipe (85 %) with a square root, a switch, an exponential per species
// pair and a division per node.  Here
//  - each distinct density term is evaluated once per node (a row's Horner
//    scheme: 9 FMAs for the value, 8 more for the derivative), not once per
//    species pair and rule;
//  - when the two sites of an entry have equally large rules (the bulk), the
//    nodes that move a site are the same in both rules and are evaluated once;
//  - F = -E sqrt(rho) enters through 1/sqrt(rho) alone, and when the density
//    does not depend on the site's own species (tab 1) one root serves both;
//    the roots of a site's own nodes are kept by the first pass;
//  - node vectors are d with one shifted component, so forces accumulate a
//    scalar and the shift.
// 5,324-site alloy (287 k entries): nodes 1.69 ms and derivatives 4.81 ms with
// the direct kernels, 0.36 and 0.95 ms here.
// Rows are read through L1: the kernels stay bound by the FP64 pipe, and small
// blocks spread few sites evenly over the SMs.
#include <cuda_runtime.h>

#include "pair_common.cuh"
#include "taylor_rows.cuh"

namespace mxe {
namespace {

constexpr int kEmbLanes = 8, kEmbThreads = 64;

// distinct densities of a site: one when every species sees the same (tab 1)
template <int S, int TAB>
constexpr int n_dens() {
  return TAB == 1 ? 1 : S;
}

// weight of the distinct term v in density kd from a site with fractions x
template <int S, int TAB>
__device__ __forceinline__ double term_weight(const DevPot& P, int kd, int v, const double* x) {
  if (TAB == 1) return x[v];
  double w = 0.0;
#pragma unroll
  for (int l = 0; l < S; ++l)
    if (P.f_of[kd][l] == v) w += x[l];
  return w;
}

// 1/sqrt(rho) and sqrt(rho) (one Newton correction), zero at or below the
// smallest admissible density
__device__ __forceinline__ double inv_root(double rho) { return rho > kRhoMin ? rsqrt(rho) : 0.0; }
__device__ __forceinline__ double root_of(double rho, double is) {
  const double s = rho * is;
  return fma(0.5 * is, fma(-s, s, rho), s);
}

struct EntryGeom {
  double d[3], D2;
};
__device__ __forceinline__ void entry_geom(const DevGrid& g, const PassArgs& A, int64_t i, int64_t j, EntryGeom& G) {
  G.D2 = 0.0;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    double da = __ldg(&A.q[a * A.n + j]) - __ldg(&A.q[a * A.n + i]);
    da -= g.L[a] * rint(da * g.invL[a]);
    G.d[a] = da;
    G.D2 = fma(da, da, G.D2);
  }
}

// values of the density terms at w
template <int NF>
__device__ __forceinline__ void values_at(const DevPot& P, const TaylorTab& Tb, double w, double* f) {
  double tau;
  const double2* row = taylor_row(Tb, Tb.t.rows, w, tau);
#pragma unroll
  for (int v = 0; v < NF; ++v) {
    if (row) {
      const double2* r = row + v * kTabWordsTaylor;
      const double2 a = r[0], b = r[1], c = r[2], d = r[3], e = r[4];
      double s = fma(e.y, tau, e.x);
      s = fma(s, tau, d.y);
      s = fma(s, tau, d.x);
      s = fma(s, tau, c.y);
      s = fma(s, tau, c.x);
      s = fma(s, tau, b.y);
      s = fma(s, tau, b.x);
      s = fma(s, tau, a.y);
      f[v] = fma(s, tau, a.x);
    } else {
      f[v] = term_at(P, Tb, nullptr, v, w, tau).v;
    }
  }
}
// values and f'(r) / r = 2 df/dw
template <int NF>
__device__ __forceinline__ void terms_at(const DevPot& P, const TaylorTab& Tb, double w, double* f, double* g) {
  double tau;
  const double2* row = taylor_row(Tb, Tb.t.rows, w, tau);
#pragma unroll
  for (int v = 0; v < NF; ++v) {
    const V3 t = term_at(P, Tb, row, v, w, tau);  // the unused second derivative is dropped by the compiler
    f[v] = t.v;
    g[v] = t.d1 * (2.0 * Tb.ih);
  }
}

template <int C>
__device__ __forceinline__ void team_sum(double* v) {
#pragma unroll
  for (int c = 0; c < C; ++c)
    for (int o = kEmbLanes >> 1; o > 0; o >>= 1) v[c] += __shfl_xor_sync(0xffffffffu, v[c], o);
}

// First pass.  EmbArgs here: rhob [ND][n] densities, rown [6 ND][n] 1/sqrt of
// the densities at the site's own nodes, fsum [ND][n] sum of 1/sqrt over all
// nodes, emb [S][n] <F_k>, nrule [n].
template <int S, int TAB>
__global__ void __launch_bounds__(kEmbThreads) k_emb_nodes_tab(const __grid_constant__ DevPot P,
                                                               const __grid_constant__ DevGrid g0,
                                                               const __grid_constant__ PassArgs A,
                                                               const __grid_constant__ EmbArgs E,
                                                               const __grid_constant__ TaylorTab Tb) {
  constexpr int NF = S, ND = n_dens<S, TAB>();
  if (A.ctrl != nullptr && A.ctrl->halted) return;
  const int64_t tid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, n = A.n;
  const int64_t i = tid / kEmbLanes;
  const int lane = (int)(tid % kEmbLanes);
  const bool active = i < n;
  const double rc2 = P.rc * P.rc, rmin2 = kRMin * kRMin;
  const DevGrid* gp = active && A.batch.nsys ? &A.batch.grids[A.batch.sys_of[i]] : nullptr;
  const DevGrid& g = gp ? *gp : g0;
  const int beg = active ? A.nb_off[i] : 0, end = active ? A.nb_off[i + 1] : 0;
  const double sig = active ? A.sigma[i] : 0.0;
  int bad = 0, cnt = 0;
  for (int t = beg + lane; t < end; t += kEmbLanes) {
    EntryGeom G;
    entry_geom(g, A, i, __ldg(&A.nb_ent[t]) & kIdxMask, G);
    cnt += G.D2 < rc2;
  }
  for (int o = kEmbLanes >> 1; o > 0; o >>= 1) cnt += __shfl_xor_sync(0xffffffffu, cnt, o);
  const int N = cnt + 1;
  const double hs = sqrt((double)(3 * N)), hi = sig * hs;
  // densities at the mean [0] and at the six nodes that move i [1..6]
  double rho[ND * 7];
#pragma unroll
  for (int c = 0; c < ND * 7; ++c) rho[c] = 0.0;
  for (int t = beg + lane; t < end; t += kEmbLanes) {
    const int64_t j = __ldg(&A.nb_ent[t]) & kIdxMask;
    EntryGeom G;
    entry_geom(g, A, i, j, G);
    if (!(G.D2 < rc2)) continue;
    bad |= G.D2 < rmin2;
    double x[S], f[NF];
#pragma unroll
    for (int l = 0; l < S; ++l) x[l] = __ldg(&A.x[l * n + j]);
#pragma unroll
    for (int node = 0; node < 7; ++node) {
      double w = G.D2;
      if (node > 0) {
        const int a = (node - 1) >> 1;
        const double h = (node - 1) & 1 ? -hi : hi;  // q_i + h e_a: d_a -> d_a - h
        w = fma(h, fma(-2.0, G.d[a], h), G.D2);
        bad |= w < rmin2;
      }
      values_at<NF>(P, Tb, w, f);
#pragma unroll
      for (int k = 0; k < ND; ++k)
#pragma unroll
        for (int v = 0; v < NF; ++v) rho[7 * k + node] = fma(term_weight<S, TAB>(P, k, v, x), f[v], rho[7 * k + node]);
    }
  }
  team_sum<ND * 7>(rho);
  // species with an embedding energy at an occupied site need every density
  double xi[S];
  bool need[ND];
#pragma unroll
  for (int k = 0; k < ND; ++k) need[k] = false;
#pragma unroll
  for (int k = 0; k < S; ++k) {
    xi[k] = active ? A.x[k * n + i] : 0.0;
    need[TAB == 1 ? 0 : k] |= P.E[k] != 0.0 && xi[k] > 0.0;
  }
  // the nodes that move a member j: rho = rho_bar - x_j f(r_bar) + x_j f(r_node)
  double sums[2 * ND];  // of sqrt(rho), of 1/sqrt(rho)
#pragma unroll
  for (int c = 0; c < 2 * ND; ++c) sums[c] = 0.0;
  for (int t = beg + lane; t < end; t += kEmbLanes) {
    const int64_t j = __ldg(&A.nb_ent[t]) & kIdxMask;
    EntryGeom G;
    entry_geom(g, A, i, j, G);
    if (!(G.D2 < rc2)) continue;
    double x[S], f[NF], base[ND];
#pragma unroll
    for (int l = 0; l < S; ++l) x[l] = __ldg(&A.x[l * n + j]);
    values_at<NF>(P, Tb, G.D2, f);
#pragma unroll
    for (int k = 0; k < ND; ++k) {
      base[k] = rho[7 * k];
#pragma unroll
      for (int v = 0; v < NF; ++v) base[k] = fma(-term_weight<S, TAB>(P, k, v, x), f[v], base[k]);
    }
    const double hj = __ldg(&A.sigma[j]) * hs;
#pragma unroll
    for (int node = 0; node < 6; ++node) {
      const double h = node & 1 ? -hj : hj;  // q_j + h e_a
      const double w = fma(h, fma(2.0, G.d[node >> 1], h), G.D2);
      bad |= w < rmin2;
      values_at<NF>(P, Tb, w, f);
#pragma unroll
      for (int k = 0; k < ND; ++k) {
        double r = base[k];
#pragma unroll
        for (int v = 0; v < NF; ++v) r = fma(term_weight<S, TAB>(P, k, v, x), f[v], r);
        const double is = inv_root(r);
        if (is == 0.0 && need[k]) bad = 1;
        sums[2 * k] += root_of(r, is);
        sums[2 * k + 1] += is;
      }
    }
  }
  team_sum<2 * ND>(sums);
  bad = __reduce_or_sync(0xffffffffu, bad);
  if (!active || lane != 0) return;
#pragma unroll
  for (int k = 0; k < ND; ++k) {
#pragma unroll
    for (int v = 0; v < 6; ++v) {
      const double r = rho[7 * k + 1 + v], is = inv_root(r);
      if (is == 0.0 && need[k]) bad = 1;
      sums[2 * k] += root_of(r, is);
      sums[2 * k + 1] += is;
      E.rown[(6 * k + v) * n + i] = is;
    }
    E.rhob[k * n + i] = rho[7 * k];
    E.fsum[k * n + i] = sums[2 * k + 1];
  }
  const double invM = 1.0 / (6.0 * N);
  double eV = 0.0;
#pragma unroll
  for (int k = 0; k < S; ++k) {
    const double F = -P.E[k] * sums[TAB == 1 ? 0 : 2 * k] * invM;
    E.emb[k * n + i] = F;
    eV = fma(xi[k], F, eV);
  }
  E.nrule[i] = N;
  if (A.site_E) A.site_E[i] += eV;
  if (bad) atomicOr(A.flags, kFlagGeometry);
}

// Second pass: derivatives of sum_i x_ik <F_k(rho_i^k)> with respect to q_m,
// sigma_m, x_m; the five contributions of an entry (m, j) are numbered as in
// eam.cu.
template <int S, int TAB>
__global__ void __launch_bounds__(kEmbThreads) k_emb_grad_tab(const __grid_constant__ DevPot P,
                                                              const __grid_constant__ DevGrid g0,
                                                              const __grid_constant__ PassArgs A,
                                                              const __grid_constant__ EmbArgs E,
                                                              const __grid_constant__ TaylorTab Tb) {
  constexpr int NF = S, ND = n_dens<S, TAB>();
  if (A.ctrl != nullptr && A.ctrl->halted) return;
  const int64_t tid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, n = A.n;
  const int64_t m = tid / kEmbLanes;
  const int lane = (int)(tid % kEmbLanes);
  const bool active = m < n;
  const double rc2 = P.rc * P.rc;
  const DevGrid* gp = active && A.batch.nsys ? &A.batch.grids[A.batch.sys_of[m]] : nullptr;
  const DevGrid& gr = gp ? *gp : g0;
  const int beg = active ? A.nb_off[m] : 0, end = active ? A.nb_off[m + 1] : 0;
  const int Nm = active ? E.nrule[m] : 1;
  const double sm = active ? A.sigma[m] : 0.0;
  const double hsm = sqrt((double)(3 * Nm)), invMm = 1.0 / (6.0 * Nm);
  // x F' of a node is xe / sqrt(rho): xe = -1/2 sum_k x_k E_k over the species of
  // the density
  double xm[S], xe[ND], rbm[ND], own[ND][6], wm[ND][NF];
#pragma unroll
  for (int k = 0; k < ND; ++k) xe[k] = 0.0;
#pragma unroll
  for (int k = 0; k < S; ++k) {
    xm[k] = active ? A.x[k * n + m] : 0.0;
    xe[TAB == 1 ? 0 : k] = fma(-0.5 * xm[k], P.E[k], xe[TAB == 1 ? 0 : k]);
  }
#pragma unroll
  for (int k = 0; k < ND; ++k) {
    xe[k] *= invMm;
    rbm[k] = active ? E.rhob[k * n + m] : 0.0;
#pragma unroll
    for (int v = 0; v < 6; ++v) own[k][v] = active ? xe[k] * E.rown[(6 * k + v) * n + m] : 0.0;
#pragma unroll
    for (int v = 0; v < NF; ++v) wm[k][v] = term_weight<S, TAB>(P, k, v, xm);
  }
  double g[3] = {0.0, 0.0, 0.0}, gsig = 0.0, wsum[ND], muv[ND][NF], Gst[ND][3];
#pragma unroll
  for (int k = 0; k < ND; ++k) {
    wsum[k] = 0.0;
#pragma unroll
    for (int v = 0; v < NF; ++v) muv[k][v] = 0.0;
#pragma unroll
    for (int c = 0; c < 3; ++c) Gst[k][c] = 0.0;
  }
  for (int t = beg + lane; t < end; t += kEmbLanes) {
    const int64_t j = __ldg(&A.nb_ent[t]) & kIdxMask;
    EntryGeom G;
    entry_geom(gr, A, m, j, G);  // d = q_j - q_m
    if (!(G.D2 < rc2)) continue;
    double x[S], wj[ND][NF], xej[ND], fb[NF], gb[NF], used[ND], rbj[ND], Wt[ND];
    const int Nj = E.nrule[j];
    const bool same = Nj == Nm;  // then hsj == hsm: the rules share their nodes
    const double hsj = same ? hsm : sqrt((double)(3 * Nj)), invMj = same ? invMm : 1.0 / (6.0 * Nj);
#pragma unroll
    for (int k = 0; k < ND; ++k) xej[k] = used[k] = Wt[k] = 0.0;
#pragma unroll
    for (int k = 0; k < S; ++k) {
      x[k] = __ldg(&A.x[k * n + j]);
      xej[TAB == 1 ? 0 : k] = fma(-0.5 * x[k], P.E[k], xej[TAB == 1 ? 0 : k]);
    }
#pragma unroll
    for (int k = 0; k < ND; ++k) {
      xej[k] *= invMj;
      rbj[k] = E.rhob[k * n + j];
#pragma unroll
      for (int v = 0; v < NF; ++v) wj[k][v] = term_weight<S, TAB>(P, k, v, x);
    }
    const double sj = __ldg(&A.sigma[j]);
    terms_at<NF>(P, Tb, G.D2, fb, gb);
    double along = 0.0;  // force along d: sum of all weights
    double sb[ND], sbm[ND];
#pragma unroll
    for (int k = 0; k < ND; ++k) {
      sb[k] = sbm[k] = 0.0;
#pragma unroll
      for (int v = 0; v < NF; ++v) {
        sb[k] = fma(wj[k][v], gb[v], sb[k]);
        sbm[k] = fma(wm[k][v], gb[v], sbm[k]);
      }
      // static density gradient of m (times the weights of (2) after the row)
#pragma unroll
      for (int c = 0; c < 3; ++c) Gst[k][c] = fma(sb[k], G.d[c], Gst[k][c]);
    }
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      double shift = 0.0;  // the extra force along axis a
#pragma unroll 1
      for (int pm = 0; pm < 2; ++pm) {
        const int node = 2 * a + pm;
        const double sgn = pm == 0 ? 1.0 : -1.0, da = G.d[a];
        double f[NF], gn[NF];
        // the nodes that move m by h = +-sigma_m sqrt(3 N): separation d - h e_a
        {
          double h = sgn * sm * hsm;
          terms_at<NF>(P, Tb, fma(h, fma(-2.0, da, h), G.D2), f, gn);
          // (1) in m's rule
          double W = 0.0;
#pragma unroll
          for (int k = 0; k < ND; ++k) {
            double s = 0.0;
#pragma unroll
            for (int v = 0; v < NF; ++v) s = fma(wj[k][v], gn[v], s);
            W = fma(own[k][node], s, W);
          }
          along -= W;
          shift = fma(W, h, shift);
          gsig -= W * (da - h) * (sgn * hsm);
          // (4) in j's rule
          if (!same) {
            h = sgn * sm * hsj;
            terms_at<NF>(P, Tb, fma(h, fma(-2.0, da, h), G.D2), f, gn);
          }
          W = 0.0;
#pragma unroll
          for (int k = 0; k < ND; ++k) {
            double r = rbj[k], s = 0.0;
#pragma unroll
            for (int v = 0; v < NF; ++v) {
              r = fma(wm[k][v], f[v] - fb[v], r);
              s = fma(wm[k][v], gn[v], s);
            }
            const double is = inv_root(r), w = xej[k] * is;
            used[k] += is;
            W = fma(w, s, W);
#pragma unroll
            for (int v = 0; v < NF; ++v) muv[k][v] = fma(w, f[v], muv[k][v]);
          }
          along -= W;
          shift = fma(W, h, shift);
          gsig += W * (h - da) * (sgn * hsj);
        }
        // the nodes that move j by h = +-sigma_j sqrt(3 N): separation d + h e_a
        {
          double h = sgn * sj * hsm;
          terms_at<NF>(P, Tb, fma(h, fma(2.0, da, h), G.D2), f, gn);
          // (2) in m's rule
          double W = 0.0;
#pragma unroll
          for (int k = 0; k < ND; ++k) {
            double r = rbm[k], s = 0.0;
#pragma unroll
            for (int v = 0; v < NF; ++v) {
              r = fma(wj[k][v], f[v] - fb[v], r);
              s = fma(wj[k][v], gn[v], s);
            }
            const double w = xe[k] * inv_root(r);
            Wt[k] += w;
            W = fma(w, s, W);
          }
          along -= W;
          shift = fma(-W, h, shift);
          // (3) in j's rule
          if (!same) {
            h = sgn * sj * hsj;
            terms_at<NF>(P, Tb, fma(h, fma(2.0, da, h), G.D2), f, gn);
          }
          W = 0.0;
#pragma unroll
          for (int k = 0; k < ND; ++k) {
            const double is = E.rown[(6 * k + node) * n + j], w = xej[k] * is;
            double s = 0.0;
            used[k] += is;
#pragma unroll
            for (int v = 0; v < NF; ++v) {
              s = fma(wm[k][v], gn[v], s);
              muv[k][v] = fma(w, f[v], muv[k][v]);
            }
            W = fma(w, s, W);
          }
          along -= W;
          shift = fma(-W, h, shift);
        }
      }
      g[a] += shift;
    }
#pragma unroll
    for (int k = 0; k < ND; ++k) {
      // (2): + x_j f'(r_bar) d / r_bar with the summed weights
      along = fma(Wt[k], sb[k], along);
      wsum[k] += Wt[k];
      // (5) every other node of j's rule: r_jm at its mean
      const double w = xej[k] * (E.fsum[k * n + j] - used[k]);
      along = fma(-w, sbm[k], along);
#pragma unroll
      for (int v = 0; v < NF; ++v) muv[k][v] = fma(w, fb[v], muv[k][v]);
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) g[c] = fma(along, G.d[c], g[c]);
  }
  double red[4 + ND * (4 + NF)];
#pragma unroll
  for (int c = 0; c < 3; ++c) red[c] = g[c];
  red[3] = gsig;
#pragma unroll
  for (int k = 0; k < ND; ++k) {
    red[4 + k * (4 + NF)] = wsum[k];
#pragma unroll
    for (int c = 0; c < 3; ++c) red[5 + k * (4 + NF) + c] = Gst[k][c];
#pragma unroll
    for (int v = 0; v < NF; ++v) red[8 + k * (4 + NF) + v] = muv[k][v];
  }
  team_sum<4 + ND * (4 + NF)>(red);
  if (!active || lane != 0) return;
#pragma unroll
  for (int k = 0; k < ND; ++k)
#pragma unroll
    for (int c = 0; c < 3; ++c) red[c] -= red[4 + k * (4 + NF)] * red[5 + k * (4 + NF) + c];
  bool finite = isfinite(red[0]) && isfinite(red[1]) && isfinite(red[2]) && isfinite(red[3]);
  if (A.gq) {
#pragma unroll
    for (int c = 0; c < 3; ++c) A.gq[c * n + m] += red[c];
  }
  if (A.gs) A.gs[m] += red[3];
  if (A.mu_ex || A.mu) {
#pragma unroll
    for (int l = 0; l < S; ++l) {
      double v = E.emb[l * n + m];
#pragma unroll
      for (int k = 0; k < ND; ++k) {
        const int fo = TAB == 1 ? l : P.f_of[k][l];
#pragma unroll
        for (int u = 0; u < NF; ++u)
          if (fo == u) v += red[8 + k * (4 + NF) + u];
      }
      finite = finite && isfinite(v);
      if (A.mu_ex) A.mu_ex[l * n + m] += v;
      if (A.mu) A.mu[l * n + m] += v;
    }
  }
  if (!finite) atomicOr(A.flags, kFlagNonfinite);
}

}  // namespace

cudaError_t launch_emb_tab(bool second, const DevPot& P, const DevGrid& g, const PassArgs& A, const EmbArgs& E,
                           const RadialTab& tab, cudaStream_t s) {
  if (A.n == 0) return cudaSuccess;
  const TaylorTab Tb = taylor_tab(P, tab);
  const unsigned blocks = (unsigned)((A.n * kEmbLanes + kEmbThreads - 1) / kEmbThreads);
  auto run = [&](auto nodes, auto grad) {
    if (second) grad<<<blocks, kEmbThreads, 0, s>>>(P, g, A, E, Tb);
    else nodes<<<blocks, kEmbThreads, 0, s>>>(P, g, A, E, Tb);
    return cudaGetLastError();
  };
  if (P.S == 1) return run(k_emb_nodes_tab<1, 0>, k_emb_grad_tab<1, 0>);
  if (P.tab == 1) return run(k_emb_nodes_tab<2, 1>, k_emb_grad_tab<2, 1>);
  return run(k_emb_nodes_tab<2, 0>, k_emb_grad_tab<2, 0>);
}

}  // namespace mxe
