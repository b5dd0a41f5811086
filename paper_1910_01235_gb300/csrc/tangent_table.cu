// tangent_table.cu -- the forward-mode passes of deriv.cu over unordered pairs,
// with the radial terms from a table of FP64 Taylor rows (radial_table.cuh).
//
// Everything the tangents need of a term at a node is its value and its first
// two derivatives in w = r^2 (V, V', V''): one row, one Horner scheme of three
// accumulators.  With e = (1/12) sum over the 12 nodes of sum_u C_u V_u(w) plus
// the static term sum_v c_v f_v(|d|^2), and dw/dd, dw/ds polynomial in (d, s),
//   de/dd = (2/12) (d T + U) + 2 d A,   de/ds = (2/12) W_s,
// T = sum G, U_a = sum +-s G, W_s = sum (s +- d_a) G with G = sum_u C_u V'_u, and
// the tangents follow from G' = sum_u (C'_u V'_u + C_u V''_u w').  The pair is
// evaluated once (the dual-number passes do it from both ends, each node with
// an exponential per term): its record goes to both entries, and a gather sums
// the rows.  Term sensitivities are summed over the pairs in a fixed order.
//
// Bound by the FP64 pipe: about 24 FMAs per term and node.  10,976-site alloy
// (296 k pairs), values, tangents and term sensitivities: 11.5 ms with the
// dual-number passes, 2.1 ms here (FP64 pipe 93 % busy in the gradient kernel).
#include <cuda_runtime.h>

#include <algorithm>

#include "pair_common.cuh"
#include "radial_table.cuh"
#include "taylor_rows.cuh"

namespace mxe {
namespace {

constexpr int kTanThreads = 256;

// tangent of the separation and of the node offsets
struct PairRate {
  double d[3], dd, s_i, s_j;  // rates of d, d . d', rates of s_i and s_j
};
__device__ __forceinline__ void pair_rate(const TanArgs& A, int64_t i, int64_t j, const PairGeom& G, PairRate& D) {
#pragma unroll
  for (int a = 0; a < 3; ++a) D.d[a] = A.dq ? __ldg(&A.dq[a * A.n + j]) - __ldg(&A.dq[a * A.n + i]) : 0.0;
  D.dd = G.d[0] * D.d[0] + G.d[1] * D.d[1] + G.d[2] * D.d[2];
  D.s_i = A.dsigma ? kSqrt6 * __ldg(&A.dsigma[i]) : 0.0;
  D.s_j = A.dsigma ? kSqrt6 * __ldg(&A.dsigma[j]) : 0.0;
}
__device__ __forceinline__ double rate_of(const double* __restrict__ t, int64_t k) { return t ? __ldg(&t[k]) : 0.0; }

// Two doubles of a record of C (TanRec: the geometry records' buffer, idle during
// these passes, holds as many of a record's doubles as fit; with a buffer of its
// own the 12 doubles of two species took 46 GB for the lists of 4 million sites)
template <int C>
__device__ __forceinline__ double2* rec_at(const TanRec& R, int64_t t, int c) {
  const int ca = min(R.ca, C);
  return reinterpret_cast<double2*>(2 * c < ca ? R.a + t * ca + 2 * c : R.b + t * (C - ca) + (2 * c - ca));
}

// ---------------------------------------------------------------- densities
// Record of an entry: rho_bar, 12 <rho> of its site from the other one, per
// species, then their tangents: 4 S doubles.
template <int S>
__global__ void __launch_bounds__(kTanThreads) k_tan_pair_density(
    const __grid_constant__ DevPot P, const __grid_constant__ DevGrid g0, const __grid_constant__ TanArgs A,
    const __grid_constant__ TaylorTab Tb, const int4* __restrict__ pair_rec, int64_t npair, const TanRec rec) {
  constexpr int NF = S;
  extern __shared__ uint4 sm[];
  tab_stage(Tb.t, sm);
  __syncthreads();
  const int64_t n = A.n, stride = (int64_t)gridDim.x * blockDim.x;
  const double ih = 1.0 / Tb.t.h;
  for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < npair; p += stride) {
    PairRef pr;
    if (!load_pair(A, pair_rec, p, pr)) continue;
    PairGeom G;
    pair_geometry(g0, A, pr.i, pr.j, G);
    PairRate D;
    pair_rate(A, pr.i, pr.j, G, D);
    int bad = G.D2 < kRMin * kRMin;
    double fst[NF], fst_t[NF], fav[NF], fav_t[NF];
    {
      double tau;
      const double2* row = taylor_row(Tb, sm, G.D2, tau);
      const double td = 2.0 * D.dd * ih;
#pragma unroll
      for (int v = 0; v < NF; ++v) {
        const V3 f = term_at(P, Tb, row, v, G.D2, tau);
        fst[v] = f.v;
        fst_t[v] = f.d1 * td;
        fav[v] = fav_t[v] = 0.0;
      }
    }
#pragma unroll 1
    for (int k = 0; k < 12; ++k) {
      const int a = (k >> 1) % 3;
      const double da = a == 0 ? G.d[0] : a == 1 ? G.d[1] : G.d[2];
      const double dda = a == 0 ? D.d[0] : a == 1 ? D.d[1] : D.d[2];
      double s = k < 6 ? G.s_i : G.s_j, sd = k < 6 ? D.s_i : D.s_j;
      if (k & 1) {
        s = -s;
        sd = -sd;
      }
      const double w = fma(s, fma(2.0, da, s), G.D2);
      const double td = 2.0 * (D.dd + fma(sd, s + da, s * dda)) * ih;
      bad |= w < kRMin * kRMin;
      double tau;
      const double2* row = taylor_row(Tb, sm, w, tau);
#pragma unroll
      for (int v = 0; v < NF; ++v) {
        const V3 f = term_at(P, Tb, row, v, w, tau);
        fav[v] += f.v;
        fav_t[v] = fma(f.d1, td, fav_t[v]);
      }
    }
    double ri[4 * S], rj[4 * S];
#pragma unroll
    for (int c = 0; c < 4 * S; ++c) ri[c] = rj[c] = 0.0;
#pragma unroll
    for (int l = 0; l < S; ++l) {
      const double xi = __ldg(&A.x[l * n + pr.i]), xj = __ldg(&A.x[l * n + pr.j]);
      const double xid = rate_of(A.dx, l * n + pr.i), xjd = rate_of(A.dx, l * n + pr.j);
#pragma unroll
      for (int k = 0; k < S; ++k) {
        const int fo = P.f_of[k][l];
#pragma unroll
        for (int v = 0; v < NF; ++v)
          if (fo == v) {
            ri[k] += xj * fst[v];
            ri[S + k] += xj * fav[v];
            ri[2 * S + k] += xjd * fst[v] + xj * fst_t[v];
            ri[3 * S + k] += xjd * fav[v] + xj * fav_t[v];
            rj[k] += xi * fst[v];
            rj[S + k] += xi * fav[v];
            rj[2 * S + k] += xid * fst[v] + xi * fst_t[v];
            rj[3 * S + k] += xid * fav[v] + xi * fav_t[v];
          }
      }
    }
#pragma unroll
    for (int c = 0; c < 2 * S; ++c) {
      *rec_at<4 * S>(rec, pr.tp, c) = make_double2(ri[2 * c], ri[2 * c + 1]);
      *rec_at<4 * S>(rec, pr.tr, c) = make_double2(rj[2 * c], rj[2 * c + 1]);
    }
    if (bad) atomicOr(A.flags, kFlagGeometry);
  }
}

constexpr int kTanLanes = 8;  // lanes per site of the gathers

// sum of C doubles per entry over a site's row, complete on every lane of the team
template <int C>
__device__ __forceinline__ void team_sum(const TanRec& rec, int beg, int end, int lane, double* s) {
#pragma unroll
  for (int c = 0; c < C; ++c) s[c] = 0.0;
  for (int t = beg + lane; t < end; t += kTanLanes) {
#pragma unroll
    for (int c = 0; c < C / 2; ++c) {
      const double2 v = __ldg(rec_at<C>(rec, t, c));
      s[2 * c] += v.x;
      s[2 * c + 1] += v.y;
    }
  }
#pragma unroll
  for (int c = 0; c < C; ++c)
    for (int o = kTanLanes >> 1; o > 0; o >>= 1) s[c] += __shfl_xor_sync(0xffffffffu, s[c], o);
}

// rho_bar, <rho> and their tangents of every site, then the embedding terms e,
// a = x F'' (<rho> - rho_bar), b = x F' with F = -E sqrt(rho) (one lane per species)
template <int S>
__global__ void __launch_bounds__(256) k_tan_density_gather(const __grid_constant__ DevPot P,
                                                            const __grid_constant__ TanArgs A, const TanRec rec) {
  const int64_t tid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, n = A.n;
  const int64_t i = tid / kTanLanes;
  const int lane = (int)(tid % kTanLanes);
  const bool active = i < n;
  double s[4 * S];
  team_sum<4 * S>(rec, active ? A.nb_off[i] : 0, active ? A.nb_off[i + 1] : 0, lane, s);
  if (!active || lane >= S) return;
  const int k = lane;
  const double rb = S > 1 && k == 1 ? s[S - 1] : s[0], ra = (S > 1 && k == 1 ? s[2 * S - 1] : s[S]) * (1.0 / 12.0);
  const double rbt = S > 1 && k == 1 ? s[3 * S - 1] : s[2 * S];
  const double rat = (S > 1 && k == 1 ? s[4 * S - 1] : s[3 * S]) * (1.0 / 12.0);
  double e = 0.0, et = 0.0, a = 0.0, at = 0.0, b = 0.0, bt = 0.0;
  if (rb > kRhoMin) {
    const double E = P.E[k], x = A.x[k * n + i], xd = rate_of(A.dx, k * n + i);
    const double sq = sqrt(rb), inv = 1.0 / rb;
    const double F1 = -0.5 * E / sq, F2 = -0.5 * F1 * inv;  // F', F''
    const double F2t = -1.5 * F2 * inv * rbt, F1t = F2 * rbt;
    const double dr = ra - rb, drt = rat - rbt;
    e = -E * sq + F1 * dr;
    et = F1 * rbt + F1t * dr + F1 * drt;
    a = x * F2 * dr;
    at = xd * F2 * dr + x * (F2t * dr + F2 * drt);
    b = x * F1;
    bt = xd * F1 + x * F1t;
  } else {
    atomicOr(A.flags, kFlagGeometry);
  }
  A.e_v[k * n + i] = e;
  A.e_t[k * n + i] = et;
  A.a_v[k * n + i] = a;
  A.a_t[k * n + i] = at;
  A.b_v[k * n + i] = b;
  A.b_t[k * n + i] = bt;
}

// ---------------------------------------------------------------- gradients
// Record of an entry: dF/dq (3), dF/dsigma, mu (S) of its site from this pair,
// then their tangents: 2 (4 + S) doubles.  FULL false: only the tangents of
// dF/dq and dF/dsigma are wanted (Hessian products): 4 doubles.
template <int S, bool FULL>
constexpr int grad_len() {
  return FULL ? 2 * (4 + S) : 4;
}

template <int S, int NP, bool FULL>
__global__ void __launch_bounds__(kTanThreads) k_tan_pair_grad(
    const __grid_constant__ DevPot P, const __grid_constant__ DevGrid g0, const __grid_constant__ TanArgs A,
    const __grid_constant__ TaylorTab Tb, const int4* __restrict__ pair_rec, int64_t npair, const TanRec rec,
    double* __restrict__ th_part) {
  constexpr int NF = S, NT = NF + NP, RL = grad_len<S, FULL>();
  extern __shared__ uint4 sm[];
  tab_stage(Tb.t, sm);
  __syncthreads();
  const int64_t n = A.n, stride = (int64_t)gridDim.x * blockDim.x;
  const double h = Tb.t.h, ih = 1.0 / h, inv12 = 1.0 / 12.0;
  const bool theta = FULL && th_part != nullptr;
  // sums over this thread's pairs: dE/dc, dE/dlambda, their tangents
  double th[4][NT];
#pragma unroll
  for (int c = 0; c < 4; ++c)
#pragma unroll
    for (int u = 0; u < NT; ++u) th[c][u] = 0.0;
  for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < npair; p += stride) {
    PairRef pr;
    if (!load_pair(A, pair_rec, p, pr)) continue;
    const int64_t i = pr.i, j = pr.j;
    PairGeom G;
    pair_geometry(g0, A, i, j, G);
    PairRate D;
    pair_rate(A, i, j, G, D);
    int bad = G.D2 < kRMin * kRMin;
    // weights of the terms at the nodes (C) and at the static point (cs)
    double C[NT], Cd[NT], cs[NF], csd[NF];
#pragma unroll
    for (int u = 0; u < NT; ++u) C[u] = Cd[u] = 0.0;
#pragma unroll
    for (int v = 0; v < NF; ++v) cs[v] = csd[v] = 0.0;
#pragma unroll
    for (int k = 0; k < S; ++k) {
      const double xi = __ldg(&A.x[k * n + i]), xid = rate_of(A.dx, k * n + i);
      const double ai = A.a_v[k * n + i], aid = A.a_t[k * n + i], bi = A.b_v[k * n + i], bid = A.b_t[k * n + i];
      const double aj = A.a_v[k * n + j], ajd = A.a_t[k * n + j], bj = A.b_v[k * n + j], bjd = A.b_t[k * n + j];
#pragma unroll
      for (int l = 0; l < S; ++l) {
        const double yi = __ldg(&A.x[l * n + i]), yid = rate_of(A.dx, l * n + i);
        const double yj = __ldg(&A.x[l * n + j]), yjd = rate_of(A.dx, l * n + j);
        const int po = P.phi_of[k][l], fo = P.f_of[k][l];
#pragma unroll
        for (int u = 0; u < NP; ++u)
          if (po == u) {
            C[NF + u] += xi * yj;
            Cd[NF + u] += xid * yj + xi * yjd;
          }
#pragma unroll
        for (int v = 0; v < NF; ++v)
          if (fo == v) {
            C[v] += bi * yj + bj * yi;
            Cd[v] += bid * yj + bi * yjd + bjd * yi + bj * yid;
            cs[v] += ai * yj + aj * yi;
            csd[v] += aid * yj + ai * yjd + ajd * yi + aj * yid;
          }
      }
    }
    // static point
    double fst[NF], fst_t[NF], A1 = 0.0, A1d = 0.0;
    {
      double tau;
      const double2* row = taylor_row(Tb, sm, G.D2, tau);
      const double td = 2.0 * D.dd * ih;
      double r = 0.0, rd = 0.0;
      if (theta) {
        r = sqrt(G.D2);
        rd = D.dd / r;
      }
      double A2 = 0.0;
#pragma unroll
      for (int v = 0; v < NF; ++v) {
        const V3 f = term_at(P, Tb, row, v, G.D2, tau);
        fst[v] = f.v;
        fst_t[v] = f.d1 * td;
        A1 = fma(cs[v], f.d1, A1);
        A1d = fma(csd[v], f.d1, A1d);
        A2 = fma(cs[v], f.h2, A2);
        if (theta) {
          th[0][v] = fma(cs[v], f.v, th[0][v]);
          th[1][v] -= cs[v] * (r * f.v);
          th[2][v] += csd[v] * f.v + cs[v] * fst_t[v];
          th[3][v] -= csd[v] * (r * f.v) + cs[v] * (rd * f.v + r * fst_t[v]);
        }
      }
      A1d = fma(2.0 * A2, td, A1d);
    }
    // nodes: sums of G and of its tangent, and of every term's value
    double T = 0.0, Td = 0.0, U[3], Ud[3], W[2], Wd[2];
    double av[NT], avt[NT], lv[NT], lvt[NT];
#pragma unroll
    for (int u = 0; u < NT; ++u) av[u] = avt[u] = lv[u] = lvt[u] = 0.0;
#pragma unroll
    for (int a = 0; a < 3; ++a) U[a] = Ud[a] = 0.0;
#pragma unroll 1
    for (int site = 0; site < 2; ++site) {
      const double s = site == 0 ? G.s_i : G.s_j, sd = site == 0 ? D.s_i : D.s_j;
      double Ws = 0.0, Wsd = 0.0;
#pragma unroll 1
      for (int a = 0; a < 3; ++a) {
        const double da = a == 0 ? G.d[0] : a == 1 ? G.d[1] : G.d[2];
        const double dda = a == 0 ? D.d[0] : a == 1 ? D.d[1] : D.d[2];
        double ua = 0.0, uad = 0.0;
#pragma unroll
        for (int pm = 0; pm < 2; ++pm) {
          const double sg = pm == 0 ? s : -s, sgd = pm == 0 ? sd : -sd;
          const double w = fma(sg, fma(2.0, da, sg), G.D2);
          const double td = 2.0 * (D.dd + fma(sgd, sg + da, sg * dda)) * ih;
          bad |= w < kRMin * kRMin;
          double tau;
          const double2* row = taylor_row(Tb, sm, w, tau);
          double r = 0.0, rd = 0.0;
          if (theta) {
            const double ir = rsqrt(w);
            r = w * ir;
            rd = 0.5 * h * td * ir;
          }
          double g = 0.0, gd = 0.0, g2 = 0.0;
#pragma unroll
          for (int u = 0; u < NT; ++u) {
            const V3 f = term_at(P, Tb, row, u, w, tau);
            g = fma(C[u], f.d1, g);
            gd = fma(Cd[u], f.d1, gd);
            g2 = fma(C[u], f.h2, g2);
            if (FULL) {
              const double ft = f.d1 * td;
              av[u] += f.v;
              avt[u] += ft;
              if (theta) {
                lv[u] = fma(r, f.v, lv[u]);
                lvt[u] = fma(rd, f.v, fma(r, ft, lvt[u]));
              }
            }
          }
          gd = fma(2.0 * g2, td, gd);
          T += g;
          Td += gd;
          ua = fma(sg, g, ua);
          uad = fma(sgd, g, fma(sg, gd, uad));
          // dw/ds = 2 (s +- d_a)
          const double m = pm == 0 ? s + da : s - da, md = pm == 0 ? sd + dda : sd - dda;
          Ws = fma(m, g, Ws);
          Wsd = fma(md, g, fma(m, gd, Wsd));
        }
        if (a == 0) {
          U[0] += ua;
          Ud[0] += uad;
        } else if (a == 1) {
          U[1] += ua;
          Ud[1] += uad;
        } else {
          U[2] += ua;
          Ud[2] += uad;
        }
      }
      W[1] = Ws;
      Wd[1] = Wsd;
      if (site == 0) {
        W[0] = Ws;
        Wd[0] = Wsd;
      }
    }
    // (2/12)(d T + U) + 2 d A1, all sums still per tau: factor 1/h
    const double k12 = 2.0 * inv12 * ih, k2 = 2.0 * ih, ks = kSqrt6 * 2.0 * inv12 * ih;
    double gv[4], gt[4], gsj, gsjt;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      gv[a] = k12 * fma(G.d[a], T, U[a]) + k2 * G.d[a] * A1;
      gt[a] = k12 * (D.d[a] * T + G.d[a] * Td + Ud[a]) + k2 * (D.d[a] * A1 + G.d[a] * A1d);
    }
    gv[3] = ks * W[0];
    gt[3] = ks * Wd[0];
    gsj = ks * W[1];
    gsjt = ks * Wd[1];
    if constexpr (!FULL) {
      *rec_at<RL>(rec, pr.tp, 0) = make_double2(-gt[0], -gt[1]);
      *rec_at<RL>(rec, pr.tp, 1) = make_double2(-gt[2], gt[3]);
      *rec_at<RL>(rec, pr.tr, 0) = make_double2(gt[0], gt[1]);
      *rec_at<RL>(rec, pr.tr, 1) = make_double2(gt[2], gsjt);
    } else {
      double ri[RL], rj[RL];
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        ri[a] = -gv[a];
        rj[a] = gv[a];
        ri[4 + S + a] = -gt[a];
        rj[4 + S + a] = gt[a];
      }
      ri[3] = gv[3];
      rj[3] = gsj;
      ri[4 + S + 3] = gt[3];
      rj[4 + S + 3] = gsjt;
      // mu of species k: sum_l x_l phi_kl / 12 + sum_l (a_l f_lk + b_l f_lk / 12), the other site's x, a, b
#pragma unroll
      for (int k = 0; k < S; ++k) {
        double mi = 0.0, mit = 0.0, mj = 0.0, mjt = 0.0;
#pragma unroll
        for (int l = 0; l < S; ++l) {
          const int po = P.phi_of[k][l], fo = P.f_of[l][k];
          const double yi = __ldg(&A.x[l * n + i]), yid = rate_of(A.dx, l * n + i);
          const double yj = __ldg(&A.x[l * n + j]), yjd = rate_of(A.dx, l * n + j);
          const double ai = A.a_v[l * n + i], aid = A.a_t[l * n + i], bi = A.b_v[l * n + i], bid = A.b_t[l * n + i];
          const double aj = A.a_v[l * n + j], ajd = A.a_t[l * n + j], bj = A.b_v[l * n + j], bjd = A.b_t[l * n + j];
#pragma unroll
          for (int u = 0; u < NP; ++u)
            if (po == u) {
              const double q = av[NF + u] * inv12, qt = avt[NF + u] * inv12;
              mi += yj * q;
              mit += yjd * q + yj * qt;
              mj += yi * q;
              mjt += yid * q + yi * qt;
            }
#pragma unroll
          for (int v = 0; v < NF; ++v)
            if (fo == v) {
              const double q = av[v] * inv12, qt = avt[v] * inv12;
              mi += aj * fst[v] + bj * q;
              mit += ajd * fst[v] + aj * fst_t[v] + bjd * q + bj * qt;
              mj += ai * fst[v] + bi * q;
              mjt += aid * fst[v] + ai * fst_t[v] + bid * q + bi * qt;
            }
        }
        ri[4 + k] = mi;
        rj[4 + k] = mj;
        ri[2 * (4 + S) - S + k] = mit;
        rj[2 * (4 + S) - S + k] = mjt;
      }
#pragma unroll
      for (int c = 0; c < RL / 2; ++c) {
        *rec_at<RL>(rec, pr.tp, c) = make_double2(ri[2 * c], ri[2 * c + 1]);
        *rec_at<RL>(rec, pr.tr, c) = make_double2(rj[2 * c], rj[2 * c + 1]);
      }
      if (theta) {
#pragma unroll
        for (int u = 0; u < NT; ++u) {
          th[0][u] += inv12 * (C[u] * av[u]);
          th[1][u] -= inv12 * (C[u] * lv[u]);
          th[2][u] += inv12 * (Cd[u] * av[u] + C[u] * avt[u]);
          th[3][u] -= inv12 * (Cd[u] * lv[u] + C[u] * lvt[u]);
        }
      }
    }
    if (bad) atomicOr(A.flags, kFlagGeometry);
  }
  if (theta) {
    // block sums in a fixed order: lanes by butterfly, then the warps in turn
    __shared__ double red[kTanThreads / 32];
    for (int c = 0; c < 4; ++c)
#pragma unroll
      for (int u = 0; u < NT; ++u) {
        double v = th[0][u];
        if (c == 1) v = th[1][u];
        if (c == 2) v = th[2][u];
        if (c == 3) v = th[3][u];
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
        __syncthreads();
        if (threadIdx.x == 0) {
          double t = 0.0;
          for (int w = 0; w < (int)blockDim.x / 32; ++w) t += red[w];
          th_part[(int64_t)(c * NT + u) * gridDim.x + blockIdx.x] = t;
        }
        __syncthreads();
      }
  }
}

// th_out [4 T]: values of dE/dc, dE/dlambda, then their tangents; terms numbered
// pair terms first.  One warp per output, partials in a fixed order.
__global__ void __launch_bounds__(32) k_tan_theta(const __grid_constant__ DevPot P, int nf_slots, int nterm, int blocks,
                                                  const double* __restrict__ th_part, double* __restrict__ out) {
  const int T = P.n_phi + P.n_f, c = blockIdx.y, u = blockIdx.x;
  const int slot = u < P.n_phi ? nf_slots + u : u - P.n_phi;
  const double* col = th_part + (int64_t)(c * nterm + slot) * blocks;
  double v = 0.0;
  for (int b = threadIdx.x; b < blocks; b += 32) v += col[b];
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if (threadIdx.x == 0) out[c * T + u] = v;
}

template <int S, bool FULL>
__global__ void __launch_bounds__(256) k_tan_grad_gather(const __grid_constant__ TanArgs A, const TanRec rec) {
  constexpr int RL = grad_len<S, FULL>();
  const int64_t tid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, n = A.n;
  const int64_t i = tid / kTanLanes;
  const int lane = (int)(tid % kTanLanes);
  const bool active = i < n;
  double s[RL];
  team_sum<RL>(rec, active ? A.nb_off[i] : 0, active ? A.nb_off[i + 1] : 0, lane, s);
  if (!active) return;
  constexpr int t0 = FULL ? 4 + S : 0;  // first tangent
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    if (FULL && lane == c && A.gq_v) A.gq_v[c * n + i] = s[c];
    if (lane == c && A.gq_t) A.gq_t[c * n + i] = s[t0 + c];
  }
  if (lane == 3) {
    const double sg = A.sigma[i], th = 3.0 * kKB * A.T[i] / sg;
    if (FULL && A.gs_v) A.gs_v[i] = s[3] - th;
    if (A.gs_t) A.gs_t[i] = s[t0 + 3] + th * (rate_of(A.dsigma, i) / sg);
  }
  if constexpr (FULL) {
#pragma unroll
    for (int k = 0; k < S; ++k)
      if (lane == 4 + k) {
        if (A.mu_v) A.mu_v[k * n + i] = s[4 + k] + A.e_v[k * n + i];
        if (A.mu_t) A.mu_t[k * n + i] = s[t0 + 4 + k] + A.e_t[k * n + i];
      }
  }
}

bool wants_values(const TanArgs& A, bool theta) { return theta || A.gq_v || A.gs_v || A.mu_v || A.mu_t; }

template <typename... KArgs, typename... Args>
cudaError_t launch_staged(void (*kernel)(KArgs...), const RadialTab& Tb, int blocks, cudaStream_t s, Args... args) {
  const size_t shm = (size_t)Tb.nrow * Tb.stride * 16;
  cudaError_t e =
      cudaFuncSetAttribute((const void*)kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kTabMaxBytes);
  if (e != cudaSuccess) return e;
  kernel<<<blocks, kTanThreads, shm, s>>>(static_cast<KArgs>(args)...);
  return cudaGetLastError();
}

template <int S, int NP>
cudaError_t tangent_pairs(const DevPot& P, const DevGrid& g, const TanArgs& A, const RadialTab& dens_tab,
                          const RadialTab& tab, const int4* pair_rec, int64_t npair, const TanRec& rec,
                          double* th_part, double* th_out, cudaStream_t s) {
  const int blocks = tangent_blocks(npair);
  const unsigned gblocks = (unsigned)((A.n * kTanLanes + 255) / 256);
  cudaError_t e = launch_staged(k_tan_pair_density<S>, dens_tab, blocks, s, P, g, A, taylor_tab(P, dens_tab), pair_rec,
                                npair, rec);
  if (e != cudaSuccess) return e;
  k_tan_density_gather<S><<<gblocks, 256, 0, s>>>(P, A, rec);
  if (wants_values(A, th_out != nullptr)) {
    e = launch_staged(k_tan_pair_grad<S, NP, true>, tab, blocks, s, P, g, A, taylor_tab(P, tab), pair_rec, npair, rec,
                      th_out ? th_part : nullptr);
    if (e != cudaSuccess) return e;
    k_tan_grad_gather<S, true><<<gblocks, 256, 0, s>>>(A, rec);
    if (th_out)
      k_tan_theta<<<dim3(P.n_phi + P.n_f, 4), 32, 0, s>>>(P, tab.nf_slots, tab.nf_slots + tab.np_slots, blocks,
                                                          th_part, th_out);
  } else {
    e = launch_staged(k_tan_pair_grad<S, NP, false>, tab, blocks, s, P, g, A, taylor_tab(P, tab), pair_rec, npair, rec,
                      (double*)nullptr);
    if (e != cudaSuccess) return e;
    k_tan_grad_gather<S, false><<<gblocks, 256, 0, s>>>(A, rec);
  }
  return cudaGetLastError();
}

}  // namespace

int tangent_record_len(const DevPot& P, const TanArgs& A, bool theta) {
  return wants_values(A, theta) ? 2 * (4 + P.S) : 4 * P.S;  // the longer of both passes' records
}

int tangent_blocks(int64_t npair) {
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return 1;
  return (int)std::max<int64_t>(1, std::min<int64_t>((npair + kTanThreads - 1) / kTanThreads, sms));
}

cudaError_t launch_tangent_pairs(const DevPot& P, const DevGrid& g, const TanArgs& A, const RadialTab& dens_tab,
                                 const RadialTab& tab, const int4* pair_rec, int64_t npair, const TanRec& rec,
                                 double* th_part, double* th_out, cudaStream_t s) {
  if (A.n == 0) return cudaSuccess;
  if (P.S == 1) return tangent_pairs<1, 1>(P, g, A, dens_tab, tab, pair_rec, npair, rec, th_part, th_out, s);
  if (tab.np_slots == 2)
    return tangent_pairs<2, 2>(P, g, A, dens_tab, tab, pair_rec, npair, rec, th_part, th_out, s);
  return tangent_pairs<2, 3>(P, g, A, dens_tab, tab, pair_rec, npair, rec, th_part, th_out, s);
}

}  // namespace mxe
