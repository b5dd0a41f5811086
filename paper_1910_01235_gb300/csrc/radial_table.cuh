// radial_table.cuh -- the radial terms of a potential as piecewise polynomials
// in the squared distance, for the FP64 passes and the accurate passes of the
// FP32 modes.
//
// Every node of App. A's rule needs g(r) (or dg/dr / r) of each radial term at
// r^2 = |d|^2 + s^2 +- 2 s d_a, which is known before any square root.  A term
// with its switch is a function of w = r^2 alone, so it is tabulated once per
// context: intervals of width h in w, on each a Taylor polynomial about the
// centre in tau = (w - w_k)/h, |tau| <= 1/2, formed in double-double arithmetic
// (radial_table.cu).  The square root, the exponentials and the switch leave
// the node loop.  On GB300, whose FP64 pipe has 2 lanes per SM against 128 FP32
// lanes, the point is the split of the polynomial: consecutive Taylor terms
// fall by about 2^-7, so only the constant term needs 53 bits.  It is an
// integer with the exponent of its own row: 55 bits for values (shifted to the
// grid of the pair's nearest node and added in 64-bit integers), 54 bits for
// derivatives (multiplied by the pair's weight in integer arithmetic first); the
// terms tau c1 .. tau^3 c3 run in float-float, tau^4 c4 .. in FP32.  One grid for
// all rows, set by the value at r_cut / 4, left the outer shells short of bits:
// with every neighbour at 4.95 A (r_cut 5, decay rate 1.96 / A) the energy was off
// by 5e-14 in FP64 and 2e-12 in float-float, 3e-15 and 9e-14 direct.
//
// The switch is only twice differentiable at r_switch and r_cut: the interval
// that holds a breakpoint has two rows, one per side, and the row index steps
// by one at each breakpoint; from r_cut on every w takes one row of zeros.
//
// w is a 64-bit integer in units of 2^-55 (w < 256): node distances are integer
// additions, the interval is a shift, and tau is the remaining bits.  Pairs
// with a node below the first row (float-float: 0.5 A; else r_cut / 4 or 1.25 A),
// with |d|^2 >= 128 or with a non-finite coordinate take the direct evaluation.
// (Units of 2^-56 sent pairs from 8 A on there, in lists of the longest cut-offs a
// quarter of all: 32,000 sites, r_cut 7.6 A, float-float free-energy call 1.8 ms
// with the direct kernels, 5.0 ms, now 1.5; FP64 15.8, 11.3, now 2.1.)
#pragma once

#include "mxe_internal.cuh"

namespace mxe {

// A row of one term, FP64 quality: c0, c1, c2, c3 as float pairs, c4..c7
// floats: three 16-byte words.  c0 of a value row is an int64 m with its low byte
// e8 in place of its own, for (m & ~255) 2^(e8 - kTabValueBias), 2^62 <= |m| <
// 2^63; of a derivative row m_hi (signed high word) and m_lo | e8 (low word, bit
// 31 clear), for (m_hi 2^31 + m_lo) 2^(e8 - kTabExpBias), |m_hi| < 2^31; both
// zero where e8 is 0.  Float-float quality (degree 5): c0, c1 and c2 pairs, c3,
// c4, c5 (tab_polyff): two words.
// All FP64 (degree 9, c0..c9; the tangent passes): five words.
constexpr int kTabWords64 = 3, kTabWordsFF = 2, kTabWordsTaylor = 5;
constexpr int kTabFixedBits = 55;   // w in units of 2^-55
constexpr int kTabExpBias = 128 + 61;    // of the derivative rows' exponents
constexpr int kTabValueBias = 128 + 62;  // of the value rows' exponents
constexpr double kTabRLow = 0.25, kTabRMin = 1.25;  // first row at r_cut / 4, not below 1.25 A
// Float-float rows hold c2 to 32 and c3, c5 to 24 and 8 bits.  Where the switch
// u = (r_cut - r) / (r_cut - r_switch) falls to the offset's share du of it, the
// terms are (du / u)^n of the value and those bits show (at u = 0.1, 4.95 A of 5:
// 1e-12 of the value, the direct kernels 1e-13).  Rows a quarter as wide from
// u = 0.3 on: du^2 / 16.
constexpr int kTabNarrow = 2;
constexpr double kTabNearU = 0.3;
// Below w = 2 (or (r_cut / 4)^2) float-float rows are 1/64 wide, from w = 1 down
// 64 to an octave, to w = 1/4: down to the smallest admissible node distance.
// For speed: a pair with a node below the first row took the direct evaluation in
// FP64, and its warp with it (host-solute slab of 16,384 sites, solute widths of
// 0.25 A: free-energy call 1495 us, 484 with the direct kernels, 285 now).  For
// precision: the terms dropped after degree 5 fall as w^-6 and left 8e-14 of the
// value at 1.25 A (decay rate 2.5 / A), the direct kernels 2e-14.
constexpr double kTabMainW = 2.0;

// 16-byte words between the rows of consecutive intervals: all terms of an
// interval lie side by side; an odd count spreads random intervals over the
// eight 16-byte bank groups of shared memory.
inline int tab_stride(int nterm, int words) { return (nterm * words) | 1; }

__device__ __forceinline__ void tab_stage(const RadialTab& Tb, uint4* __restrict__ sm) {
  const int n = Tb.nrow * Tb.stride;
  for (int t = threadIdx.x; t < n; t += blockDim.x) {
    const unsigned dst = (unsigned)__cvta_generic_to_shared(sm + t);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(Tb.rows + t) : "memory");
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
}

// x >= 0 in units of 2^-55, truncated; `big` collects x >= 128, infinities and NaN
__device__ __forceinline__ long long tab_fixed(double x, int& big) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const int e = (int)(b >> 52);  // biased exponent (x >= 0)
  big |= e >= 1023 + 7;  // two of them add up to less than 2^63
  const unsigned long long m = (b << 11) | 0x8000000000000000ull;
  const int sh = 1023 + 63 - kTabFixedBits - e;
  return (long long)(sh > 63 ? 0ull : m >> (sh < 1 ? 1 : sh));
}

// Row of w and the offset from the row's centre; `low` collects w below the
// first row, and below zero (a node that falls on a site to rounding).  The
// index is clamped, so every access stays inside the table whatever w is.
// GRADED: the row width changes with w (float-float tables); LOWS: w may lie below
// the rows of the common width (a few instructions that every node would pay).
template <bool GRADED, bool LOWS>
__device__ __forceinline__ const uint4* tab_row(const RadialTab& Tb, const uint4* sm, long long w, float& th, float& tl,
                                                int& low) {
  const unsigned hi = (unsigned)((unsigned long long)w >> 32), lo = (unsigned)w;
  int sh = Tb.shift, first = Tb.first;
  if constexpr (GRADED) {
    if (hi >= Tb.near_hi) {
      sh -= kTabNarrow;
      first = Tb.first_near;
    }
    if (LOWS && hi < Tb.main_hi) {
      constexpr int kOne = kTabFixedBits - 32;  // the bit of w = 1
      const int o = min(max(31 - __clz((int)hi), kOne - 3), kOne);  // kOne - 2: w in [1/4, 1/2)
      sh = o - 6;
      first = 64 * (o - kOne + 1);
    }
  }
  int k = (int)(hi >> sh) + first;
  low |= k | (int)hi;  // negative below the first row; the high bit of a negative w
  k += hi >= Tb.rs_hi ? 1 : 0;
  if (hi >= Tb.rc_hi) k = Tb.nrow - 1;
  k = (int)min((unsigned)k, (unsigned)(Tb.nrow - 1));
  const unsigned f1 = __funnelshift_r(lo, hi, sh + 9) & 0x7fffffu;
  const unsigned f2 = (lo >> (sh - 14)) & 0x7fffffu;
  th = __uint_as_float(0x3f800000u | f1) - 1.5f;
  // the next 23 bits, at the middle of what they truncate
  tl = fmaf(__uint_as_float(0x3f800000u | f2), 0x1p-23f, -0x1p-23f * (1.0f - 0x1p-24f));
  return sm + k * Tb.stride;
}

// tau c1 + ... + tau^7 c7 as a float pair (the row without its constant term)
__device__ __forceinline__ ff tab_poly64(float c1h, float c1l, uint4 b, uint4 c, float th, float tl) {
  float e = fmaf(__uint_as_float(c.w), th, __uint_as_float(c.z));
  e = fmaf(e, th, __uint_as_float(c.y));
  e = fmaf(e, th, __uint_as_float(c.x));
  ff s = fast_two_sum(__uint_as_float(b.z), e * th);
  s.lo += __uint_as_float(b.w);
  auto times_tau = [&](ff v) {
    ff m = two_prod(v.hi, th);
    m.lo = fmaf(v.lo, th, fmaf(v.hi, tl, m.lo));
    return m;
  };
  ff m = times_tau(s);
  s = two_sum(__uint_as_float(b.x), m.hi);
  s.lo += m.lo + __uint_as_float(b.y);
  m = times_tau(s);
  s = two_sum(c1h, m.hi);
  s.lo += m.lo + c1l;
  return times_tau(s);
}

// the float-float quality row: tau c1 + ... + tau^5 c5; the low part of c2 and
// c5 need 8 bits and share a word
__device__ __forceinline__ ff tab_polyff(float c1h, float c1l, uint4 b, float th, float tl) {
  float e = fmaf(__uint_as_float(b.y << 16), th, __uint_as_float(b.w));
  e = fmaf(e, th, __uint_as_float(b.z)) * th;
  auto times_tau = [&](ff v) {
    ff m = two_prod(v.hi, th);
    m.lo = fmaf(v.lo, th, fmaf(v.hi, tl, m.lo));
    return m;
  };
  ff s = two_sum(__uint_as_float(b.x), e);
  s.lo += __uint_as_float(b.y & 0xffff0000u);
  const ff m = times_tau(s);
  s = two_sum(c1h, m.hi);
  s.lo += m.lo + c1l;
  return times_tau(s);
}

// v 2^e to the nearest double (ties to even), on bits (no FP64 instruction); the result is
// zero or normal, which the callers' ranges of e ensure
__device__ __forceinline__ double fixed_double(long long v, int e) {
  const unsigned long long u = (unsigned long long)(v < 0 ? -v : v);
  const int lz = __clzll((long long)u);
  const unsigned long long m = u << (lz & 63);  // bit 63 set; below, its leading bit adds one to the exponent
  const unsigned lo = (unsigned)m;
  const unsigned long long b = (m >> 11) + ((lo & 0x7ffu) + ((lo >> 11) & 1u) > 0x400u ? 1ull : 0ull) +
                               ((unsigned long long)(unsigned)(e + 1085 - lz) << 52);
  return u == 0 ? 0.0 : __longlong_as_double((long long)(b | ((unsigned long long)v & 0x8000000000000000ull)));
}
__device__ __forceinline__ float exp2f_bits(int e) { return __uint_as_float((unsigned)(e + 127) << 23); }  // |e| < 127

// v >> n, all sign bits from n = 64 on (PTX clamps the count)
__device__ __forceinline__ long long shift_right(long long v, int n) {
  long long r;
  asm("shr.s64 %0, %1, %2;" : "=l"(r) : "l"(v), "r"(n));
  return r;
}

// running sum of float pairs without renormalisation
__device__ __forceinline__ void tab_acc(ff& a, ff v) {
  const ff s = two_sum(a.hi, v.hi);
  a.hi = s.hi;
  a.lo += s.lo + v.lo;
}

}  // namespace mxe
