// accum.cuh -- per-site sums of the gathers and full-list passes: FP64 (AccD),
// float-float of float terms (AccFF) or of float pairs (AccF2), three floats
// (AccT).  team_reduce sums over teams of nl consecutive lanes by butterfly.
#pragma once

#include "ff.cuh"

namespace mxe {

struct AccD {
  double v;
  __device__ __forceinline__ void zero() { v = 0.0; }
  __device__ __forceinline__ void add(double x) { v += x; }
  __device__ __forceinline__ void add(float x) { v += (double)x; }
  __device__ __forceinline__ void add(ff x) { v += ff_to_double(x); }
  __device__ __forceinline__ double get() const { return v; }
  __device__ __forceinline__ float2 get_pair() const {
    const float h = (float)v;
    return make_float2(h, (float)(v - (double)h));
  }
  __device__ __forceinline__ void team_reduce(int nl) {
    for (int o = nl >> 1; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  }
};

// Unevaluated sum hi + lo of floats; TwoSum (Knuth) keeps the rounding error
// of every addition, so the pair carries about twice the float significand.
struct AccFF {
  float hi, lo;
  __device__ __forceinline__ void zero() { hi = 0.f; lo = 0.f; }
  __device__ __forceinline__ void add(float x) {
    float s = hi + x;
    float bp = s - hi;
    float err = (hi - (s - bp)) + (x - bp);
    hi = s;
    lo += err;
  }
  __device__ __forceinline__ double get() const { return (double)hi + (double)lo; }
  __device__ __forceinline__ float2 get_pair() const { return make_float2(hi, lo); }
  __device__ __forceinline__ void team_reduce(int nl) {
    for (int o = nl >> 1; o > 0; o >>= 1) {
      float oh = __shfl_xor_sync(0xffffffffu, hi, o);
      float ol = __shfl_xor_sync(0xffffffffu, lo, o);
      add(oh);
      lo += ol;
    }
  }
};

// Unevaluated sum of three floats (TwoSum cascade, about 70 bits): the
// per-site sums of the mixed mode's gathers, at least as exact as an FP64 sum.
// A conversion and an FP64 addition per value cost 128 FP32 issue slots on
// GB300 (2 FP64 lanes per SM) and kept the gathers on the FP64 pipe; this takes
// 13 (float) or 20 (float pair).
struct AccT {
  float h, m, l;
  __device__ __forceinline__ void zero() { h = m = l = 0.f; }
  __device__ __forceinline__ void add(float x) {
    const ff s = two_sum(h, x), t = two_sum(m, s.lo);
    h = s.hi;
    m = t.hi;
    l += t.lo;
  }
  __device__ __forceinline__ void add(ff x) {
    const ff s = two_sum(h, x.hi), t = two_sum(m, s.lo), u = two_sum(t.hi, x.lo);
    h = s.hi;
    m = u.hi;
    l += t.lo + u.lo;
  }
  __device__ __forceinline__ double get() const { return (double)h + ((double)m + (double)l); }
  __device__ __forceinline__ float2 get_pair() const {
    const ff s = two_sum(h, m);
    const ff t = fast_two_sum(s.hi, s.lo + l);
    return make_float2(t.hi, t.lo);
  }
  __device__ __forceinline__ void team_reduce(int nl) {
    for (int o = nl >> 1; o > 0; o >>= 1) {
      const float oh = __shfl_xor_sync(0xffffffffu, h, o), om = __shfl_xor_sync(0xffffffffu, m, o),
                  ol = __shfl_xor_sync(0xffffffffu, l, o);
      add(ff{oh, om});
      l += ol;
    }
  }
};

// A sum of float pairs kept as one float pair (the float-float mode's accurate
// gathers).
struct AccF2 {
  ff v;
  __device__ __forceinline__ void zero() { v = ff(0.f, 0.f); }
  __device__ __forceinline__ void add(ff x) { v = v + x; }
  __device__ __forceinline__ double get() const { return ff_to_double(v); }
  __device__ __forceinline__ void team_reduce(int nl) {
    for (int o = nl >> 1; o > 0; o >>= 1) {
      const ff w(__shfl_xor_sync(0xffffffffu, v.hi, o), __shfl_xor_sync(0xffffffffu, v.lo, o));
      v = v + w;
    }
  }
};

}  // namespace mxe
