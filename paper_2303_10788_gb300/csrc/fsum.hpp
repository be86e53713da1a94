// Sums of FP32 values carried in three FP32 parts: at least the 53 bits of a
// double, at FP32 rates (13 additions a value; the FP64 units of sm_103a add a
// 64th as many values per clock).
#pragma once

#ifdef __CUDACC__
#define CCS_FSUM_FN __host__ __device__ __forceinline__
#else
#define CCS_FSUM_FN inline
#endif

namespace ccs {

// a + b exactly, as the rounded sum (returned) and what it lost (Knuth's TwoSum).
CCS_FSUM_FN float two_sum(float a, float b, float& lost) {
  const float t = a + b, bb = t - a;
  lost = (a - (t - bb)) + (b - bb);
  return t;
}

// s: the rounded sum; c: what s lost, rounded; e: what c lost.  Only e's own
// additions round: 2^-24 of values 2^-48 of the sum.
struct Sum3 {
  float s = 0.f, c = 0.f, e = 0.f;
  CCS_FSUM_FN void add(float v) {
    float l;
    s = two_sum(s, v, l);
    c = two_sum(c, l, l);
    e += l;
  }
  CCS_FSUM_FN void add(const Sum3& o) {
    add(o.s);
    float l;
    c = two_sum(c, o.c, l);
    e += l + o.e;
  }
  CCS_FSUM_FN double value() const { return ((double)s + (double)c) + (double)e; }
};

}  // namespace ccs
