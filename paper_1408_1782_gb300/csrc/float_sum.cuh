// Sums of many FP32 values, no less accurate than FP64 additions, on the FP32 pipe: an unevaluated sum of
// three floats, each addition passing its rounding error (exact, the TwoSum of Knuth) to the next.  A GB300 SM
// has 128 FP32 lanes and two FP64 lanes per clock, so converting and adding every value in FP64 takes several
// times the loads' time.
//
// Error of a run of m <= kRun values: below (2 m u)^3 of the sum of their magnitudes, u = 2^-24 (the two
// cascaded error-free additions of Ogita, Rump and Oishi's Sum3), and the three floats are added in FP64: for
// m = kRun 2^-51, against m 2^-53 for FP64 additions one by one; up to m = 256, which merged sums may reach, it
// is no larger than that.  A pair of floats (one TwoSum) is not enough:
// its (2 m u)^2 is 2^-34, and sums of 1,024 values of mixed magnitudes are 1e-13 off where FP64 is 5e-16 off.
#pragma once

#if defined(__CUDACC__)
#define QBE_SUM_FN __host__ __device__ __forceinline__
#else
#define QBE_SUM_FN inline
#endif

namespace qbe {

struct FloatSum {
  static constexpr int kRun = 64;      // values after which value() is to be taken
  static constexpr int kMerged = 256;  // values of merged sums
  float hi = 0.f, mid = 0.f, lo = 0.f;
  QBE_SUM_FN static float two_sum(float a, float b, float& err) {
    const float t = a + b, z = t - a;
    err = (a - (t - z)) + (b - z);
    return t;
  }
  QBE_SUM_FN void add(float x) {
    float e, f;
    hi = two_sum(hi, x, e);
    mid = two_sum(mid, e, f);
    lo += f;
  }
  QBE_SUM_FN void merge(float h, float m, float l) {   // the sum h + m + l of another
    float e;
    add(h);
    mid = two_sum(mid, m, e);
    lo += e + l;
  }
  // (an infinity among the values leaves NaN in the errors)
  QBE_SUM_FN double value() const { return hi - hi == 0.f ? (double)hi + ((double)mid + (double)lo) : (double)hi; }
};

}  // namespace qbe
