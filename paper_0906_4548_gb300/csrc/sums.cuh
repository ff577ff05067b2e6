// Sums that a thread carries over the points or modes it visits: in FP64 for FP64 data, for FP32 data
// in three floats (eft.cuh), which lose less than FP64 does and stay off the FP64 pipe that a pass
// with FP64 arithmetic on converted values waits for.  What FP32 cannot hold of a small term is below 2^-148;
// callers scale their data to about one and add in FP64 where the terms are below kSumSmall.
#pragma once

#include "eft.cuh"

namespace dgp {

// 2^-70: with terms of this size the parts lost below 2^-148, of up to 2^17 terms, are below 2^-60 of the sum
constexpr float kSumSmall = 8.470329472543003e-22f;

// Sums of a P(k) shell: sqrt(n2) and |a|^2.  P(k) at 256^3, 128 shells: 232 us a call; with pairs of
// floats, about 48 bits, 205 us; with FP64 sums staged mode by mode 1.78 ms.
template <typename T> struct ShellSum {
  double s = 0.0;
  __device__ __forceinline__ void add_root(int n2, bool twice) {
    const double r = sqrt((double)n2);
    s += twice ? 2.0 * r : r;
  }
  __device__ __forceinline__ void add_norm(double x, double y) { s += x * x + y * y; }
  __device__ __forceinline__ double value() const { return s; }
};
template <> struct ShellSum<float> {
  FP3 s{0.f, 0.f, 0.f};
  __device__ __forceinline__ void add_root(int n2, bool twice) {
    // sqrt(n2) = r + d - d^2 / (2 r) + ..., d = (n2 - r^2) / (2 r): the remainder of a rounded root is exact
    // (n2 < 2^24), and the approximate 1 / (2 r) is made up for in the next term
    const float f = (float)n2, r = sqrtf(f), h = 0.5f * rsqrtf(f), g = twice ? 2.f : 1.f;
    const float rem = fmaf(-r, r, f), d = rem * h;
    const float d2 = (fmaf(-2.f * r, d, rem) - d * d) * h;
    fp3_acc(s, FP{g * r, g * d});
    s.lo += g * d2;
  }
  __device__ __forceinline__ void add_norm(float x, float y) {
    fp3_acc(s, fp_prod(x, x));
    fp3_acc(s, fp_prod(y, y));
  }
  __device__ __forceinline__ double value() const { return fp3_value(s); }
};

// Sums of values and of their inverses.
template <typename T> struct ThreadSum {
  double s = 0.0;
  __device__ __forceinline__ void add(double v) { s += v; }
  __device__ __forceinline__ void add_inverse(double v) { s += 1.0 / v; }
  __device__ __forceinline__ double value() const { return s; }
};
template <> struct ThreadSum<float> {
  FP3 s{0.f, 0.f, 0.f};
  __device__ __forceinline__ void add(float v) { fp3_acc(s, v); }
  __device__ __forceinline__ void add_inverse(float v) {
    // 1 / v = r (1 + t + t^2 + ...), t = 1 - r v exactly, |t| < 2^-23
    const float r = 1.f / v, t = fmaf(-r, v, 1.f);
    const FP p = fp_prod(r, t);
    fp3_acc(s, FP{r, p.hi});
    s.lo += fmaf(r * t, t, p.lo);
  }
  __device__ __forceinline__ double value() const { return fp3_value(s); }
};

// Sums of products of two and of three factors; small(): the products are out of the range where the
// sum is as good as FP64.
template <typename T> struct ProductSum {
  double s = 0.0;
  __device__ __forceinline__ void add(double a, double b) { s += a * b; }
  __device__ __forceinline__ void add(double a, double b, double c) { s += a * b * c; }
  __device__ __forceinline__ bool small() const { return false; }
  __device__ __forceinline__ double value() const { return s; }
};
template <> struct ProductSum<float> {
  FP3 s{0.f, 0.f, 0.f};
  float top = 0.f;  // largest product
  __device__ __forceinline__ void add(float a, float b) {
    const FP p = fp_prod(a, b);
    fp3_acc(s, p);
    top = fmaxf(top, fabsf(p.hi));
  }
  __device__ __forceinline__ void add(float a, float b, float c) {
    const FP p = fp_prod(a, b), q = fp_prod(p.hi, c), r = fp_prod(p.lo, c);
    fp3_acc(s, q);
    fp3_acc_mid(s, r.hi);
    s.lo += r.lo;
    top = fmaxf(top, fabsf(q.hi));
  }
  __device__ __forceinline__ bool small() const { return !(top >= kSumSmall && isfinite(s.hi)); }
  __device__ __forceinline__ double value() const { return fp3_value(s); }
};

}  // namespace dgp
