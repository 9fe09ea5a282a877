// How many CTAs of a thread-block cluster hold one 1d instance of n = 2^L (L = 8 .. 14, the split
// kernels of sgn_split_1d.cuh): what each kernel can run on, and the choice for a layout.  Host
// code, no CUDA.
#pragma once

namespace sgn {

#ifdef __CUDACC__
#define SGN_PLAN_FN __host__ __device__ constexpr
#else
#define SGN_PLAN_FN constexpr
#endif

constexpr int kSplitMinLog = 8, kSplitMaxLog = 14, kSplitClasses = 16;

// log2 of a thread's elements: float64 2 up to n = 1024 and 4 above, mixed 4
SGN_PLAN_FN int split_log_e(int L, bool mixed) { return mixed || L > 10 ? 2 : 1; }
// n = N1 x N2: N1 = 64 from n = 2048 (N1 / 2 >= 8 CTAs' rows and N2 / CL >= 8 columns), 32 and
// 16 below
SGN_PLAN_FN int split_log_n1(int L) { return L >= 11 ? 6 : (L >= 9 ? 5 : 4); }
// Fewest CTAs: a CTA has at most 256 threads (512 for float64 and mixed at n = 16384), which
// leaves 128 registers for each: 1024 points, 512 in float64 up to n = 1024, 2048 at n = 16384.
SGN_PLAN_FN int split_min_lcl(int L, int log_e) {
  const int l = L - log_e - 8;
  return l < 0 ? 0 : (l > 3 ? 3 : l);
}
// Most CTAs, 8: a CTA keeps 32 threads, 8 columns and a pair of rows.
SGN_PLAN_FN int split_max_lcl(int L, int log_e) {
  const int a = L - split_log_n1(L) - 3, b = L - log_e - 5, m = a < b ? a : b;
  return m < 3 ? m : 3;
}

// log2 of the CTAs per instance of every class: num[c] instances of n = 2^c (class 0: other sizes),
// ctas[c] > 1 where another kernel runs them on that many CTAs each.  A class starts on the
// fewest CTAs that its kernel runs on; the classes are then halved, the one with the largest
// share per CTA first, while every CTA of the launch has an SM of its own.  Splitting further
// would only add exchanges: two CTAs on an SM share its issue slots and its float64 pipe.
// Batches of 23 to 39 instances of 512 .. 8192, 2 RK4 steps, against a count that began below
// the kernels' minima (and so split on SMs already taken, or left some idle): float64 5.42 ->
// 5.35, 6.56 -> 5.83 and 6.90 -> 5.86 ms, at worst 5.79 -> 5.87; mixed 1.79 -> 1.76, at worst
// 1.65 -> 1.74 ms.  One instance and the batches from 48 up have the same plan either way.
inline void split_plan(const int* num, const int* ctas, bool mixed, int sms, int* lcl) {
  long long total = 0;
  auto split = [&](int c) { return c >= kSplitMinLog && c <= kSplitMaxLog && ctas[c] < 2; };
  for (int c = 0; c < kSplitClasses; ++c) {
    lcl[c] = split(c) ? split_min_lcl(c, split_log_e(c, mixed)) : 0;
    total += ctas[c] > 1 ? (long long)num[c] * ctas[c] : (long long)num[c] << lcl[c];
  }
  for (;;) {
    int best = -1;
    for (int c = kSplitMinLog; c <= kSplitMaxLog; ++c)
      if (num[c] > 0 && split(c) && lcl[c] < split_max_lcl(c, split_log_e(c, mixed)) &&
          (best < 0 || c - lcl[c] >= best - lcl[best]))
        best = c;
    if (best < 0 || total + ((long long)num[best] << lcl[best]) > sms) return;
    total += (long long)num[best] << lcl[best];
    lcl[best] += 1;
  }
}

}  // namespace sgn
