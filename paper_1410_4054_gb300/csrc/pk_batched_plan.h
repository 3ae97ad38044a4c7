// Which clusters the batched solver's cluster engine gives a batch: plain host code, so that its rules can be
// tried without a GPU against a device that lacks some cluster sizes.
//
// A class is (CTA shape, log2 of the cluster size): shape * kClSizes + c.  Shape 0 holds the most rows per CTA.
// Limits (a template parameter) says what the device can run:
//   int shapes() const;            CTA shapes
//   int max_rows(int shape) const; rows a CTA holds
//   int capacity(int shape, int C) const;  clusters of C CTAs at once, 0: not usable
#pragma once

#include <algorithm>

namespace pk {

constexpr int kClSizes = 5;  // clusters of 1, 2, 4, 8, 16 CTAs

// log2 of the largest cluster of `shape` that the device can run, -1: none.
template <class Limits>
int largest_cluster(const Limits& d, int shape) {
  int c = kClSizes - 1;
  while (c >= 0 && d.capacity(shape, 1 << c) <= 0) --c;
  return c;
}

// What the automatic choice plans: CTAs of shape 0 (512 threads, two per SM) with up to t rows each,
// half as many for a system of at most 2 t rows; shape 0's log2 of the cluster size, at most `most` (the
// CTAs then take more than t rows).
inline int auto_cluster(int n, int t, int most) {
  const int rows = n <= 2 * t ? t / 2 : t;
  int c = 0;
  while (c < most && ((long long)rows << c) < n) ++c;
  return c;
}

// Class of a system of n rows when the batch aims at rows_cta rows per CTA: the CTA shape
// whose row limit is rows_cta, else the next larger one that holds n on 16 CTAs, with the
// smallest power-of-2 cluster that holds n; or -1.
template <class Limits>
int fixed_cluster(const Limits& d, int n, int rows_cta) {
  int s0 = -1;
  for (int sh = 0; sh < d.shapes(); ++sh)
    if (d.max_rows(sh) == rows_cta) s0 = sh;
  for (int sh = s0; sh >= 0; --sh) {
    const long long mx = d.max_rows(sh);
    for (int c = 0; c < kClSizes; ++c)
      if (mx << c >= n) return sh * kClSizes + c;
  }
  return -1;
}

// cls[k]: the class of system k of n[k] rows.  false: the device cannot run what that needs.
// rows_cta 0: the automatic choice.  An SM takes two CTAs of shape 0, so that one system's reductions
// and barriers overlap another's FP64 work; t, the rows per CTA, is the largest the CTAs hold as long
// as the batch fills the device (fewer barriers per row), else smaller (an iteration's latency).
// The short systems at the end of the queues run on shares half as large: their iterations are the
// batch's tail.  Measured (512 shifted 2D Laplacians, ms): 256 threads x 2048 rows, two per SM 13.5, this
// 10.9.  With t everywhere / halved up to t / 2 t / 4 t rows (rectangles, sides log-uniform): 512 of 32-256
// 9.6 / 9.6 / 9.0 / 9.5, another 512 8.9 / 8.2 / 8.2 / 8.7, 200 of them 4.3 / 4.3 / 3.6 / 3.8, 60 of them 2.4 in
// all, 300 of 100-250 12.0 / 12.1 / 12.1 / 11.8, 400 of 128 x 128 10.1 / 10.1 / 10.1 / 10.4; only short systems
// lose by it: 1,000 of 20-90 3.2 / 3.5 / 3.7 / 3.6, 2,000 of 16-64 3.7 / 3.8 / 3.8 / 3.8.
template <class Limits>
bool cluster_classes(const Limits& d, const int* n, int nsys, int rows_cta, int* cls) {
  int t = d.max_rows(0);
  const int most = rows_cta == 0 ? largest_cluster(d, 0) : 0;
  const int device_ctas = rows_cta == 0 ? d.capacity(0, 1) : 0;
  while (rows_cta == 0 && t > 512) {
    long long ctas = 0;
    for (int k = 0; k < nsys; ++k) ctas += 1ll << auto_cluster(n[k], t, most);
    if (ctas >= device_ctas) break;
    t /= 2;
  }
  for (int k = 0; k < nsys; ++k) {
    int c = -1;
    if (rows_cta) c = fixed_cluster(d, std::max(n[k], 1), rows_cta);
    else if (most >= 0 && ((long long)d.max_rows(0) << most) >= n[k]) c = auto_cluster(n[k], t, most);
    if (c < 0 || d.capacity(c / kClSizes, 1 << (c % kClSizes)) <= 0) return false;
    cls[k] = c;
  }
  return true;
}

// The rows per CTA to run with: `wanted` (0: automatic), else `fixed`, else -1 (no clusters).  cls: the plan.
template <class Limits>
int choose_clusters(const Limits& d, const int* n, int nsys, int wanted, int fixed, int* cls) {
  if (cluster_classes(d, n, nsys, wanted, cls)) return wanted;
  if (wanted != fixed && cluster_classes(d, n, nsys, fixed, cls)) return fixed;
  return -1;
}

}  // namespace pk
