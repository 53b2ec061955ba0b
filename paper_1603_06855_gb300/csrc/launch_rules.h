// Rules that choose between launch forms, in plain C++ (also compiled for the host alone, to be checked).
#pragma once

// CTAs of a cluster that shares one FP64 projected problem (small_rr64.cu).
constexpr int kRr64Cluster = 8;

// Whether each of nk FP64 projected problems (n basis columns, m wanted) gets a cluster.  The cluster shares the
// four products of the FP32 stage's correction (n > m) and its CTAs take a whole SM each, so it pays while
// there is an SM for every CTA, counting the `others` problems that calls running beside this one solve.
// Solves of 12 bands at N = 125, 4 k-points each, by clusters or one CTA a problem: one design 37.4 and 41.4 ms, two
// 41.2 and 43.3, four 52.2 and 53.2 (128 CTAs), eight 79 and 61, sixteen 148 and 110; two of 12 k-points 62 and 57;
// sixteen of 14 k-points, 6 bands at N = 27, 112 and 43.
inline bool rr64_uses_clusters(int n, int m, long long nk, long long others, int sms) {
  return n > m && kRr64Cluster * (nk + others) <= sms;
}

// Projected problems of one launch: larger sets take several launches over the same scratch (0.66 MB a problem in the
// mixed form, 1.58 MB in FP64, at the widest blocks), which would else be the largest array of a set of many k-points:
// 103 GB of 239 for 65535 k-points of the FP64 form at N = 27, 3.8 GB now.  Each problem has an SM to itself and a
// launch ends with its slowest, so sixteen per SM: with four, solves of 700 and 1300 k-points (FP64, 20 bands)
// were 4 and 5.5 % slower.
inline int rr_problems_per_launch(long long nk, int sms) { return (int)(nk < 16LL * sms ? nk : 16LL * sms); }

// Chunks of the adjoint's (k, band) pairs, each summed in FP32 before FP64 adds the sums up: the `wave` chunks that the
// chip holds at once, or a whole multiple, so that a sum runs over at most 128 pairs while there is room for all
// (`most` sums a voxel; 128 most / 2 pairs and more may take longer ones).  A wave follows the chip and the cell: from some 72^3
// voxels on it is one chunk, which alone would be one sum over 2000 pairs of a hundred k-points and 20 bands.
inline int adj_chunks(int pairs, int wave, int most) {
  const int want = (int)((pairs + 128LL * wave - 1) / (128LL * wave)), room = most / wave;
  return wave * (want < room ? want : (room > 1 ? room : 1));
}
