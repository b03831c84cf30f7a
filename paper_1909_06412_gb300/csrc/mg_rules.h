// Host rules of the dispatch that need no device: which variant serves a call,
// from sizes and counts alone.
#pragma once
#include <stdint.h>

namespace mgk {

// The kernel that runs two CTAs per SM (where the shared memory of two fits)
// pays from four problems per team on: with fewer the longest problem decides,
// and each team is slower with half the registers.  Measured on uneven 2D and 3D
// batches, FP32, one CTA per SM against two at p problems per team: teams of two
// CTAs p = 2.0 0.85x, 2.6 0.87x, 3.2 0.96x, 3.7 0.99x, 4.2 1.25x, 4.7 1.45x, 6.0
// 1.37x (only 3D grids 2.0 0.96x, 3.2 1.40x, 4.2 1.54x); teams of one 2.0 0.85x,
// 3.0 0.91x, 3.9 1.01x, 5.0 1.22x; of four 2.6 0.87x, 3.9 1.14x, 5.3 1.54x.  In
// FP64 the shared memory of two fits for few batches (368 problems of one: 1.06x).
constexpr int BATCH_TWO_CTAS = 4;

// Whether the two-CTA kernel is worth asking for, with `teams1` teams of the
// one-CTA kernel.
inline bool batch_wants_two(int nprob, int teams1) { return nprob > BATCH_TWO_CTAS * teams1; }

// CTAs per SM of the batched kernel: `teams2` teams could run of the two-CTA
// kernel (0: none, or the question failed).
inline int batch_ctas(int nprob, int teams1, int teams2) {
  return batch_wants_two(nprob, teams1) && teams2 > teams1 ? 2 : 1;
}

// Whether the general kernel's FP64 passes run on the integer units
// (mg_pass64.cuh).  They have the higher throughput and the longer latency for a
// few points; a grid of more axes has more passes with less work in each.  FP64
// units against integer units, yoshida4 calls, by points per SM: two axes 431
// 0.89x, 1035 1.26-1.29x, 1091 1.14-1.15x, 1724 1.27x; three 216 0.80x, 1035
// 1.13-1.16x, 1091 1.03-1.05x, 13,800 1.36x; four 1227 0.98x, 1381 1.04-1.06x,
// 2182 1.05x, 11,050 1.23x; five 1091 0.93x, 2182 1.01x, 2910 0.99x, 12,431
// 1.05x; axes of 12.8 points on average and six of them 29,466 1.09x, but of 8.7
// (six) 2910 0.98x, of 7.7 (seven) 10,347 0.97x, of 6.9 (eight) 34,923 0.90x.
inline bool integer_passes(int D, int64_t npts, int sms) {
  const int64_t per_sm = D <= 3 ? 1024 : 1024 * (int64_t)D / 3;
  if (npts < per_sm * sms) return false;
  int64_t n9 = 1;
  for (int l = 0; l < D; ++l) n9 *= 9;
  return D <= 3 || npts >= n9;  // nine points an axis on average
}

// Cost of the passes of the FP64 short-axis kernel over one group of g axes, for
// `nchunks` chunks of `lines` lines on `sms` SMs, in thousands of cycles.  A pass
// is bound by latency, not by throughput: measured, a warp takes about 4000
// cycles for its lines of one axis whether it shares its scheduler with none or
// two others, a chunk about 8000 for its copies and waits, and 3000 stand for the
// barrier of a pass.  Chunks are dealt to two teams per SM.
inline double short_pass_cost(int64_t nchunks, int g, int lines, int threads, int sms) {
  const int64_t teams = 2 * (int64_t)sms, waves = (nchunks + teams - 1) / teams;
  const int team = threads / 2, rounds = (lines + team - 1) / team;
  return (double)waves * (4.0 * g * rounds + 8.0) + 3.0;
}

}  // namespace mgk
