// Launch shapes of the substitution over the symmetric tile storage: which one serves a number
// of boxes, widths and right-hand sides best.  Plain host code (hd_subst_sym.cu launches it).
#pragma once

#include <algorithm>
#include <cstdint>

namespace hd {

// K CTAs per box and group of NR right-hand sides (a cluster), P sets of SW warps in a CTA, made
// so that PER_SM of them share an SM.
struct SymPick {
  int K, P, SW, NR, per_sm;
};

// Complex FP32 arithmetic.  Boxes up to 96 wide: with more CTAs than SMs the small form, three
// warps and a producer, four CTAs to an SM; a step of so few tiles is a chain of latencies that
// one CTA cannot fill an SM with.  Measured per application of one source, ms, one large CTA / small
// ones: 1024 boxes of 32 0.458 / 0.152, of 64 1.02 / 0.50, of 96 1.75 / 1.31; 144 boxes of 64 0.162 /
// 0.195.  (At 112 wide a form of four warps, three to an SM: 2.29 / 2.22.)
constexpr int SYM_NARROW = 96;
// Complex FP64: up to 80 wide, with more than two CTAs per SM (up to 48, more than one); wider boxes
// keep the FP64 pipe busy with two large CTAs.  400 boxes of 48 1.50 / 0.95 ms, of 80 5.28 / 3.92;
// 256 of 64 1.48 / 1.61; 800 of 96 12.9 / 15.2.
constexpr int SYM_NARROW64 = 80;

inline int64_t sym_waves(int64_t ctas, int64_t at_once) { return (ctas + at_once - 1) / at_once; }

// Complex FP64: one right-hand side per CTA (two shared the reads, which are not the bound, and left SMs
// idle: 2 sources in 64 boxes of 240 40.3 ms, one each 34.1).  K by waves times the length of a step,
// in units of one tile's products (0.6 us): a step takes as long as its tiles, spread over K CTAs at
// 0.58 and 0.33, and not less than one warp's segment of three tiles.  K = 1 / 2 / 4, ms: 36 boxes of
// 112 3.90 / 2.16 / 1.89, 64 boxes 3.92 / 2.17 / 3.77, 100 boxes 3.93 / 4.31 / 5.64, 169 boxes 6.96 /
// 6.43 / 9.38; of 240, 64 boxes 34.1 / 21.0 / 20.8, 100 boxes 34.1 / 41.9 / 31.2, 169 boxes 67.8 / 62.7 / 51.9.
inline SymPick sym_pick64(int m, int64_t nsub, int nrhs, int sms) {
  const int64_t c = nsub * nrhs;
  if (c > (m <= 48 ? 1 : 2) * (int64_t)sms && m <= SYM_NARROW64) return {1, 1, 3, 1, 4};
  const int mt = (m + 15) / 16;
  const double nt = mt * (mt + 1) / 2;
  // four warps, three CTAs to an SM, where that saves a wave: 400 boxes of 112 13.99 -> 10.4 ms
  if (m > SYM_NARROW64 && m <= 112 && c > 2 * (int64_t)sms && 2.9 * sym_waves(c, 3 * (int64_t)sms) < 2 * sym_waves(c, 2 * (int64_t)sms))
    return {1, 1, 4, 1, 3};
  const double t1 = sym_waves(c, sms) * std::max(14.5, nt);
  const double t2 = sym_waves(2 * c, sms) * std::max(14.0, 0.58 * nt);
  const double t4 = sym_waves(4 * c, sms) * std::max(14.0, 0.33 * nt + 0.3);
  if (t4 < t1 && t4 < t2) return {4, 1, 8, 1, 1};
  if (t2 < t1) return {2, 1, 8, 1, 1};
  // more CTAs than SMs: two to an SM, one's sums under the other's products
  return {1, 1, 8, 1, c > sms ? 2 : 1};
}

// Complex FP32 with NR right-hand sides per CTA: enough clusters to give every SM about one CTA.
// Measured per application (one right-hand side; K = 1 / 2 / 4): 16 boxes of 176 708 / 566 / 481 us,
// 64 boxes 718 / 564 / 928 us, 144 boxes 1000 / 1131 / 1877 us, 256 boxes 1815 / 2236 / 3695 us.
// A set has 224 threads, a step one thread per row: wider boxes take two sets.
inline SymPick sym_pick32(int m, int64_t nsub, int nrhs, int sms) {
  int NR = nrhs >= 3 ? 4 : nrhs;
  if (m <= SYM_NARROW) {
    // Right-hand sides per CTA by waves times the length of a step: 1, 1.75 and 3 for 1, 2 and 4 in the small
    // form (four to an SM), about 0.55, 0.75 and 1.25 in the large one (64 wide, 608 small CTAs of one
    // source 0.27 ms).  4 sources in 256 boxes of 64: 1 / 2 / 4 per CTA 0.55 / 0.48 / 0.64 ms.
    const double large[3] = {0.55, 0.75, 1.25}, small[3] = {1.0, 1.75, 3.0};
    double best = 1e300;
    for (int i = nrhs >= 3 ? 2 : nrhs - 1; i >= 0; --i) {
      const int64_t c = nsub * sym_waves(nrhs, 1 << i);
      const double t = c <= sms ? large[i] : sym_waves(c, 4 * (int64_t)sms) * small[i];
      if (t < best) { best = t; NR = 1 << i; }
    }
  }
  const int64_t c = nsub * sym_waves(nrhs, NR);
  if (m <= SYM_NARROW && c > sms) return {1, 1, 3, NR, 4};
  if (4 * c <= sms && m <= 224) return {4, 1, 7, NR, 1};
  return {2 * c <= sms ? 2 : 1, 2, 7, NR, 1};
}

}  // namespace hd
