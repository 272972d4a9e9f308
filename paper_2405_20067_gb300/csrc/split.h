// split.h -- how many CTAs share a tile's candidates in the backward.
//
// An entry's record depends on its own Gaussian and the tile's queries alone,
// so a tile's candidates may be split over CTAs (grid y) without changing a
// bit.  The kernels take the candidates in steps (a chunk of 128 on the tensor
// cores, 256 per pass of the FP32 form); a part costs its tile's setup and its
// steps, and T tiles in S parts run in ceil(T S / SMs) waves:
//
//   cost(S) = ceil(T S / SMs) (setup + ceil(steps / S))
//
// with the setup in steps.  Lists of a step or two are therefore never split
// where that adds a wave: a part would be mostly setup.  The FP32 form keeps
// several CTAs on an SM; over many waves its longer and shorter parts mix, and
// the part counts as steps / S.
#pragma once

#ifdef __CUDACC__
#define NDG_SPLIT_FN __host__ __device__ inline
#else
#define NDG_SPLIT_FN inline
#endif

namespace ndg {

// Costs are in 1/840 of a step, which every count up to 8 divides.
constexpr int kMaxParts = 8;
constexpr unsigned kStep = 840;

struct SplitCost {
  int step;        // candidates per step
  unsigned setup;  // a part's setup
  unsigned lone;   // a part's time when every SM has at most one, against its
                   // share of a full SM, in tenths
  unsigned mix;    // waves from which parts of uneven length mix
};

// Measured at N = 1..12, tiles of 32 to 256 queries, 8 to 1,400 tiles with 64
// to 4,000 candidates each, every part count from 1 to 8:
//   * tensor cores (one CTA per SM): setup of three steps in the E Psi form
//     and of one and a quarter in the beta form; the choice is at most 1%
//     slower than one part anywhere and within 0.1% of the best count on
//     average.  N = 6: 256 tiles of 600 candidates 43 us in one part (86 in
//     four), 40 tiles of 4,000 78 us in one and 37 in three; N = 10: 64 tiles
//     of 4,000 176 us in one and 93 in two.
//   * FP32: a tenth of a step; a CTA alone on its SM takes about 1.3 times its
//     share of a full one (several hide one another's latency), so that
//     splitting pays before every SM is full.  From N = 11 on, registers spill
//     and co-resident CTAs slow one another down (N = 12: 64 candidates a
//     tile, 180 us with one CTA on each SM and 506 with two), which a lone
//     CTA's smaller share expresses.  Never slower than one part, within 2% of
//     the best count on average.  N = 3: 300 tiles of 4,000 candidates 334 us
//     in one part (414 in three), N = 6: 200 tiles of 1,200 244 us in one and
//     166 in five.
constexpr SplitCost kSplitPsi{128, 3 * kStep, 10, ~0u};
constexpr SplitCost kSplitBeta{128, kStep + kStep / 4, 10, ~0u};
NDG_SPLIT_FN constexpr SplitCost split_fp32(int N) {
  return SplitCost{256, kStep / 10, N <= 10 ? 13u : N == 11 ? 10u : 7u, 8};
}

// The cheapest count of parts, 1 .. max_parts, for T tiles of `steps` steps
// (T <= 2^20, steps <= 2^20); of equal ones the smallest, or the largest
// (ties_up).
NDG_SPLIT_FN int split_parts(unsigned T, unsigned steps, unsigned max_parts, unsigned sms,
                             SplitCost k, bool ties_up) {
  unsigned best = 1;
  unsigned long long cost = ~0ull;
#ifdef __CUDACC__
#pragma unroll 1
#endif
  for (unsigned S = 1; S <= max_parts && (S == 1 || S <= steps); ++S) {
    const unsigned waves = (T * S + sms - 1) / sms;
    const unsigned part = waves >= k.mix ? steps * kStep / S : (steps + S - 1) / S * kStep;
    const unsigned long long c = (unsigned long long)waves * (k.setup + part) * (waves > 1 ? 10 : k.lone);
    if (c < cost || (ties_up && c == cost)) {
      cost = c;
      best = S;
    }
  }
  return (int)best;
}

// Parts of the launch (grid y), from the average list that the capacity
// allows.  Tensor cores: a tile then takes what its own list asks for, at most
// as many, and the other CTAs leave at once (0.9 us per 152 of them).  In the
// FP32 form such CTAs unbalance the SMs (N = 3, 304 tiles of 4,000: 567 us
// against 334), so that it takes the launch's count, and of equal counts the
// smallest; a capacity of three to four times the lists, where these are a step
// or two long, measured up to 1.3 to 1.5 times one part's time (twice the
// lists: 1.2).
constexpr long long kMaxSteps = 1 << 20;
inline int launch_parts(long long T, long long E_cap, int sms, SplitCost k, bool ties_up) {
  if (T <= 0 || T > (1 << 20) || sms <= 0) return 1;
  const long long len = (E_cap + T - 1) / T, steps = (len + k.step - 1) / k.step;
  return split_parts((unsigned)T, (unsigned)(steps < kMaxSteps ? steps : kMaxSteps), kMaxParts,
                     (unsigned)sms, k, ties_up);
}

}  // namespace ndg
