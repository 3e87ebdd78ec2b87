// Which batches take the CTA-pair FFN kernels (ffn_pair.cu), host side.
#pragma once

#include <initializer_list>

#include "xshare.h"

namespace xs {

// At most this many experts can be selected (budgets add to the warm-up
// sets).  Groups are filled in whole rounds, so that without warm-up sets S
// has m_g G experts; with them the last round may go beyond by G - 1.  (That
// G - 1 at k0 = 0 made the rule see 47 experts where 40 are selected: N = 64, d =
// 7168, F = 1024, G = 8, m_g = 5, B = 32 274.7 -> 286.4 us.)
inline int selected_at_most(int mode, int B, int N, int budget, int k0, int T, int m_r, int G, int m_g) {
  const long long warm = static_cast<long long>(B) * k0;
  long long n = N;
  if (mode == XS_MODE_BATCH) {
    n = warm + budget;
  } else if (mode == XS_MODE_HIER) {
    n = warm + static_cast<long long>(B / T) * m_r + budget;
  } else if (mode == XS_MODE_GROUP) {
    const long long rounds = static_cast<long long>(m_g) * G + (k0 > 0 ? G - 1 : 0);
    n = warm > rounds ? warm : rounds;
  }
  return static_cast<int>(n < N ? n : N);
}

// By T, the pairs per expert that can be selected, and by the time that SMs
// wait because the pair kernels cut no unit (ffn_tc.cu does):
//   - T >= kPairAllTok: always;
//   - T >= kPairMinTok: unless phases of several rounds of units take more
//     than kPairWait K steps (and more than kPairWaitShare of both phases'
//     work) longer than their work spread evenly over the pairs would, or
//     (T < kPairWaitTok) phases of one round more than kPairWaitOne;
//   - T >= kPairFewTok, or T K >= kPairWork (long units hide a unit's fixed
//     costs): if neither phase idles more than kPairIdle of its time in the
//     last round of units, or on the missing half of an odd down block.
// A phase's share of idle time says little from kPairMinTok on (a layer of one
// round of units idles most SMs and still gains, since stream-K pays for its
// cuts); the steps waited do.  Shared experts are left out: with them the pairs
// win at every point measured (T = 8 to 256).
// Layer forward on GB300, plain top-k, ffn_tc.cu | ffn_pair.cu, us, by steps
// waited (gate/up + down; * one round of units):
//   T = 24: N = 8, d = 2048, F = 256 (25* + 1*) 37.5 | 34.2; N = 32, d = 7168,
//   F = 2048 (29 + 7) 424.2 | 414.2; N = 16, d = 2048, F = 2048 (20 + 10) 79.7 |
//   82.2; N = 16, d = 7168, F = 2048 (71 + 3) 226.9 | 229.4; N = 300, d = 640,
//   F = 1920 (8 + 64) 362.7 | 373.1; N = 16, d = 5120, F = 2048 (51 + 25) 168.6 |
//   175.4; N = 16, d = 6144, F = 1408 (66 + 21) 152.5 | 155.8; N = 8, d = 7168,
//   F = 256 (88* + 0) 66.0 | 64.3; N = 4, d = 7168, F = 256 (100* + 2) 55.8 | 58.6
//   T = 32: N = 16, d = 5120, F = 2048 174.2 | 178.7; N = 4, d = 7168, F = 256
//   68.0 | 61.5; N = 8, d = 7168, F = 256 75.9 | 64.7
//   T = 48: N = 16, d = 5120, F = 2048 181.6 | 180.3; N = 16, d = 6144, F = 1408
//   165.8 | 159.1; N = 300, d = 640, F = 1920 406.6 | 413.6; T = 64: 504.2 | 479.2
//   a small share of the work: d = 7168, F = 2048, 40 experts, T = 25.6 (65 + 8,
//   5.2 %) 552.7 | 542.5; 64 experts, T = 32 (59 + 14, 3.2 %) 874.3 | 859.4
// Below T = 24, by the share of idle time:
//   N = 64, d = 2048, F = 1024 (3.9 %): T = 8 142.1 | 143.5, 12.5 144.4 | 141.1
//   N = 128, d = 2048, F = 768 (8.9 %): T = 8 201.4 | 203.1, 16 208.1 | 211.4
//   N = 16, d = 5120, F = 2048 (18.7 %): T = 19 171.2 | 176.0
//   N = 300, d = 640, F = 1920 (21 % in the down phase): T = 15 361.9 | 367.3
//   N = 256, d = 7168, F = 2048, budget 24, k0 = 1: B = 32 (T = 4.6) 552 | 561,
//   B = 64 (5.8) 739 | 727, B = 96 (6.4) 858 | 838, B = 128 (6.7) 950 | 938;
//   groups, B = 256 (8) 772 | 763, B = 32 (5.4) 557 | 565
constexpr int kPairAllTok = 48;
constexpr int kPairMinTok = 24;
constexpr double kPairWait = 70.0;
constexpr double kPairWaitShare = 0.055;
constexpr int kPairWaitTok = 32;
constexpr double kPairWaitOne = 95.0;
constexpr int kPairFewTok = 12;
constexpr int kPairWork = 650 * 64;
constexpr double kPairIdle = 0.045;

// `pairs` routed pairs over at most `experts` experts, `here` of them on this
// GPU, which for a rank's share of a selection is a guess (`sure` false): below
// kPairMinTok a rank then stays on ffn_tc.cu, since what pairs gain there is
// less than a round that the guess misses (N = 256, d = 7168, F = 2048, groups,
// B = 256, a rank of eight with 32 of the 256 experts that the bound allows and
// about 8 used: 326.5 | 336.8 us; plain top-k, B = 512, all 32 used: 493 | 467).
// P CTA pairs run at once (0: the kernels cannot run).
inline bool pair_rule(long long pairs, int experts, int here, bool sure, int P, int d, int F) {
  if (P <= 0 || experts <= 0) return false;
  auto tokens = [&](int t) { return pairs >= static_cast<long long>(t) * experts; };
  if (tokens(kPairAllTok)) return true;
  // A phase: `units` whole units per expert, `blocks` of them counted exactly,
  // of `steps` K steps.
  struct Phase {
    long long rounds;
    double even;      // rounds, if the work were spread evenly
    double steps;
    double waited() const { return (static_cast<double>(rounds) - even) * steps; }
    bool idles() const { return static_cast<double>(rounds) > even * (1.0 + kPairIdle); }
  };
  auto phase = [&](int units, double blocks, int K) {
    return Phase{(static_cast<long long>(here) * units + P - 1) / P, here * blocks / P, K / 64.0};
  };
  const Phase gate_up = phase(F / 128, F / 128.0, d), down = phase((d + 255) / 256, d / 256.0, F);
  if (tokens(kPairMinTok)) {
    double several = 0.0, one = 0.0;
    for (const Phase *p : {&gate_up, &down}) (p->rounds > 1 ? several : one) += p->waited();
    const double share = kPairWaitShare * (gate_up.even * gate_up.steps + down.even * down.steps);
    return several <= (share > kPairWait ? share : kPairWait) && (tokens(kPairWaitTok) || one <= kPairWaitOne);
  }
  if (!sure) return false;
  if (!tokens(kPairFewTok) && pairs * d < static_cast<long long>(kPairWork) * experts) return false;
  return !gate_up.idles() && !down.idles();
}

}  // namespace xs
