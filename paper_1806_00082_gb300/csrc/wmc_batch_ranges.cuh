// The work ranges of the batched step by its run-time parameter, in plain C++ so
// that the rule can be checked on the host.
//
// per_thread counts survivor ids per lane: the schedule's largest ranges are
// 32 per_thread ids in windows of 128, and never fewer than the single
// simulation's 16 windows, since shorter ones only add their own cost (512
// simulations of 2.67e8 particles, four steps: largest ranges of 4, 8, 16, 32, 64
// and 128 windows 4762, 3769, 3290, 3050, 3020 and 3340 us; 100 simulations of
// 5.1e7: 1104, 948, 895, 937, 990 and 990 us).  Values up to 64 are therefore one
// schedule; the candidates that are timed against each other are one of each.
#pragma once

#include <stdint.h>

namespace wmc {

constexpr uint32_t kMaxRange = 16;  // windows

constexpr bool valid_per_thread(int per) {
  return per == 4 || per == 8 || per == 16 || per == 32 || per == 64 || per == 128 || per == 256;
}

constexpr uint32_t batch_max_range(int per_thread) {
  return per_thread / 4 > (int)kMaxRange ? (uint32_t)per_thread / 4u : kMaxRange;
}

constexpr int kTuneCandidates[] = {16, 128, 256};

}  // namespace wmc
