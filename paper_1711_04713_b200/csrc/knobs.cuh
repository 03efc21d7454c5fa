// Test and experiment overrides of the dispatch heuristics (adaption_debug_set).
#pragma once

#include <atomic>

namespace adaption {

enum Knob { kSplits, kPair, kFast, kStaged, kStages, kBK, kBN, kKps, kBres, kWide, kEpiGroups, kTimeoutUs, kStallAt,
            kSplitHh, kPdl, kStagger, kStageBufs, kCluster, kClusterSize, kClusterBN, kPixels, kBox, kHalo, kNumKnobs };

// Each holds its default until set; the setter is the only writer.
extern std::atomic<int> g_knobs[kNumKnobs];
extern const int kKnobDefaults[kNumKnobs];

inline int knob(Knob k) { return g_knobs[k].load(std::memory_order_relaxed); }

// limit of a device-side wait in nanoseconds
inline unsigned long long wait_limit_ns() {
  return knob(kTimeoutUs) > 0 ? 1000ull * (unsigned long long)knob(kTimeoutUs) : 2000000000ull;
}

}  // namespace adaption
