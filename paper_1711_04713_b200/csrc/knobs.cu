#include "knobs.cuh"

#include <cstring>

#include "common.cuh"

namespace adaption {

static const char* const kKnobNames[kNumKnobs] = {
    "splits", "pair", "fast", "staged", "stages", "bk", "bn", "kps", "bres", "wide", "epigroups", "timeout_us", "stall_at",
    "split_hh", "pdl", "stagger", "stage_bufs", "cluster", "cluster_size", "cluster_bn",
    "pixels", "box", "halo"};
const int kKnobDefaults[kNumKnobs] = {0, -1, 1, 1, 0, 0, 0, 0, 1, 1, 4, 0, -1, 1, 1, 1, 2, 1, 0, 0, 1, 1, 1};
std::atomic<int> g_knobs[kNumKnobs] = {{0}, {-1}, {1}, {1}, {0}, {0}, {0}, {0}, {1}, {1}, {4}, {0}, {-1}, {1}, {1},
                                       {1}, {2}, {1}, {0}, {0}, {1}, {1}, {1}};

int debug_set(const char* name, int value) {
  if (name == nullptr) return ADAPTION_ERR_INVALID_ARG;
  if (std::strcmp(name, "reset") == 0) {
    for (int k = 0; k < kNumKnobs; ++k) g_knobs[k].store(kKnobDefaults[k], std::memory_order_relaxed);
    return ADAPTION_OK;
  }
  for (int k = 0; k < kNumKnobs; ++k)
    if (std::strcmp(name, kKnobNames[k]) == 0) {
      g_knobs[k].store(value, std::memory_order_relaxed);
      return ADAPTION_OK;
    }
  return ADAPTION_ERR_INVALID_ARG;
}

bool pdl_enabled() { return knob(kPdl) != 0; }

}  // namespace adaption
