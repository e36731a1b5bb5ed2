// hist_plan.h -- the host's split of a launch's inputs (chunks, requests) into
// the CTAs' ranges, passed in the launch's parameters.
//
// The inputs are placed end to end at their costs, total W; CTA b takes the
// cost range [W b / grid, W (b + 1) / grid).  Planned on the host because a
// kernel that computes the split reads every input's size from the
// parameters and divides (about 8 us a launch of 1024 inputs).
#pragma once

#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>
#include <string.h>

namespace histlib {

constexpr uint32_t kPlanCtas = 160;  // largest grid

struct RangePlan {
  unsigned long long range;                // W / grid
  unsigned long long lo[kPlanCtas + 1];    // CTA b's range is [lo[b], lo[b + 1])
  unsigned long long pre[kPlanCtas];       // cost position of its first input
  uint16_t j[kPlanCtas];                   // its first input: the last whose cost position is at most lo[b]
  // CTA b with bit b of `groups` set has only whole inputs for the groups:
  // inputs [s[b], s[b + 1]) start in its range, and any input that overlaps
  // the range from before is whole (an earlier CTA's)
  uint16_t s[kPlanCtas + 1];
  uint32_t groups[(kPlanCtas + 31) / 32];
  uint32_t group_max;                      // largest input left to the groups (0: a launch without groups)
};

// Whether an input of n bytes is counted whole by the CTA whose range holds
// its first cost position: at most a quarter of a range.
__host__ __device__ constexpr bool plan_whole(unsigned long long n, unsigned long long range) { return n * 4 <= range; }

// Fill `p` for inputs of sizes size(i) and costs cost(i) on `grid` CTAs (at
// most kPlanCtas).  Whole inputs of at most small_max bytes go to the groups
// if at least half of the launch's cost is theirs.
template <class Size, class Cost>
void plan_ranges(RangePlan* p, uint32_t count, uint32_t grid, unsigned long long small_max, Size size, Cost cost) {
  unsigned long long W = 0;
  for (uint32_t i = 0; i < count; ++i) W += cost(i);
  p->range = W / grid;
  uint32_t j = 0;
  unsigned long long pj = 0;  // cost position of input j
  for (uint32_t b = 0; b <= grid; ++b) {
    const unsigned long long lo = W * b / grid;
    p->lo[b] = lo;
    if (b == grid) break;
    while (j + 1 < count && pj + cost(j) <= lo) {
      pj += cost(j);
      ++j;
    }
    p->j[b] = (uint16_t)j;
    p->pre[b] = pj;
  }
  // the inputs the groups take (as the kernels decide)
  const unsigned long long range = p->range;
  auto small = [&](uint32_t i) { return size(i) != 0 && size(i) <= small_max && plan_whole(size(i), range); };
  unsigned long long small_cost = 0;
  for (uint32_t i = 0; i < count; ++i)
    if (small(i)) small_cost += cost(i);
  p->group_max = 2 * small_cost >= W ? (uint32_t)small_max : 0;
  uint32_t i = 0;  // first input whose cost position is at least the range's start
  unsigned long long pi = 0;
  for (uint32_t b = 0; b <= grid; ++b) {
    const unsigned long long lo = p->lo[b];
    while (i < count && pi < lo) {
      pi += cost(i);
      ++i;
    }
    p->s[b] = (uint16_t)i;
  }
  // (a launch without groups has no memory for their tables: no CTA of it may
  // take their path, whatever its range holds)
  memset(p->groups, 0, sizeof(p->groups));
  for (uint32_t b = 0; p->group_max && b < grid; ++b) {
    bool only = true;
    const uint32_t j0 = p->j[b], s0 = p->s[b], s1 = p->s[b + 1];
    // an input that starts before the range and reaches into it
    for (uint32_t k = j0; k < s0 && only; ++k) only = plan_whole(size(k), range);
    for (uint32_t k = s0; k < s1 && only; ++k) only = small(k);
    if (only) p->groups[b >> 5] |= 1u << (b & 31);
  }
}

}  // namespace histlib
