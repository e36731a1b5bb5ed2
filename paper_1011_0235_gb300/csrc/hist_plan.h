// hist_plan.h -- the host's split of a launch's inputs (chunks, requests) into
// the CTAs' ranges, passed in the launch's parameters.
//
// The inputs are placed end to end at their costs, total W; CTA b takes the
// cost range [W b / grid, W (b + 1) / grid).  Planned on the host because a
// kernel that computes the split reads every input's size from the
// parameters and divides (about 8 us a launch of 1024 inputs).  On the host
// the split itself is a part of the call's time: one pass for the positions,
// one over the CTAs without divisions, and a third only where an input is too
// large for the groups.  1000 chunks of 1 KiB, whose counting takes 7.2 us:
// 6.0 us for the whole call (9.0 with a pass over the inputs for each of the
// plan's parts and a 64-bit division per CTA).
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

// The inputs' cost positions pos[0 .. count] (pos[count]: the total; `pos` has
// room for MAX + 1), their bytes, and their largest and smallest size.
template <uint32_t MAX>
struct PlanCosts {
  unsigned long long pos[MAX + 1];
  unsigned long long bytes, largest, smallest;
};
template <uint32_t MAX, class Size, class Cost>
void plan_costs(PlanCosts<MAX>* c, uint32_t count, Size size, Cost cost) {
  unsigned long long x = 0, bytes = 0, hi = 0, lo = ~0ull;
  for (uint32_t i = 0; i < count; ++i) {
    const unsigned long long n = size(i);
    c->pos[i] = x;
    x += cost(i);
    bytes += n;
    hi = n > hi ? n : hi;
    lo = n < lo ? n : lo;
  }
  c->pos[count] = x;
  c->bytes = bytes;
  c->largest = hi;
  c->smallest = lo;
}

// Fill `p` for inputs of costs `c` and sizes size(i) on `grid` CTAs (at most
// kPlanCtas).  Whole inputs of at most small_max bytes go to the groups if at
// least half of the launch's cost is theirs.
template <uint32_t MAX, class Size>
void plan_ranges(RangePlan* p, const PlanCosts<MAX>& c, uint32_t count, uint32_t grid, unsigned long long small_max,
                 Size size) {
  const unsigned long long W = c.pos[count], range = W / grid, rest = W % grid;
  p->range = range;
  uint32_t j = 0;
  unsigned long long lo = 0, part = 0;  // lo = W b / grid, part = rest b mod grid
  for (uint32_t b = 0; b < grid; ++b) {
    while (j + 1 < count && c.pos[j + 1] <= lo) ++j;
    p->lo[b] = lo;
    p->pre[b] = c.pos[j];
    p->j[b] = (uint16_t)j;
    p->s[b] = (uint16_t)(c.pos[j] == lo ? j : j + 1);  // the first whose cost position is at least lo
    lo += range;
    part += rest;
    if (part >= grid) {
      part -= grid;
      ++lo;
    }
  }
  p->lo[grid] = W;
  p->s[grid] = (uint16_t)count;
  // the inputs the groups take (as the kernels decide); a launch without
  // groups has no memory for their tables: no CTA of it may take their path,
  // whatever its range holds
  memset(p->groups, 0, sizeof(p->groups));
  if (c.smallest != 0 && c.largest <= small_max && plan_whole(c.largest, range)) {  // all of them
    p->group_max = (uint32_t)small_max;
    memset(p->groups, 0xff, sizeof(p->groups));
    return;
  }
  auto small = [&](uint32_t i) { return size(i) != 0 && size(i) <= small_max && plan_whole(size(i), range); };
  unsigned long long small_cost = 0;
  for (uint32_t i = 0; i < count; ++i)
    if (small(i)) small_cost += c.pos[i + 1] - c.pos[i];
  p->group_max = 2 * small_cost >= W ? (uint32_t)small_max : 0;
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
