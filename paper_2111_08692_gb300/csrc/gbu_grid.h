// gbu_grid.h -- CTAs of a single-buffer launch (plain host code).
#pragma once

#include <stdint.h>

namespace gbu {

// The completion word (finish_packed in gbu_device.cuh) counts a launch's CTAs, and those of them
// with an error, in this many bits each: with more CTAs than they hold no CTA would be the last one.
constexpr int FIN_CTA_BITS = 12;
constexpr uint32_t MAX_GRID = (1u << FIN_CTA_BITS) - 1;

// resident: CTAs that run at once; useful: CTAs that have something to do.
constexpr uint32_t launch_grid(uint64_t resident, uint64_t useful) {
  const uint64_t g = useful < resident ? useful : resident;
  return g < 1 ? 1u : (g < MAX_GRID ? (uint32_t)g : MAX_GRID);
}

}  // namespace gbu
