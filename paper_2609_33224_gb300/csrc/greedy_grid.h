// Blocks of the greedy pass's cooperative launch, which wait on one another and so must all be resident at
// once.  Plain C++ (no CUDA).
#pragma once

#include <cstdint>

namespace psgrid {

constexpr uint32_t kInsertBlocks = 64;  // insert blocks
constexpr uint32_t kProbeBlocks = 64;   // probe blocks
constexpr uint32_t kInsertGroup = 4;    // insert blocks that share a job (whole groups only)
constexpr uint32_t kMinBlocks = 1 + kInsertGroup + 1;
static_assert(kInsertBlocks % kInsertGroup == 0, "whole insert groups");

struct PipeGrid {
  uint32_t insert, probe;
  uint32_t blocks() const { return 1 + insert + probe; }  // and the deciding block
};

// The launch for a window of R requests where `resident` blocks fit on the device at once: a probe block per
// request and insert blocks if any request comes `lag` or more places after another (otherwise no row reads
// the delta table), up to 64 of each.  Any smaller number decides the same, only slower (each block takes its
// rows or jobs in order and only waits for earlier requests), so on a part of a GPU the two kinds share what
// fits; below kMinBlocks the launch is refused.
inline PipeGrid pipe_grid(uint32_t R, uint32_t lag, uint32_t resident) {
  PipeGrid g{R > lag ? kInsertBlocks : 0u, R < kProbeBlocks ? R : kProbeBlocks};
  const uint32_t room = resident > kMinBlocks ? resident - 1u : kMinBlocks - 1u;
  if (g.insert + g.probe > room) {
    if (g.insert) {
      const uint32_t half = room / 2u / kInsertGroup * kInsertGroup;
      const uint32_t left = g.probe < room ? (room - g.probe) / kInsertGroup * kInsertGroup : 0u;
      g.insert = half > left ? half : left;
      g.insert = g.insert < kInsertGroup ? kInsertGroup : (g.insert > kInsertBlocks ? kInsertBlocks : g.insert);
    }
    g.probe = g.probe < room - g.insert ? g.probe : room - g.insert;
  }
  return g;
}

}  // namespace psgrid
