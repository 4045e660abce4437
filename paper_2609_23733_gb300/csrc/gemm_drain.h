// What is still in flight in the GEMM's ring after a failed wait: plain C++, so that the host can check it
// against a model of the barriers.
#pragma once

#include <stdint.h>

#include "host_device.h"

namespace vp {

// Uses of ring stage s by a producer that has issued n K blocks.
VP_HOST_DEVICE uint32_t stage_uses(uint32_t n, uint32_t s, uint32_t stages) {
  return n > s ? (n - 1 - s) / stages + 1 : 0;
}

// A stage's barrier (the leader's) expects both CTAs' halves once the leader has issued the K block, but
// a failed wait can stop the two producers at different ones (at most one use of a stage apart: a use
// begins when the MMAs have read the one before).
struct StageDrain {
  uint32_t uses;   // phases to see completed (0: the stage was never used)
  int fix;         // of the last use: +1 the leader has yet to expect the peer's half alone,
                   // -1 it expects a half that the peer never issued, 0 neither
  uint32_t block;  // the K block of the last use
};
VP_HOST_DEVICE StageDrain stage_drain(uint32_t leader, uint32_t peer, uint32_t s, uint32_t stages) {
  const uint32_t a = stage_uses(leader, s, stages), b = stage_uses(peer, s, stages);
  StageDrain d;
  d.uses = a > b ? a : b;
  d.fix = (int)b - (int)a;
  d.block = d.uses == 0 ? 0 : (d.uses - 1) * stages + s;
  return d;
}

}  // namespace vp
