// Where the cheap-heads kernel keeps a surrogate head's vectors while items are handed out one by one:
// plain C++, so that the host can go through the interleavings of the warps.
#pragma once

#include <stdint.h>

#include "host_device.h"

namespace vp {

// Shared-memory entry of the n-th head (0, 1, ..) that epilogue group g meets.  The entries are the
// group's own (the other group may be reading the same head's), and two, taken in turn: a warp writes
// entry n only after the hand-over of head n - 1, when every warp of the group is done with head n - 2.
VP_HOST_DEVICE int vec_entry(int g, uint32_t n) { return 2 * g + (int)(n & 1); }

}  // namespace vp
