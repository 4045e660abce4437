// Into how many parts the groups of full attention's last round are split along the keys: plain C++,
// in whole numbers.  The attention kernel and the kernel behind it that combines the parts each work
// the split out, in translation units of their own, so it may not depend on how a compiler rounds or
// contracts; and the host can evaluate it.
#pragma once

#include <stdint.h>

#include "host_device.h"

namespace vp {

#ifndef VP_ATTN_CHAINS
#define VP_ATTN_CHAINS 3
#endif
#ifndef VP_ATTN_BN
#define VP_ATTN_BN 64
#endif
constexpr int kFaChains = VP_ATTN_CHAINS;  // query tiles (chains) of a group
constexpr int kFaRows = 128;               // query rows of a tile
constexpr int kFaKeys = VP_ATTN_BN;        // keys of a tile

// Part units that the scratch holds if a group had four chains, and with kFaChains.
constexpr int kFaTailUnits = 512;
constexpr int kMaxTailUnits = kFaTailUnits * 4 / kFaChains;

// The number of parts S of each of the T groups of the last round, over P CTAs.  The fewest parts it may
// be is the S that a part's overhead of kPartShare per cent of a group makes the cheapest
// (ceil(T S / P) (1 / S + kPartShare / 100)).  Not below it, S minimises the last round's length in key
// tiles,
//   ceil(T S / P) (n_kv / S + kUnitTiles) + kCombineTiles S   (S = 1: no combine).
// kUnitTiles, the cost of a unit beyond its keys (Q load, pipeline fill and drain, partial store),
// and kCombineTiles, what a part adds to the combine, are fitted to sweeps at 1 to 16 heads and
// 2,748 to 137,400 tokens; being costs in time they do not shrink with n_kv.  Against the share alone
// (captured calls with 6 surrogate heads beside): one head at 43,968 tokens 478 -> 463 us (115 groups, whole ->
// 5 parts), at 137,400 3,785 -> 3,670 (54 groups, 5 -> 11); the same within 1 % for 3 heads at 10,992 and one at
// 15,432; the same S up to 60 key tiles.  Not below the share's S, although fewer parts would be quicker at
// some short lengths (16 heads at 10,992 tokens 384 us with 13 parts, 390 with 19; 1,044 tokens, 4 heads
// 18.5 us with 6 to 8, 25.2 with 12): a part takes its rows' exponentials against its own first maxima, whose
// weights, 1, bf16 holds exactly, and fewer parts are further off.  One head at 2,618 tokens against 64 bits,
// rms of four draws: 7.49e-5 with 6 parts, 7.18e-5 with 21.
constexpr int kMaxParts = 64;
constexpr int kUnitTiles = 7, kCombineTiles = 1;
constexpr int kPartShare = 3;  // per cent

// The argument of the smallest cost is taken, and among equal ones the smallest; kNoSplit: not to be taken.
constexpr uint32_t kNoSplit = 0xffffffffu;

VP_HOST_DEVICE uint32_t split_rounds(int T, int P, int S) { return (uint32_t)((T * S + P - 1) / P); }

// In 2^-16 of a per cent of a group.
VP_HOST_DEVICE uint32_t share_cost(int T, int P, int n_kv, int S) {
  if (S == 1) return 100u << 16;
  if (S > n_kv || T * S > kFaTailUnits) return kNoSplit;
  return (split_rounds(T, P, S) * (uint32_t)(100 + kPartShare * S) << 16) / (uint32_t)S;
}

// In 1/4,096 of a key tile, S not below least (n_kv capped at 2^19, 33.5 million tokens, so that 32 bits hold
// it: rounds <= S).
VP_HOST_DEVICE uint32_t split_cost(int T, int P, int n_kv, int S, int least) {
  if (S < least || (S > 1 && (S > n_kv || T * S > kMaxTailUnits))) return kNoSplit;
  const uint32_t n = (uint32_t)(n_kv < (1 << 19) - 1024 ? n_kv : (1 << 19) - 1024), s = (uint32_t)S;
  return split_rounds(T, P, S) * ((n << 12) / s + (kUnitTiles << 12)) + (S > 1 ? kCombineTiles * s << 12 : 0);
}

}  // namespace vp
