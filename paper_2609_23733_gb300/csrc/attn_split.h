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

// From kShortTiles key tiles on, the number of parts S of each of the T groups minimises the last
// round's length over P CTAs in key tiles,
//   ceil(T S / P) (n_kv / S + kUnitTiles) + kCombineTiles S   (S = 1: no combine).
// kUnitTiles, the cost of a unit beyond its keys (Q load, pipeline fill and drain, partial store),
// and kCombineTiles, what a part adds to the combine, are fitted to sweeps at 1 to 16 heads and
// 2,748 to 137,400 tokens; being costs in time they do not shrink with n_kv.  (13 and 1.5, which fitted
// while a group's last part combined it, took 1.1 % longer in the mean of 17 shapes: 3 heads at
// 10,992 tokens 116.7 us against 111.8, 1 at 15,432 84.0 against 79.7, at 43,968 435 against 432.)
// Against a share of 3 % of a group per part at every length (captured calls with 6 surrogate heads beside):
// 16 heads at 10,992 tokens 390 -> 384 us (8 groups left over, 19 parts -> 13), one head at 43,968 478 -> 463
// (115 groups, whole -> 5 parts), at 137,400 3,785 -> 3,670 (54 groups, 5 -> 11); the same within 1 % for 3
// heads at 10,992 and one at 15,432.  Below kShortTiles the share rule stays although fewer parts are quicker
// (1,044 tokens: 4 heads 25.2 us with its 12 parts, 18.5 with 6 to 8; one head 18.5 with 17, 17.2 with 8): a
// deep stack of short sequences, which amplifies any other rounding, then gives the bits it always gave.
constexpr int kMaxParts = 64;
constexpr int kUnitTiles = 7, kCombineTiles = 1;
constexpr int kShortTiles = 41;
constexpr int kPartShare = 3;  // per cent

VP_HOST_DEVICE bool split_allowed(int T, int n_kv, int S) {
  return S == 1 || (S <= n_kv && T * S <= (n_kv < kShortTiles ? kFaTailUnits : kMaxTailUnits));
}

// Cost of S parts: in 1/4,096 of a key tile (n_kv capped at 2^19, 33.5 million tokens, so that 32 bits
// hold it: rounds <= S), and below kShortTiles in 2^-16 of a per cent of a group.  The smallest cost wins,
// and among equal ones the smallest S.
VP_HOST_DEVICE uint32_t split_cost(int T, int P, int n_kv, int S) {
  const uint32_t rounds = (uint32_t)((T * S + P - 1) / P), s = (uint32_t)S;
  if (n_kv < kShortTiles) return S == 1 ? 100u << 16 : (rounds * (100 + kPartShare * s) << 16) / s;
  const uint32_t n = (uint32_t)(n_kv < (1 << 19) - 1024 ? n_kv : (1 << 19) - 1024);
  return rounds * ((n << 12) / s + (kUnitTiles << 12)) + (S > 1 ? kCombineTiles * s << 12 : 0);
}

}  // namespace vp
