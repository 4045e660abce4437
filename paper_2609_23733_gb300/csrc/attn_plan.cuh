// How the full-attention work of a layer is cut (attn_full.cu), and the combine of the groups that
// were split along the keys, which the kernel behind the attention runs (combine_split_heads).
#pragma once

#include <math.h>

#include "attn_split.h"
#include "common.cuh"
#include "internal.h"

namespace vp {

struct Plan {
  int R, T, S, units;
  int whole;  // units of the whole-group instance (they come first)
};

// The work of one launch: G groups (head, kFaChains query tiles) over P persistent CTAs.  The
// first R = floor(G / P) rounds take whole groups; the T = G - R P groups of the last round
// are split along the keys into S parts each (at most the number of key tiles), T S part units,
// so the last round lasts about ceil(T S / P) parts of a group instead of one whole group on T
// CTAs.  Unit u < R P is group u; unit R P + S t + s is part s of group R P + t.  attn_split.h chooses S.
//
// Called by whole warps: lane l weighs S = l + 1 and l + 33 (a loop over S in every thread took
// several microseconds of every launch).
__device__ __forceinline__ Plan make_plan(int G, int P, int n_kv, bool parts_only) {
  static_assert(kMaxParts == 64, "two values of S per lane");
  Plan pl;
  pl.R = G / P;
  pl.T = G - pl.R * P;
  pl.S = 1;
  if (pl.T > 0) {
    const int s0 = lane_id() + 1, s1 = s0 + 32;
    auto cheapest = [](uint32_t c0, uint32_t c1) -> int {
      const uint32_t best = __reduce_min_sync(0xffffffffu, min(c0, c1));
      const uint32_t lo = __ballot_sync(0xffffffffu, c0 == best), hi = __ballot_sync(0xffffffffu, c1 == best);
      return lo ? __ffs(lo) : 32 + __ffs(hi);
    };
    pl.S = cheapest(share_cost(pl.T, P, n_kv, s0), share_cost(pl.T, P, n_kv, s1));
    pl.S = cheapest(split_cost(pl.T, P, n_kv, s0, pl.S), split_cost(pl.T, P, n_kv, s1, pl.S));
  }
  pl.units = pl.S == 1 ? G : pl.R * P + pl.T * pl.S;
  pl.whole = parts_only ? 0 : (pl.S == 1 ? G : pl.R * P);
  return pl;
}

// A part's rows in the scratch: slot t S + s holds [chain][quarter] blocks of 32 rows (lanes); a
// block's O lies lane-minor ([16-byte chunk of the row][lane]), its (m, l, xmax) a float4 per lane,
// so that every store and load of a warp is 512 contiguous bytes.
constexpr size_t kFaSlotRows = (size_t)kFaChains * 4 * 32;

// The split groups' rows of Y (and their share of the saliency) from the parts of a finished
// attention launch over P CTAs: M = max m_s, O = sum 2^(m_s - M) O_s, l = sum 2^(m_s - M) l_s,
// parts in order.  Called by whole warps, warp w of n_warps of the grid behind the attention
// kernel: a warp takes 8 channels of a block of 32 rows at a time, so the partial rows come in
// over every SM (one group's are up to 1.7 MB; the last part's CTA on its own took 15 us for
// them at 1,044 tokens).
// Not inlined: the kernels that end with it keep their code and registers.
static __device__ __noinline__ void combine_split_heads(const HeadAttnArgs& a, int P, int w, int n_warps) {
  const int first = a.offsets[2], n_heads = a.offsets[3] - first;
  const int n_groups = (a.N + kFaChains * kFaRows - 1) / (kFaChains * kFaRows);
  const Plan pl = make_plan(n_heads * n_groups, P, (a.N + kFaKeys - 1) / kFaKeys, false);
  if (pl.S == 1) return;
  const int lane = lane_id();
  for (int task = w; task < pl.T * kFaChains * 32; task += n_warps) {
    const int piece = task & 7, quarter = (task >> 3) & 3, ct = task >> 5;
    const int t = ct / kFaChains, c = ct - t * kFaChains;
    const int group = pl.R * P + t;
    const int h = a.head_ids[first + group / n_groups];
    const int row = ((group % n_groups) * kFaChains + c) * kFaRows + quarter * 32 + lane;
    const size_t blk = (size_t)t * pl.S * kFaSlotRows + (size_t)(c * 4 + quarter) * 32;
    const float4* st = reinterpret_cast<const float4*>(a.fa_stats) + blk + lane;
    const float4* pq = reinterpret_cast<const float4*>(a.fa_part) + blk * 16 + piece * 64 + lane;
    float M = -INFINITY, X = -INFINITY;
#pragma unroll 8
    for (int sp = 0; sp < pl.S; ++sp) {
      const float4 s4 = __ldcg(st + sp * kFaSlotRows);
      M = fmaxf(M, s4.x);
      X = fmaxf(X, s4.z);
    }
    float L = 0.f, acc[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) acc[i] = 0.f;
#pragma unroll 6
    for (int sp = 0; sp < pl.S; ++sp) {
      const float2 s4 = __ldcg(reinterpret_cast<const float2*>(st + sp * kFaSlotRows));
      float4 f[2];
#pragma unroll
      for (int q = 0; q < 2; ++q) f[q] = __ldcg(pq + sp * kFaSlotRows * 16 + q * 32);
      const float wgt = fast_exp2(s4.x - M);
      L = fmaf(wgt, s4.y, L);
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        acc[4 * q] = fmaf(wgt, f[q].x, acc[4 * q]);
        acc[4 * q + 1] = fmaf(wgt, f[q].y, acc[4 * q + 1]);
        acc[4 * q + 2] = fmaf(wgt, f[q].z, acc[4 * q + 2]);
        acc[4 * q + 3] = fmaf(wgt, f[q].w, acc[4 * q + 3]);
      }
    }
    const float inv = 1.f / L;
    if (row < a.N) {
      uint4 v;
      v.x = pack_bf16x2(acc[0] * inv, acc[1] * inv);
      v.y = pack_bf16x2(acc[2] * inv, acc[3] * inv);
      v.z = pack_bf16x2(acc[4] * inv, acc[5] * inv);
      v.w = pack_bf16x2(acc[6] * inv, acc[7] * inv);
      reinterpret_cast<uint4*>(a.y + ((size_t)row * a.H + h) * 64)[piece] = v;
    }
    if (a.s_attn && piece == 0) {
      float v = row < a.N ? fast_exp2(X - M) * inv : 0.f;
#pragma unroll
      for (int k = 16; k > 0; k >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, k));
      if (lane == 0) atomicMax(reinterpret_cast<int*>(a.s_attn + h), __float_as_int(v));
    }
  }
}

}  // namespace vp
