// Surrogate heads (§4.3) and mean heads (Algorithm 1, step 2, s_h <= tau_low) of a layer on
// the sm_103a tensor cores, queued behind the full-attention kernel with programmatic
// dependent launch (its CTAs take the SMs that full attention's last round frees).
//
// Surrogate head h, per token i:  z_i = [v_i, C_h],
//   y_i = C_h + sigma(MLP_gamma(z_i)) (.) MLP_delta(z_i),  MLP = Linear(2d -> 64) -> GELU ->
//   Linear(64 -> d).
// The first layer splits as W1 z = W1[:, :d] v_i + (W1[:, d:] C_h + b1): the second term (c1)
// is one vector per head.  Per 128-token tile, with both MLPs side by side:
//   D1 = V W1v^T      [128 x 128] = tcgen05.mma M128 N128 K16 x 4 (V and [W1v_gamma; W1v_delta]
//                     from shared memory, 128-byte swizzle), fp32 in TMEM;
//   H = 2 GELU(D1 + c1) as bf16 pairs in 64 TMEM columns of their own (x2 exact in bf16);
//   D2g = H[:, :64] W2g^T, D2d = H[:, 64:] W2d^T  [128 x 64] each = tcgen05.mma M128 N64 K16
//                     x 4 each, A read from TMEM (TS form), W2 from shared memory, into D1's
//                     columns (D1 has been read by then);
//   y = C + sigma(D2g + b2g) (.) (D2d + b2d), bf16, staged in shared memory (128-byte swizzle)
//                     and written by a TMA tensor store into Y[:, h, :].
// A mean item writes Broadcast(mean of V_h) over 1,024 tokens with coalesced 16-byte stores.
//
// Roles (576 threads, one CTA per SM, persistent over items taken kBatch at a time from a
// device counter: surrogate tiles of 128 tokens head-major, then mean items of 1,024 tokens):
//   warp 0     producer: items, TMA loads of the V tiles (kStages ring) and of each head's
//              weights into one of two weight slots (a slot is reloaded once the MMAs of the
//              head before the previous one have completed);
//   warp 1     TMEM owner (512 columns) and MMA issue: the first layer of the next tile and
//              the second layer of a tile whose H is written, each as soon as it is ready;
//   warps 2-9, 10-17  two epilogue groups of eight warps, each with 256 TMEM columns; group g takes
//              tiles t = g (mod 2): D1 and, in place, H in its first 128 columns, D2g | D2d in
//              the other 128.  The tensor pipe runs the MMAs in the order of issue, so the first
//              layer of the group's next tile goes out right behind the second layer that reads
//              H.  The two warps of a TMEM lane quarter split a token row's columns, and no warp
//              waits for another one: each stages and stores its own 32 x 32 block of y (TMA),
//              and the hand-overs are mbarriers.  With group barriers around a staged tile (three
//              a tile) the same work took 171 us for 16 surrogate heads at 87,936 tokens, now 165.
//              The surrogate heads' vectors (c1 = W1[:, d:] C_h + b1, the second layer's biases,
//              C_h) are put into shared memory beside the first copies and MMAs.
// Bounded by the latency of that chain with two tiles in flight: issue, FMA and MUFU are each below
// half of their rate.  All 16 warps on one tile at a time, the gate one tile behind, measured slower
// (184 vs 171 us): the phases of the warps then coincide.
// The register file is split between the four SM sub-partitions: 18 warps put 5 on some of
// them, which caps a thread at 96 registers (16,384 / (5 x 32), in steps of 8).  Three warps
// per lane quarter (26 warps, 72 registers) measured slower: 0.301 vs 0.269 ms for 16 heads
// at 137,400 tokens.
// Every wait is bounded (mbar_wait); on timeout the CTA records VP_DEVERR_WAIT_TIMEOUT, stops,
// waits (bounded) for its own copies and MMAs, frees TMEM and exits.
#include "attn_plan.cuh"
#include "common.cuh"
#include "heads_vec.h"
#include "internal.h"

namespace vp {

namespace {

constexpr int kTcTile = 128;      // tokens per surrogate item
constexpr int kMeanRows = 1024;   // tokens per mean item (a pure write, handed over less often)
constexpr int kTcStages = 4;      // V tiles in flight
constexpr int kTcGroups = 2;      // epilogue groups (= TMEM accumulators)
constexpr int kTcBatch = 4;       // items taken from the counter at a time (one when there are few)
constexpr int kTcParts = 2;       // epilogue warps per TMEM lane quarter in a group
constexpr int kGroupThreads = 128 * kTcParts;
static_assert(2 * kTcGroups <= kMaxHeads, "vec_entry");
constexpr int kTcThreads = 64 + kGroupThreads * kTcGroups;
// A row's work split over the kTcParts warps of its lane quarter: part p takes the chunk
// range [begin(p), begin(p + 1)) of the n chunks, as even as possible.  The first layer's
// 8 chunks go in part order and the second layer's 4 in reverse, so that a part short of
// first-layer chunks takes more second-layer ones.
__host__ __device__ constexpr int part_begin(int p, int n) { return (p * n + kTcParts - 1) / kTcParts; }
constexpr int kMaxGChunks = (8 + kTcParts - 1) / kTcParts;
constexpr int kMaxFChunks = (4 + kTcParts - 1) / kTcParts;
constexpr uint32_t kTcTmemCols = 512;
constexpr uint32_t kVTileBytes = kTcTile * 64 * 2;
constexpr uint32_t kW1Bytes = 128 * 64 * 2;  // [W1v_gamma; W1v_delta]: 128 hidden x 64 inputs
constexpr uint32_t kW2Bytes = 128 * 64 * 2;  // [W2_gamma; W2_delta]: 2 x (64 outputs x 64 hidden)

struct TcSmem {
  __nv_bfloat16 v[kTcStages][kTcTile * 64];
  __nv_bfloat16 w1[2][128 * 64];
  __nv_bfloat16 w2[2][128 * 64];
  __nv_bfloat16 ys[4 * kTcParts * kTcGroups][32 * 32];  // a warp's output block, 64-byte swizzle
  // Surrogate heads' vectors: every head's by slot in the surrogate bin, computed at kernel start, or with
  // single items two entries per epilogue group (vec_entry), computed when a tile first needs them:
  // W1[:, d:] C_h + b1 (gamma | delta), -log2(e) b2_gamma | b2_delta, and C_h.
  float c1[kMaxHeads][128];
  float b2[kMaxHeads][128];
  float cx[kMaxHeads][64];
  int stage_item[kTcStages];                  // item, or -1: no more items
  int stage_fill[kTcStages];                  // weight fill of a surrogate item (slot = fill & 1), -1
  int stage_head[kTcStages];
  int stage_slot[kTcStages], stage_tile[kTcStages];  // item = slot x tiles + tile (divided once, here)
  int acc_item[kTcGroups], acc_head[kTcGroups], acc_slot[kTcGroups], acc_tile[kTcGroups];
  uint64_t full[kTcStages], empty[kTcStages];
  uint64_t w_full[2], w_empty[2];
  uint64_t d1_full[kTcGroups], h_full[kTcGroups], d2_full[kTcGroups], taken[kTcGroups], vec_full[kTcGroups];
  uint64_t drain;
  uint32_t tmem_base;
  int abort_flag;
  int first_item;  // the first batch's start
};

// Component u (0 .. 127) of the vectors of the surrogate head h, into an entry: of c1, the first layer's context
// half folded (a 64-term dot product per hidden unit), and of the second layer's biases and C_h.
__device__ __noinline__ void head_c1(const HeadAttnArgs& a, TcSmem& sm, int entry, int h, int u) {
  const int uu = u & 63;
  const float4* ctx = reinterpret_cast<const float4*>(a.ctx + h * 64);
  const __nv_bfloat16* w = (u < 64 ? a.sw.g1_w : a.sw.d1_w) + ((size_t)h * 64 + uu) * 128 + 64;
  float acc = (u < 64 ? a.sw.g1_b : a.sw.d1_b)[h * 64 + uu];
#pragma unroll
  for (int kq = 0; kq < 8; ++kq) {
    const uint4 wv = reinterpret_cast<const uint4*>(w)[kq];
    const float4 c0 = ctx[2 * kq], c1 = ctx[2 * kq + 1];
    acc = fmaf(bf16_lo(wv.x), c0.x, fmaf(bf16_hi(wv.x), c0.y, acc));
    acc = fmaf(bf16_lo(wv.y), c0.z, fmaf(bf16_hi(wv.y), c0.w, acc));
    acc = fmaf(bf16_lo(wv.z), c1.x, fmaf(bf16_hi(wv.z), c1.y, acc));
    acc = fmaf(bf16_lo(wv.w), c1.z, fmaf(bf16_hi(wv.w), c1.w, acc));
  }
  sm.c1[entry][u] = acc;
}
__device__ __forceinline__ void head_out(const HeadAttnArgs& a, TcSmem& sm, int entry, int h, int u) {
  const float b = (u < 64 ? a.sw.g2_b : a.sw.d2_b)[h * 64 + (u & 63)];
  sm.b2[entry][u] = u < 64 ? -1.4426950408889634f * b : b;  // gamma's enters sigma's exponent
  if (u < 64) sm.cx[entry][u] = a.ctx[h * 64 + u];
}

struct TcMaps {
  CUtensorMap v, y, g1, d1, g2, d2;
};

__global__ void __launch_bounds__(kTcThreads, 1) cheap_heads_tc_kernel(const __grid_constant__ TcMaps maps, HeadAttnArgs a) {
  extern __shared__ unsigned char smem_raw[];
  TcSmem& sm = *reinterpret_cast<TcSmem*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  const int tid = threadIdx.x;
  const int warp = warp_uniform_id(), lane = lane_id();
  volatile int* abort_flag = &sm.abort_flag;
  unsigned int* err = a.err;
  const int H = a.H;
  const int m_first = a.offsets[0], s_first = a.offsets[1];
  const int n_surr = a.offsets[2] - s_first, n_mean = s_first - m_first;
  const int T = (a.N + kTcTile - 1) / kTcTile;
  const int surr_items = n_surr * T;
  const int Tm = (a.N + kMeanRows - 1) / kMeanRows;  // mean items per head
  // Mean heads folded into W_O's bias (skip_mean_y) need no rows of Y.
  const int items = surr_items + (a.skip_mean_y ? 0 : n_mean * Tm);
  // With fewer than two batches per CTA, items go out one by one (63 items of one 1,044-token layer:
  // 16 CTAs took four each, one after another).
  const int batch = items > 2 * kTcBatch * (int)gridDim.x ? kTcBatch : 1;

  pdl_launch();
  if (tid == 0) {
    sm.first_item = (int)atomicAdd(a.cheap_counter, (unsigned)batch);
    for (int s = 0; s < kTcStages; ++s) {
      mbar_init(&sm.full[s], 1);
      mbar_init(&sm.empty[s], 1);
    }
    for (int s = 0; s < 2; ++s) {
      mbar_init(&sm.w_full[s], 1);
      mbar_init(&sm.w_empty[s], 1);
    }
    for (int g = 0; g < kTcGroups; ++g) {
      mbar_init(&sm.d1_full[g], 2);  // the MMA commit (or a stand-in) + the item hand-over
      mbar_init(&sm.h_full[g], 4 * kTcParts);  // a warp each
      mbar_init(&sm.d2_full[g], 1);
      mbar_init(&sm.taken[g], 4 * kTcParts);   // every warp has read a mean item
      mbar_init(&sm.vec_full[g], 4 * kTcParts);
    }
    mbar_init(&sm.drain, 1);
    sm.abort_flag = 0;
    fence_mbarrier_init();
    fence_proxy_async_smem();
    tma_prefetch_desc(&maps.v);
    tma_prefetch_desc(&maps.y);
  }
  if (warp == 1) {
    tmem_alloc(&sm.tmem_base, kTcTmemCols);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = __shfl_sync(0xffffffffu, sm.tmem_base, 0);

  // A CTA that starts behind the attention's last round may find every item taken: it goes
  // straight to the combine.
  const int first_item = __shfl_sync(0xffffffffu, sm.first_item, 0);
  if (first_item >= items) {
  } else if (warp == 0) {
    // ------------------------------------------------------------ producer
    int fill = -1, cur_h = -1, next = first_item, left = batch;
    int tma_k[kTcStages];  // last item index k whose V tile went to stage s (-1: none)
#pragma unroll
    for (int s = 0; s < kTcStages; ++s) tma_k[s] = -1;
    bool ok = true;
    for (int k = 0;; ++k) {
      if (left == 0) {
        int b = 0;
        if (lane == 0) b = (int)atomicAdd(a.cheap_counter, (unsigned)batch);
        next = __shfl_sync(0xffffffffu, b, 0);
        left = batch;
      }
      const int it = next++;
      --left;
      const int st = k % kTcStages;
      ok = mbar_wait_warp(&sm.empty[st], ((k / kTcStages) & 1) ^ 1, err, abort_flag);
      if (!ok) break;
      if (it >= items) {
        if (elect_one()) {
          sm.stage_item[st] = -1;
          mbar_arrive(&sm.full[st]);
        }
        __syncwarp();
        break;
      }
      if (it < surr_items) {
        const int slot = it / T, tile = it - slot * T;
        const int h = a.head_ids[s_first + slot];
        if (h != cur_h) {  // this head's weights into the next slot
          ++fill;
          cur_h = h;
          const int ws = fill & 1;
          if (fill >= 2) {  // the MMAs of fill - 2 (same slot) have completed
            ok = mbar_wait_warp(&sm.w_empty[ws], ((fill - 2) >> 1) & 1, err, abort_flag);
            if (!ok) break;
          }
          if (elect_one()) {
            mbar_arrive_expect_tx(&sm.w_full[ws], kW1Bytes + kW2Bytes);
            tma_load_2d(sm.w1[ws], &maps.g1, &sm.w_full[ws], 0, h * 64);
            tma_load_2d(sm.w1[ws] + 64 * 64, &maps.d1, &sm.w_full[ws], 0, h * 64);
            tma_load_2d(sm.w2[ws], &maps.g2, &sm.w_full[ws], 0, h * 64);
            tma_load_2d(sm.w2[ws] + 64 * 64, &maps.d2, &sm.w_full[ws], 0, h * 64);
          }
          __syncwarp();
        }
        if (elect_one()) {
          sm.stage_item[st] = it;
          sm.stage_fill[st] = fill;
          sm.stage_head[st] = h;
          sm.stage_slot[st] = slot;
          sm.stage_tile[st] = tile;
          mbar_arrive_expect_tx(&sm.full[st], kVTileBytes);
          tma_load_2d(sm.v[st], &maps.v, &sm.full[st], (2 * H + h) * 64, tile * kTcTile);
        }
        __syncwarp();
        tma_k[st] = k;
      } else {
        const int slot = (it - surr_items) / Tm, tile = it - surr_items - slot * Tm;
        const int h = a.head_ids[m_first + slot];
        if (elect_one()) {
          sm.stage_item[st] = it;
          sm.stage_fill[st] = -1;
          sm.stage_head[st] = h;
          sm.stage_slot[st] = slot;
          sm.stage_tile[st] = tile;
          mbar_arrive(&sm.full[st]);
        }
        __syncwarp();
      }
    }
    if (!ok && lane == 0) {  // let issued copies land before the CTA releases its smem
      for (int s = 0; s < kTcStages; ++s)
        if (tma_k[s] >= 0)
          for (int t = 0; t < 1000000 && !mbar_try_wait(&sm.full[s], (tma_k[s] / kTcStages) & 1); ++t) {}
      for (int f = fill; f >= 0 && f >= fill - 1; --f)
        for (int t = 0; t < 1000000 && !mbar_try_wait(&sm.w_full[f & 1], (f >> 1) & 1); ++t) {}
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issue
    // A polling loop over two independent kinds of work, issued as soon as each is ready:
    // the first layer of the next tile (its V tile loaded, its accumulator free, its weights
    // loaded) and the second layer of the oldest tile whose H is written.  Tying them to one
    // order would make a group's second layer wait for the other group's epilogue.
    const uint32_t id1 = idesc_bf16(128, 128, 0, 0);  // V (K-major) x W1v^T (K-major)
    const uint32_t id2 = idesc_bf16(128, 64, 0, 0);   // H (TMEM) x W2^T (K-major)
    bool ok = true;
    int k = 0;                        // next tile for the first layer
    bool feeding = true;              // false once the stop item has been read
    int waited_fill = -1;             // newest weight fill known to be loaded
    int cur_fill = -1;                // fill of the newest surrogate tile
    int release = -1;                 // a finished fill whose slot is released once its
                                      // tiles' second layers are issued
    int qk[2], qfill[2];              // tiles waiting for their second layer (oldest first)
    uint32_t qsur[2];
    int qn = 0;
    uint32_t sur_cnt[kTcGroups] = {0u, 0u};  // surrogate tiles sent to group g
    uint32_t sec_cnt[kTcGroups] = {0u, 0u};  // their second layers issued
    uint32_t mean_cnt[kTcGroups] = {0u, 0u}; // mean items sent to group g
    int last_kind[kTcGroups] = {-1, -1};     // kind of group g's last tile (1 surrogate, 0 mean)
    // Tile kk may go to its group once the group's previous tile's second layer has been issued
    // (it reads H, which tile kk's first layer overwrites, and every warp has read the item), or,
    // for a mean item, once every warp has read it.
    auto group_free = [&](int kk) -> bool {
      const int gb = kk & 1;
      if (last_kind[gb] < 0) return true;
      if (last_kind[gb] == 1) return sec_cnt[gb] == sur_cnt[gb];
      return mbar_test_wait(&sm.taken[gb], (mean_cnt[gb] - 1) & 1);
    };
    unsigned long long t0 = 0;
    for (uint32_t spin = 1;; ++spin) {
      bool progress = false;
      if (qn > 0) {  // second layer of the oldest waiting tile
        const int pb = qk[0] & 1;
        const bool ready = __shfl_sync(0xffffffffu, (int)mbar_test_wait(&sm.h_full[pb], qsur[0] & 1), 0);
        if (ready) {
          tc_fence_after();
          const uint32_t t_h = tmem + pb * 256, t_main = t_h + 128;
          const uint64_t dg = sdesc_sw128(smem_u32(sm.w2[qfill[0] & 1]));
          const uint64_t dd = sdesc_sw128(smem_u32(sm.w2[qfill[0] & 1] + 64 * 64));
          if (elect_one()) {
#pragma unroll
            for (int kk = 0; kk < 4; ++kk)  // gamma: hidden units 0..63 = H columns 0..31
              tc_mma_ts(t_main, t_h + 8 * kk, dg + 2 * kk, id2, kk > 0 ? 1u : 0u);
#pragma unroll
            for (int kk = 0; kk < 4; ++kk)  // delta: hidden units 64..127 = H columns 64..95
              tc_mma_ts(t_main + 64, t_h + 64 + 8 * kk, dd + 2 * kk, id2, kk > 0 ? 1u : 0u);
            tc_commit(&sm.d2_full[pb]);
          }
          __syncwarp();
          ++sec_cnt[pb];
          qk[0] = qk[1];
          qfill[0] = qfill[1];
          qsur[0] = qsur[1];
          --qn;
          if (release >= 0 && (qn == 0 || qfill[0] != release)) {
            // The weights of that fill are no longer read once these second layers are done.
            if (elect_one()) tc_commit(&sm.w_empty[release & 1]);
            __syncwarp();
            release = -1;
          }
          progress = true;
        }
      }
      if (feeding && qn < 2) {  // first layer of tile k
        const int st = k % kTcStages, b = k & 1;
        const bool ready = __shfl_sync(
            0xffffffffu, (int)(mbar_test_wait(&sm.full[st], (k / kTcStages) & 1) && group_free(k)), 0);
        if (ready) {
          const int it = *reinterpret_cast<volatile int*>(&sm.stage_item[st]);
          const int fill = *reinterpret_cast<volatile int*>(&sm.stage_fill[st]);
          const int head = *reinterpret_cast<volatile int*>(&sm.stage_head[st]);
          const int item_slot = *reinterpret_cast<volatile int*>(&sm.stage_slot[st]);
          const int item_tile = *reinterpret_cast<volatile int*>(&sm.stage_tile[st]);
          if (it < 0) {
            feeding = false;
            progress = true;
          } else if (fill < 0 || fill == waited_fill ||
                     __shfl_sync(0xffffffffu, (int)mbar_test_wait(&sm.w_full[fill & 1], (fill >> 1) & 1), 0)) {
            if (fill >= 0) waited_fill = fill;
            tc_fence_after();
            if (fill >= 0) {
              const uint64_t da = sdesc_sw128(smem_u32(sm.v[st]));
              const uint64_t db = sdesc_sw128(smem_u32(sm.w1[fill & 1]));
              const uint32_t t_main = tmem + b * 256;
              if (elect_one()) {
#pragma unroll
                for (int kk = 0; kk < 4; ++kk)  // K = 64 channels: 4 x K16, +32 bytes per step
                  tc_mma_ss(t_main, da + 2 * kk, db + 2 * kk, id1, kk > 0 ? 1u : 0u);
                tc_commit(&sm.empty[st]);
                tc_commit(&sm.d1_full[b]);
              }
            } else if (elect_one()) {  // a mean tile: no MMA, release the stage and stand in
              mbar_arrive(&sm.empty[st]);
              mbar_arrive(&sm.d1_full[b]);
            }
            __syncwarp();
            if (elect_one()) {
              sm.acc_item[b] = it;
              sm.acc_head[b] = head;
              sm.acc_slot[b] = item_slot;
              sm.acc_tile[b] = item_tile;
              mbar_arrive(&sm.d1_full[b]);  // releases acc_item / acc_head to the group
            }
            __syncwarp();
            if (fill >= 0) {
              if (cur_fill >= 0 && fill != cur_fill) {  // cur_fill has no more tiles
                if (qn == 0) {
                  if (elect_one()) tc_commit(&sm.w_empty[cur_fill & 1]);
                  __syncwarp();
                } else {
                  release = cur_fill;
                }
              }
              cur_fill = fill;
              qk[qn] = k;
              qfill[qn] = fill;
              qsur[qn] = sur_cnt[b];
              ++sur_cnt[b];
              ++qn;
            }
            last_kind[b] = fill >= 0 ? 1 : 0;
            if (fill < 0) ++mean_cnt[b];
            ++k;
            progress = true;
          }
        }
      }
      if (!feeding && qn == 0) break;
      if (progress) {
        t0 = 0;
        continue;
      }
      __nanosleep(32);  // leave the issue slots to the epilogue warps on this sub-partition
      if ((spin & 255u) == 0) {  // bounded: give up after kWaitLimitNs without progress
        if (*abort_flag) {
          ok = false;
          break;
        }
        const unsigned long long now = global_timer_ns();
        if (t0 == 0) {
          t0 = now;
        } else if (now - t0 > kWaitLimitNs) {
          if (lane == 0) {
            atomicOr(err, VP_DEVERR_WAIT_TIMEOUT);
            *abort_flag = 1;
          }
          ok = false;
          break;
        }
      }
    }
    // No more items: a stop for each group (tiles k and k + 1).
    for (int kk = k; ok && kk < k + kTcGroups; ++kk) {
      const int b = kk & 1;
      for (uint32_t sp = 1; !__shfl_sync(0xffffffffu, (int)group_free(kk), 0); ++sp) {
        __nanosleep(32);
        if ((sp & 255u) == 0) {
          const unsigned long long now = global_timer_ns();
          if (*abort_flag || (t0 != 0 && now - t0 > kWaitLimitNs)) {
            if (lane == 0 && !*abort_flag) {
              atomicOr(err, VP_DEVERR_WAIT_TIMEOUT);
              *abort_flag = 1;
            }
            ok = false;
            break;
          }
          if (t0 == 0) t0 = now;
        }
      }
      if (!ok) break;
      if (elect_one()) {
        sm.acc_item[b] = -1;
        mbar_arrive(&sm.d1_full[b]);
        mbar_arrive(&sm.d1_full[b]);
      }
      __syncwarp();
    }
    if (!ok) {
      if (elect_one()) {
        tc_commit(&sm.drain);
        for (int t = 0; t < 1000000 && !mbar_try_wait(&sm.drain, 0); ++t) {}
      }
      __syncwarp();
    }
  } else {
    // ------------------------------------------------------------ epilogue groups
    const int e = warp - 2;
    const int g = e / (4 * kTcParts), part = (e % (4 * kTcParts)) >> 2;
    const int gt = tid - 64 - kGroupThreads * g;  // 0 .. kGroupThreads - 1 within the group
    const int quarter = warp & 3;                 // TMEM lanes this warp may access
    const uint32_t t_grp = tmem + ((uint32_t)(quarter * 32) << 16) + g * 256;
    unsigned char* yblk = reinterpret_cast<unsigned char*>(sm.ys[e]);
    // This warp's share of a row: hidden-unit chunks [g0, g1) of 16 (first layer, H) and
    // output-column chunks [f0, f1) of 16 (second layer, y).
    const int g0 = part_begin(part, 8), g1 = part_begin(part + 1, 8);
    const int f0 = part_begin(kTcParts - 1 - part, 4), f1 = part_begin(kTcParts - part, 4);
    uint32_t sj = 0;  // surrogate tiles of this group
    bool ok = true;
    // The heads' vectors: all of them now, while the first tile's copies and MMAs run, or with
    // single items (few of a CTA's heads are ever used) each when a tile first needs it.
    const bool all_vec = batch > 1;
    int vec_slot = -1;  // with single items: the head (by slot) whose vectors this warp can read
    // A head's vectors by the group's warps: a component of c1 in lanes 0-15, of the rest in 16-31,
    // handed over through an mbarrier (a bounded wait, unlike a named barrier).
    uint32_t n_vec = 0;
    auto group_vectors = [&](int slot, int h) -> bool {
      const int u = (4 * part + quarter) * 16 + (lane & 15);
      if (lane < 16)
        head_c1(a, sm, vec_entry(g, n_vec), h, u);
      else
        head_out(a, sm, vec_entry(g, n_vec), h, u);
      vec_slot = slot;
      __syncwarp();
      if (elect_one()) mbar_arrive(&sm.vec_full[g]);
      __syncwarp();
      return mbar_wait_warp(&sm.vec_full[g], n_vec++ & 1, err, abort_flag);
    };
    if (all_vec) {
      for (int i = tid - 64; i < n_surr * 128; i += kGroupThreads * kTcGroups) {
        head_c1(a, sm, i >> 7, a.head_ids[s_first + (i >> 7)], i & 127);
        head_out(a, sm, i >> 7, a.head_ids[s_first + (i >> 7)], i & 127);
      }
      asm volatile("bar.sync 3, %0;" ::"n"(kGroupThreads * kTcGroups) : "memory");
    } else if (g == 0 && first_item < surr_items) {
      ok = group_vectors(first_item / T, a.head_ids[s_first + first_item / T]);
    }
    for (uint32_t j = 0;; ++j) {
      ok = ok && mbar_wait_warp(&sm.d1_full[g], j & 1, err, abort_flag);
      if (!ok) break;
      tc_fence_after();
      const int it = *reinterpret_cast<volatile int*>(&sm.acc_item[g]);
      if (it < 0) break;
      const int h = *reinterpret_cast<volatile int*>(&sm.acc_head[g]);
      const bool surr = it < surr_items;
      const int tile = *reinterpret_cast<volatile int*>(&sm.acc_tile[g]);  // a mean item spans kMeanRows rows
      const int slot = *reinterpret_cast<volatile int*>(&sm.acc_slot[g]);  // surrogate head slot: its vectors
      if (surr && !all_vec && slot != vec_slot && !group_vectors(slot, h)) break;
      const int entry = all_vec ? slot : vec_entry(g, n_vec - 1);
      const float* c1 = sm.c1[entry];
      const float* b2 = sm.b2[entry];
      const float* cx = sm.cx[entry];
      const uint32_t t_d1 = t_grp, t_d2 = t_grp + 128;
      if (surr) {
        // H = 2 GELU(D1 + c1) as bf16 pairs (the factor 2 is exact in bf16 and is taken out
        // of the second layer's results): chunk c of 16 hidden units (D1 columns 16 c ..) into 8
        // columns at the start of this warp's own D1 columns (64 part ..), which it has read by
        // then.  Each chunk's TMEM load is in flight while the chunk before it is computed.
        float vb[2][16];
        tmem_ld16(t_d1 + 16 * g0, vb[0]);
#pragma unroll
        for (int i = 0; i < kMaxGChunks; ++i) {
          const int c = g0 + i;
          if (c >= g1) break;
          tmem_wait_ld();
          if (c + 1 < g1) tmem_ld16(t_d1 + 16 * (c + 1), vb[(i + 1) & 1]);
          uint32_t hw[8];
#pragma unroll
          for (int q = 0; q < 8; ++q) {
            const float2 cc = *reinterpret_cast<const float2*>(&c1[16 * c + 2 * q]);
            const float2 x = gelu2_as2(fadd2(make_float2(vb[i & 1][2 * q], vb[i & 1][2 * q + 1]), cc));
            hw[q] = pack_bf16x2(x.x, x.y);
          }
          tmem_st8(t_d1 + 64 * part + 8 * i, hw);
        }
        tmem_wait_st();
        tc_fence_before();
        __syncwarp();
        if (elect_one()) {
          mbar_arrive(&sm.h_full[g]);
          tma_store_wait_read<0>();  // the last tile's store has read the staging block
        }
        __syncwarp();
        ok = mbar_wait_warp(&sm.d2_full[g], sj & 1, err, abort_flag);
        if (!ok) break;
        ++sj;
      }
      if (!surr) {
        // Broadcast(mean of V_h) straight to Y (no staging: a store pipeline two tiles deep
        // per SM would hold these pure-write tiles back): eight threads per row, each a 16-byte
        // chunk, so that a warp writes whole 128-byte rows.
        __syncwarp();
        if (elect_one()) mbar_arrive(&sm.taken[g]);  // this warp has read the item
        const int jc = gt & 7;
        const float4 m0 = reinterpret_cast<const float4*>(a.mean_v + h * 64)[2 * jc];
        const float4 m1 = reinterpret_cast<const float4*>(a.mean_v + h * 64)[2 * jc + 1];
        const uint4 val = make_uint4(pack_bf16x2(m0.x, m0.y), pack_bf16x2(m0.z, m0.w),
                                     pack_bf16x2(m1.x, m1.y), pack_bf16x2(m1.z, m1.w));
        for (int r = gt >> 3; r < kMeanRows; r += kGroupThreads / 8) {
          const int grow = tile * kMeanRows + r;
          if (grow < a.N) *(reinterpret_cast<uint4*>(a.y + ((size_t)grow * H + h) * 64) + jc) = val;
        }
        continue;
      }
      {
        // y = C + sigma(D2g + b2g) (.) (D2d + b2d) for chunk c of 16 output columns, from
        // D2' = 2 D2: sigma(u) = 1 / (1 + 2^(-log2(e) u)) with the exponent
        // -log2(e) / 2 D2g' + nbg, nbg = -log2(e) b2g held per head.
        tc_fence_after();
        const float kS = -0.5f * 1.4426950408889634f;
#pragma unroll
        for (int i = 0; i < kMaxFChunks; ++i) {
          const int c = f0 + i;
          if (c >= f1) break;
          float og[16], od[16];
          tmem_ld16(t_d2 + 16 * c, og);
          tmem_ld16(t_d2 + 64 + 16 * c, od);
          tmem_wait_ld();
          uint32_t yw[8];
#pragma unroll
          for (int q = 0; q < 8; ++q) {
            const int col = 16 * c + 2 * q;
            const float2 C = *reinterpret_cast<const float2*>(&cx[col]);
            const float2 nbg = *reinterpret_cast<const float2*>(&b2[col]);
            const float2 bd = *reinterpret_cast<const float2*>(&b2[64 + col]);
            const float2 ea = ffma2(make_float2(og[2 * q], og[2 * q + 1]), make_float2(kS, kS), nbg);
            const float2 den = fadd2(make_float2(fast_exp2(ea.x), fast_exp2(ea.y)), make_float2(1.f, 1.f));
            float2 sg;
            asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(sg.x) : "f"(den.x));
            asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(sg.y) : "f"(den.y));
            const float2 dl = ffma2(make_float2(od[2 * q], od[2 * q + 1]), make_float2(0.5f, 0.5f), bd);
            const float2 y2 = ffma2(sg, dl, C);
            yw[q] = pack_bf16x2(y2.x, y2.y);
          }
#pragma unroll
          for (int q = 0; q < 2; ++q) {  // 64-byte swizzle: chunk jc of row r sits at jc ^ ((r >> 1) & 3)
            const int jc = 2 * i + q;
            *reinterpret_cast<uint4*>(yblk + lane * 64 + ((jc ^ ((lane >> 1) & 3)) << 4)) =
                make_uint4(yw[4 * q], yw[4 * q + 1], yw[4 * q + 2], yw[4 * q + 3]);
          }
        }
        tc_fence_before();
      }
      fence_proxy_async_smem();
      __syncwarp();
      if (elect_one()) {
        tma_store_2d(&maps.y, yblk, h * 64 + 16 * f0, tile * kTcTile + quarter * 32);
        tma_store_commit();
      }
      __syncwarp();
    }
    if (elect_one()) tma_store_wait_all();
    __syncwarp();
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, kTcTmemCols);
  }
  // The mean heads folded into W_O's bias, a warp per output column (a launch of its own between
  // the router and the heads cost 4-5 us a layer); the columns from a counter, so that the CTAs
  // without items take them.
  if (a.wo_bias) {
    for (;;) {
      if (tid == 0) sm.first_item = (int)atomicAdd(a.fold_counter, (unsigned)(kTcThreads / 32));
      __syncthreads();
      const int n0 = sm.first_item;
      __syncthreads();
      if (n0 >= H * 64) break;
      if (n0 + warp < H * 64)
        wo_mean_fold_column(n0 + warp, H, a.w_o, a.b_o, a.mean_v, a.head_ids, m_first, s_first, a.wo_bias);
    }
  }
  // Once the full-attention grid has completed: its split groups, spread over all warps.
  pdl_wait();
  combine_split_heads(a, a.attn_ctas, warp * (int)gridDim.x + (int)blockIdx.x, (kTcThreads / 32) * (int)gridDim.x);
}

}  // namespace

size_t cheap_heads_tc_smem() { return sizeof(TcSmem) + 1024; }

cudaError_t launch_cheap_heads_tc(const HeadAttnArgs& a, int num_sms, cudaStream_t st) {
  TcMaps maps;
  cudaError_t e;
  const uint64_t H = (uint64_t)a.H;
  if ((e = make_tmap_bf16_2d(&maps.v, a.qkv, 3 * H * 64, (uint64_t)a.N, 3 * H * 64, 64, kTcTile)) !=
      cudaSuccess)
    return e;
  if ((e = make_tmap_bf16_2d(&maps.y, a.y, H * 64, (uint64_t)a.N, H * 64, 32, 32, 64)) != cudaSuccess)
    return e;
  // Layer-1 weights [H][64][128]: the value half is columns 0..63; layer 2 [H][64][64].
  if ((e = make_tmap_bf16_2d(&maps.g1, a.sw.g1_w, 128, H * 64, 128, 64, 64)) != cudaSuccess) return e;
  if ((e = make_tmap_bf16_2d(&maps.d1, a.sw.d1_w, 128, H * 64, 128, 64, 64)) != cudaSuccess) return e;
  if ((e = make_tmap_bf16_2d(&maps.g2, a.sw.g2_w, 64, H * 64, 64, 64, 64)) != cudaSuccess) return e;
  if ((e = make_tmap_bf16_2d(&maps.d2, a.sw.d2_w, 64, H * 64, 64, 64, 64)) != cudaSuccess) return e;
  const int smem = (int)cheap_heads_tc_smem();
  if ((e = cudaFuncSetAttribute(cheap_heads_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                smem)) != cudaSuccess)
    return e;
  return launch_pdl(cheap_heads_tc_kernel, dim3(num_sms), kTcThreads, smem, st, maps, a);
}

}  // namespace vp
