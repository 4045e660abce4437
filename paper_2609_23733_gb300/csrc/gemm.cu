// Dense projections of Algorithm 1 (QKV, W_O, FFN) on the sm_103a tensor cores:
//   out[M][N] = residual + scale (.) act(A[M][K] W[N][K]^T + bias)
// optionally with a LayerNorm of A's rows folded in (A W^T -> rstd (A W^T - mu c^T), see
// LinearArgs) and with the output rows' LayerNorm statistics as (mean, M2) per 128 columns.
// Persistent CTA pairs (clusters of two, cta_group::2), 256 x 256 output tiles: each CTA holds 128
// rows of A and 128 of W per 64-wide K block in a 5-stage TMA ring (128-byte swizzle, 32 KB a
// stage), so a K block takes 64 B per clock and SM from L2 where a CTA on its own, with 128 x 256
// tiles, takes 96 and has a third less look-ahead.  At 137,400 tokens against that design: QKV
// 529 -> 454 us (1,900 TFLOP/s), FFN-down 683 -> 607, FFN-up + GELU 709 -> 655, W_O with LayerScale
// and residual 235 -> 183; tensor-bound except W_O, which moves 0.84 GB.  tcgen05.mma (M=256, N=256, K=16, bf16 ->
// fp32) into one of two TMEM accumulators, so the epilogue of tile i overlaps the main loop of
// tile i+1.  The tiles of a last round that would use at most half of the pairs are cut into two
// 128-wide ones each (launch_linear).
// Warp roles per CTA: warp 0 TMA, warp 1 TMEM owner and (leader CTA) MMA issue, warps 2 ..
// epilogue (eight or sixteen, launch_linear): each owns a (32-row TMEM lane quarter, half or
// quarter of the columns) of the tile, one row per thread, the tile's bias and scale in shared
// memory (from global memory they cost an L2 round trip per chunk); per 32-column chunk it loads TMEM (the next chunk's load in flight while this one
// is processed), applies bias / GELU / LayerScale / residual, packs bf16 into a 128-byte-swizzled
// 32 x 64 staging block in shared memory and writes it with a TMA tensor store (clipped at the
// tensor edge).  The residual comes the same way: its blocks are loaded by TMA into the staging
// blocks while the tile's MMAs run, and added in place (read row by row from global memory, it
// took W_O's epilogue longer than the MMAs).
// Tiles are visited N-fastest so the pairs in flight share A rows and all of W in L2.
// A second instance (kSkip) leaves chosen 64-column K-blocks out: W_O with the mean heads
// folded into its bias (wo_mean_fold_kernel) skips their copies and MMAs, and with every block
// left out it is its epilogue alone.
#include <math.h>

#include "common.cuh"
#include "gemm_drain.h"
#include "internal.h"

namespace vp {

namespace {

constexpr int kBM = 256, kBK = 64;          // rows of the pair's tile, columns of a K block
constexpr int kTailN = 128;                 // width of a cut tile
constexpr int kABytes = kBM / 2 * kBK * 2;  // 16 KB: a CTA's half of A
constexpr int kBlkBytes = 32 * 64 * 2;      // a staging block: 32 rows x 64 columns

// kTileN = 256, or 128 for launches of narrow tiles alone (launch_linear): a stage is then 24 KB, and
// seven of them cover the copies' latency, which five 32-KB ones with half of B unused did not.
template <int kTileN>
struct GemmSmem {
  static constexpr int kStages = kTileN == 256 ? 5 : 7;
  static constexpr int kBlocks = kTileN / 16;  // staging blocks, shared out over the epilogue warps
  static constexpr uint32_t kTmemCols = 2 * kTileN;
  __nv_bfloat16 a[kStages][kBM / 2 * kBK];
  __nv_bfloat16 b[kStages][kTileN / 2 * kBK];
  __nv_bfloat16 stage[kBlocks][32 * 64];
  float vec[2][kTileN];     // the tile's bias, and its LayerScale or LN-fold column sums
  float4 stats[kTileN == 256 ? 1 : 128];  // half a 128-column block's row statistics (part_out)
  uint64_t full[kStages];   // leader's: both CTAs' copies of a stage have landed
  uint64_t empty[kStages];
  uint64_t acc_full[2];
  uint64_t acc_empty[2];    // leader's: both CTAs' epilogue warps have read the accumulator
  uint64_t res_full[kBlocks];
  uint64_t drain;
  uint32_t tmem_base;
  uint32_t skip_mask;  // K-blocks left out (LinearArgs::skip_ids)
  int abort_flag;
  uint32_t peer_abort;   // the other CTA's abort_flag, seen behind the cluster barrier at the end
  uint32_t res_asked[16], res_done[16];  // per epilogue warp: residual blocks asked for, stored
  uint32_t issued;       // K blocks whose copies this CTA's producer has issued
  uint32_t peer_issued;  // leader's: the other CTA's
};
static_assert(sizeof(GemmSmem<256>) <= 232448 && sizeof(GemmSmem<128>) <= 232448, "shared memory");

struct GemmParams {
  int M, N, K;
  const float* bias;
  int act;
  const float* scale;
  const __nv_bfloat16* residual;
  __nv_bfloat16* out;
  unsigned int* err;
  const float2* ln_part;
  const float* ln_c;
  float ln_eps;
  float2* part_out;
  int qk_cols;  // > 0: the first qk_cols columns are Q | K of a QKV projection (see LinearArgs)
  const float* qn_g;
  const float* qn_b;
  const float* kn_g;
  const float* kn_b;
  float qk_eps;
  const float2* rope_cs;
  int rope_npos, tok_per_view, patch_start, grid_w;
  const int32_t* tok_index;
  const int32_t* skip_ids;
  const int32_t* skip_off;
  int w_ready;  // LinearArgs::w_ready
  int full_units, units;  // units 0 .. full_units - 1 are whole tiles, the rest halves of tiles
};

// Unit u of the launch: the pair's rows from m0, columns [n0, n0 + w).
struct TileUnit {
  int m0, n0, w;
};
template <int kBN>
__device__ __forceinline__ TileUnit tile_unit(int u, int full_units, int n_tiles) {
  const bool cut = u >= full_units;
  const int t = cut ? full_units + ((u - full_units) >> 1) : u;
  const int mt = t / n_tiles, nt = t - mt * n_tiles;
  TileUnit r;
  r.m0 = mt * kBM;
  r.n0 = nt * kBN + (cut ? ((u - full_units) & 1) * kTailN : 0);
  r.w = cut ? kTailN : kBN;
  return r;
}

__device__ unsigned int g_linear_err;  // error word of calls without a workspace (vp_linear)

// After a failed wait in either CTA of a pair, called by all their threads: waits (bounded) until the
// operand copies that either producer has issued have landed, and the residual blocks asked for, and the
// MMAs issued have completed.
template <int kBN, bool kSkip, int kEpiWarps>
__device__ __noinline__ void drain_pair(int N, int K, int full_units) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  GemmSmem<kBN>& sm = *reinterpret_cast<GemmSmem<kBN>*>(smem_raw);
  constexpr uint32_t kStages = GemmSmem<kBN>::kStages;
  const int rank = (int)cluster_cta_rank(), pair = (int)(blockIdx.x >> 1), pairs = (int)(gridDim.x >> 1);
  const int n_tiles = (N + kBN - 1) / kBN, k_blocks = (K + kBK - 1) / kBK;
  if (threadIdx.x == 0 && rank == 1) st_cluster_u32(cluster_addr(&sm.peer_issued, 0), sm.issued);
  cluster_sync_all();
  if (rank == 0 && threadIdx.x == 0) {
#pragma unroll 1
    for (uint32_t s = 0; s < kStages; ++s) {
      const StageDrain d = stage_drain(sm.issued, sm.peer_issued, s, kStages);
      if (d.uses == 0) continue;
      const int unit_blocks = k_blocks - (kSkip ? __popc(sm.skip_mask) : 0);
      const TileUnit t = tile_unit<kBN>(pair + pairs * (int)(d.block / unit_blocks), full_units, n_tiles);
      const uint32_t half = kABytes + t.w / 2 * kBK * 2;
      if (d.fix > 0) mbar_arrive_expect_tx(&sm.full[s], half);
      if (d.fix < 0) mbar_complete_tx(&sm.full[s], half);
      for (int it = 0; it < 1000000 && !mbar_try_wait(&sm.full[s], (d.uses - 1) & 1); ++it) {}
    }
  }
  const int warp = warp_uniform_id();
  if (warp >= 2 && elect_one()) {
    constexpr uint32_t kBufs = GemmSmem<kBN>::kBlocks / kEpiWarps;
#pragma unroll 1
    for (uint32_t n = sm.res_done[warp - 2]; n < sm.res_asked[warp - 2]; ++n) {
      uint64_t* bar = &sm.res_full[(warp - 2) * kBufs + n % kBufs];
      for (int it = 0; it < 1000000 && !mbar_try_wait(bar, (n / kBufs) & 1); ++it) {}
    }
  }
  __syncwarp();
  if (rank == 0 && warp == 1) {
    if (elect_one()) {  // the lane that issued the MMAs
      tc_commit_pair(&sm.drain);
      for (int it = 0; it < 1000000 && !mbar_try_wait(&sm.drain, 0); ++it) {}
    }
    __syncwarp();
  }
  __syncthreads();
  cluster_sync_all();
}

// kSkip: the instance that leaves K-blocks out (GemmParams::skip_ids); the other instance has
// none of that bookkeeping.
template <bool kSkip, int kEpiWarps, bool kQk = false, int kBN = 256>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(64 + 32 * kEpiWarps, 1)
    gemm_kernel(const __grid_constant__ CUtensorMap tmap_a,
                const __grid_constant__ CUtensorMap tmap_b,
                const __grid_constant__ CUtensorMap tmap_b_cut,
                const __grid_constant__ CUtensorMap tmap_out,
                const __grid_constant__ CUtensorMap tmap_res, const __grid_constant__ GemmParams prm) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  using Smem = GemmSmem<kBN>;
  Smem& sm = *reinterpret_cast<Smem*>(smem_raw);
  constexpr int kStages = Smem::kStages, kBlocks = Smem::kBlocks;
  constexpr uint32_t kTmemCols = Smem::kTmemCols;
  constexpr int kParts = kEpiWarps / 4;        // column parts of a tile (epilogue warps per lane quarter)
  constexpr int kBufs = kBlocks / kEpiWarps;   // staging blocks of a warp = its 64-column groups
  const int M = prm.M, N = prm.N, K = prm.K;
  unsigned int* const err = prm.err ? prm.err : &g_linear_err;
  const int n_tiles = (N + kBN - 1) / kBN;
  const int k_blocks = (K + kBK - 1) / kBK;
  const int pair = (int)(blockIdx.x >> 1), pairs = (int)(gridDim.x >> 1);
  const int warp = warp_uniform_id(), lane = lane_id();
  const int rank = __shfl_sync(0xffffffffu, (int)cluster_cta_rank(), 0);
  volatile int* abort_flag = &sm.abort_flag;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(&sm.full[s], 1);
      mbar_init(&sm.empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&sm.acc_full[b], 1);
      mbar_init(&sm.acc_empty[b], 2 * kEpiWarps);
    }
    for (int b = 0; b < kBlocks; ++b) mbar_init(&sm.res_full[b], 1);
    mbar_init(&sm.drain, 1);
    sm.abort_flag = 0;
    sm.peer_abort = 0;
    fence_mbarrier_init();
    fence_proxy_async_smem();
    tma_prefetch_desc(&tmap_a);
    tma_prefetch_desc(&tmap_b);
    tma_prefetch_desc(&tmap_out);
    if (prm.residual) tma_prefetch_desc(&tmap_res);
  }
  if (warp == 1) {
    tmem_alloc_pair(&sm.tmem_base, kTmemCols);
    tmem_relinquish_pair();
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();  // both CTAs' barriers and TMEM are there
  tc_fence_after();
  // A weight that no kernel just before writes: the first stages' halves of B while that kernel
  // still runs.
  int early = 0;  // K blocks of the first unit whose B is on its way
  if (!kSkip && warp == 0 && prm.w_ready && pair < prm.units) {
    const TileUnit t = tile_unit<kBN>(pair, prm.full_units, n_tiles);
    early = min(kStages, k_blocks);
    for (int kb = 0; kb < early; ++kb) {
      const uint32_t full = cluster_addr(&sm.full[kb], 0);
      if (elect_one()) {
        if (rank == 0) mbar_arrive_expect_tx(&sm.full[kb], 2 * (kABytes + t.w / 2 * kBK * 2));
        tma_load_2d_pair(sm.b[kb], t.w != kBN ? &tmap_b_cut : &tmap_b, full, kb * kBK, t.n0 + rank * (t.w / 2));
      }
      __syncwarp();
    }
  }
  pdl_wait();
  pdl_launch();
  if (kSkip && threadIdx.x == 0) {
    uint32_t mask = 0;
    const int s0 = prm.skip_off[0], s1 = prm.skip_off[1];
    for (int i = s0; i < s1; ++i) mask |= 1u << (prm.skip_ids[i] & 31);
    sm.skip_mask = mask;
  }
  if (kSkip) __syncthreads();
  const uint32_t tmem = __shfl_sync(0xffffffffu, sm.tmem_base, 0);
  // K-blocks left out, and whether that is all of them (A W^T is then 0).
  const uint32_t skip = kSkip ? sm.skip_mask : 0u;
  const bool acc_zero = kSkip && skip != 0 && __popc(skip & (k_blocks >= 32 ? 0xffffffffu : (1u << k_blocks) - 1u)) == k_blocks;

  if (warp == 0) {
    // TMA producer of this CTA's halves: converged warp (warp-uniform coordinates), one elected
    // lane issues.  Both CTAs' copies complete on the leader's barrier, which expects them all.
    uint32_t lc = 0;
    bool ok = true;
    for (int u = pair; u < prm.units && ok; u += pairs) {
      const TileUnit t = tile_unit<kBN>(u, prm.full_units, n_tiles);
      const bool cut = t.w != kBN;
      const int row_a = t.m0 + rank * (kBM / 2), row_b = t.n0 + rank * (t.w / 2);
      const uint32_t bytes = 2 * (kABytes + t.w / 2 * kBK * 2);
      for (int kb = 0; kb < k_blocks; ++kb) {
        if (kSkip && ((skip >> kb) & 1u)) continue;
        const int st = lc % kStages;
        ok = mbar_wait_warp(&sm.empty[st], ((lc / kStages) & 1) ^ 1, err, abort_flag);
        if (!ok) break;
        const uint32_t full = cluster_addr(&sm.full[st], 0);
        const bool b_sent = u == pair && kb < early;
        if (elect_one()) {
          if (rank == 0 && !b_sent) mbar_arrive_expect_tx(&sm.full[st], bytes);
          tma_load_2d_pair(sm.a[st], &tmap_a, full, kb * kBK, row_a);
          if (!b_sent) tma_load_2d_pair(sm.b[st], cut ? &tmap_b_cut : &tmap_b, full, kb * kBK, row_b);
        }
        __syncwarp();
        ++lc;
      }
    }
    if (lane == 0) sm.issued = lc;
  } else if (warp == 1) {
    // MMA issuer (leader): converged warp; the elected lane (always the lowest, so the same one)
    // issues the MMAs and the commits that track them, which arrive in both CTAs.
    const uint32_t id_full = idesc_bf16(kBM, kBN, 0, 0), id_cut = idesc_bf16(kBM, kTailN, 0, 0);
    uint32_t lc = 0, i = 0;
    bool ok = true;
    for (int u = pair; rank == 0 && u < prm.units && ok; u += pairs, ++i) {
      const uint32_t idesc = u >= prm.full_units ? id_cut : id_full;
      const uint32_t ab = i & 1;
      ok = mbar_wait_warp(&sm.acc_empty[ab], ((i >> 1) & 1) ^ 1, err, abort_flag);
      if (!ok) break;
      tc_fence_after();
      const uint32_t d = tmem + ab * kBN;
      bool first = true;  // the tile's first MMA overwrites the accumulator
      for (int kb = 0; kb < k_blocks; ++kb) {
        if (kSkip && ((skip >> kb) & 1u)) continue;
        const int st = lc % kStages;
        ok = mbar_wait_warp(&sm.full[st], (lc / kStages) & 1, err, abort_flag);
        if (!ok) break;
        tc_fence_after();
        const uint64_t da = sdesc_sw128(smem_u32(sm.a[st]));
        const uint64_t db = sdesc_sw128(smem_u32(sm.b[st]));
        if (elect_one()) {
#pragma unroll
          for (int kk = 0; kk < 4; ++kk)
            tc_mma_ss_pair(d, da + 2 * kk, db + 2 * kk, idesc, ((kSkip ? !first : kb > 0) || kk > 0) ? 1u : 0u);
          tc_commit_pair(&sm.empty[st]);
        }
        __syncwarp();
        first = false;
        ++lc;
      }
      if (!ok) break;
      if (elect_one()) tc_commit_pair(&sm.acc_full[ab]);
      __syncwarp();
    }
  } else {
    const int e = warp - 2;                 // epilogue warp
    const int quarter = warp & 3;           // TMEM lane quarter
    const int part = e >> 2;                // column part of the tile
    const uint32_t t_lane = tmem + ((uint32_t)(quarter * 32) << 16);
    unsigned char* stg = reinterpret_cast<unsigned char*>(&sm.stage[e * kBufs][0]);
    uint64_t* res_bar = &sm.res_full[e * kBufs];
    const uint32_t acc_empty0 = cluster_addr(&sm.acc_empty[0], 0);
    auto epi_sync = []() { asm volatile("bar.sync 1, %0;" ::"n"(32 * kEpiWarps) : "memory"); };
    // The same barrier, and whether p held on every epilogue thread: the warps leave the loop
    // together when a wait of one of them gave up, so that none is left at a barrier.
    auto epi_all = [](bool p) -> bool {
      uint32_t r;
      asm volatile(
          "{\n\t.reg .pred pi, po;\n\t"
          "setp.ne.u32 pi, %1, 0;\n\t"
          "bar.red.and.pred po, 1, %2, pi;\n\t"
          "selp.u32 %0, 1, 0, po;\n\t}"
          : "=r"(r)
          : "r"((uint32_t)p), "n"(32 * kEpiWarps)
          : "memory");
      return r != 0;
    };
    bool alive = true;
    if (acc_zero) {
      // Every K-block is left out, so no MMA writes the accumulators: zero this thread's
      // columns of both once, and every tile then reads A W^T = 0.
      float z[32];
#pragma unroll
      for (int k = 0; k < 32; ++k) z[k] = 0.f;
#pragma unroll
      for (int q = 0; q < kBN / 16 / kParts; ++q) tmem_st32(t_lane + (part * (kBN / 16 / kParts) + q) * 32, z);
      tmem_wait_st();
      // a cut tile's columns are read by other warps of the lane quarter than zeroed them
      tc_fence_before();
      epi_sync();
      tc_fence_after();
    }
    if (elect_one()) sm.res_asked[e] = 0;
    uint32_t i = 0, nst = 0;  // units, blocks stored
    for (int u = pair; u < prm.units; u += pairs, ++i) {
      const TileUnit t = tile_unit<kBN>(u, prm.full_units, n_tiles);
      const uint32_t ab = i & 1;
      // This warp's columns of the tile: n_grp groups of 64 from pcol0.  A cut tile's two groups
      // go to the first two parts, or both to the first one where a thread needs a whole
      // 128-column block (part_out, which runs with two parts).
      const bool cut = t.w != kBN;
      const bool both = cut && kParts == 2 && prm.part_out;
      const int n_grp = !cut ? kBufs : (both ? (part == 0 ? 2 : 0) : (part < 2 ? 1 : 0));
      const int pcol0 = t.n0 + (both ? 0 : part * (!cut ? kBN / kParts : 64));
      const int row0 = t.m0 + rank * (kBM / 2) + quarter * 32;
      const int row = row0 + lane;
      const bool row_ok = row < M;
      // The tile's residual blocks into the staging blocks (once the stores before have read
      // them) while the tile's MMAs run.
      if (prm.residual && alive) {
        if (elect_one()) {
          tma_store_wait_read<0>();
          for (int gi = 0; gi < n_grp; ++gi) {
            if (pcol0 + 64 * gi < N) {
              const int buf = (nst + gi) % kBufs;
              mbar_arrive_expect_tx(&res_bar[buf], kBlkBytes);
              tma_load_2d(stg + buf * kBlkBytes, &tmap_res, &res_bar[buf], pcol0 + 64 * gi, row0);
              sm.res_asked[(threadIdx.x >> 5) - 2] = nst + gi + 1;
            }
          }
        }
        __syncwarp();
      }
      // The tile's bias and scale (or LN-fold column sums) into shared memory, a column per
      // thread: read per chunk from global memory they cost an L2 round trip each.
      {
        const int et = (int)threadIdx.x - 64, col = t.n0 + et;
        const bool in = et < t.w && col < N;
        const float* second = prm.scale ? prm.scale : prm.ln_c;
        const float v0 = in && prm.bias ? prm.bias[col] : 0.f;
        const float v1 = in && second ? second[col] : 0.f;
        if (!epi_all(alive)) break;  // every warp is done with the previous tile's
        if (et < kBN) {
          sm.vec[0][et] = v0;
          sm.vec[1][et] = v1;
        }
        epi_sync();
      }
      // Folded LayerNorm: this row's mean and 1 / sqrt(var + eps) from the (mean, M2) of its
      // 128-column blocks (equal counts: M2 = sum M2_b + 128 sum (mean_b - mean)^2).  The
      // first eight blocks (K = 1,024) are loaded before the accumulator wait.
      float ln_mu = 0.f, ln_rstd = 1.f;
      float4 lnp[4];
      const int nb = K >> 7;  // even (K % 256 == 0)
      const float4* lpp = reinterpret_cast<const float4*>(prm.ln_part + (size_t)row * nb);
      if (prm.ln_part && row_ok) {
#pragma unroll
        for (int b = 0; b < 4; ++b)
          if (2 * b < nb) lnp[b] = lpp[b];
      }
      alive = mbar_wait_warp(&sm.acc_full[ab], (i >> 1) & 1, err, abort_flag);
      if (!alive) {
        if (kBN == 128 && prm.part_out) asm volatile("bar.sync %0, 64;" ::"r"(2 + quarter) : "memory");
        continue;
      }
      tc_fence_after();
      // The accumulator goes back to the leader's MMA warp once this warp has read it.
      auto release_acc = [&]() {
        tc_fence_before();
        __syncwarp();
        if (elect_one()) mbar_arrive_cluster(acc_empty0 + ab * 8);
      };
      if (n_grp == 0) {
        release_acc();
        continue;
      }
      if (prm.ln_part && row_ok) {
        float sm_ = 0.f;
#pragma unroll
        for (int b = 0; b < 4; ++b)
          if (2 * b < nb) sm_ += lnp[b].x + lnp[b].z;
        for (int b = 4; 2 * b < nb; ++b) {
          const float4 p4 = lpp[b];
          sm_ += p4.x + p4.z;
        }
        ln_mu = sm_ / (float)nb;
        float m2 = 0.f;
#pragma unroll
        for (int b = 0; b < 4; ++b) {
          if (2 * b < nb) {
            const float d0 = lnp[b].x - ln_mu, d1 = lnp[b].z - ln_mu;
            m2 += lnp[b].y + lnp[b].w + 128.f * (d0 * d0 + d1 * d1);
          }
        }
        for (int b = 4; 2 * b < nb; ++b) {
          const float4 p4 = lpp[b];
          const float d0 = p4.x - ln_mu, d1 = p4.z - ln_mu;
          m2 += p4.y + p4.w + 128.f * (d0 * d0 + d1 * d1);
        }
        ln_rstd = rsqrtf(m2 / (float)K + prm.ln_eps);
      }
      float cmean[4] = {}, cm2[4] = {};  // output statistics per 32-column chunk (part_out)
      const uint32_t tcol = t_lane + ab * kBN + (pcol0 - t.n0);
      // Bias, or the folded LayerNorm rstd (acc - mu c) + bias', on one 32-column chunk.
      auto bias_fold = [&](float* x, int col0) {
        const float4* bv = reinterpret_cast<const float4*>(&sm.vec[0][col0 - t.n0]);
        if (prm.ln_part) {  // rstd (acc - mu c) + bias'
          const float4* cv = reinterpret_cast<const float4*>(&sm.vec[1][col0 - t.n0]);
          const float2 nmu = make_float2(-ln_mu, -ln_mu), rs = make_float2(ln_rstd, ln_rstd);
#pragma unroll
          for (int q = 0; q < 8; ++q) {
            const float4 c4 = cv[q], b4 = bv[q];
            const float2 a0 = ffma2(rs, ffma2(nmu, make_float2(c4.x, c4.y),
                                              make_float2(x[4 * q], x[4 * q + 1])),
                                    make_float2(b4.x, b4.y));
            const float2 a1 = ffma2(rs, ffma2(nmu, make_float2(c4.z, c4.w),
                                              make_float2(x[4 * q + 2], x[4 * q + 3])),
                                    make_float2(b4.z, b4.w));
            x[4 * q] = a0.x;
            x[4 * q + 1] = a0.y;
            x[4 * q + 2] = a1.x;
            x[4 * q + 3] = a1.y;
          }
        } else if (prm.bias) {
#pragma unroll
          for (int q = 0; q < 8; ++q) {
            const float4 b4 = bv[q];
            const float2 a0 = fadd2(make_float2(x[4 * q], x[4 * q + 1]), make_float2(b4.x, b4.y));
            const float2 a1 = fadd2(make_float2(x[4 * q + 2], x[4 * q + 3]), make_float2(b4.z, b4.w));
            x[4 * q] = a0.x;
            x[4 * q + 1] = a0.y;
            x[4 * q + 2] = a1.x;
            x[4 * q + 3] = a1.y;
          }
        }
      };
      // A 64-column block of the row (row = lane, 128 bytes) lies in the 128-byte swizzle of the
      // output tensor map: 16-byte chunk q of row r sits at chunk q ^ (r & 7).
      // Before the first write to it: its last store has read it (with a residual: seen to above).
      auto block_begin = [&]() -> unsigned char* {
        unsigned char* buf = stg + (nst % kBufs) * kBlkBytes;
        // The elected lane (lane 0, the lowest) owns this warp's bulk stores and their groups.
        if (!prm.residual && nst >= kBufs && elect_one()) tma_store_wait_read<kBufs - 1>();
        __syncwarp();
        return buf + lane * 128;
      };
      // 32 columns (chunks 4 hc .. 4 hc + 3 of the row), packed to bf16.
      auto block_put = [&](unsigned char* brow, const float* x, int hc) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          uint4 v;
          v.x = pack_bf16x2(x[8 * q + 0], x[8 * q + 1]);
          v.y = pack_bf16x2(x[8 * q + 2], x[8 * q + 3]);
          v.z = pack_bf16x2(x[8 * q + 4], x[8 * q + 5]);
          v.w = pack_bf16x2(x[8 * q + 6], x[8 * q + 7]);
          *reinterpret_cast<uint4*>(brow + (((4 * hc + q) ^ (lane & 7)) << 4)) = v;
        }
      };
      auto block_store = [&](int col0) {
        fence_proxy_async_smem();
        __syncwarp();
        if (elect_one()) {
          tma_store_2d(&tmap_out, stg + (nst % kBufs) * kBlkBytes, col0, row0);
          tma_store_commit();
        }
        ++nst;
      };
      if (kQk && pcol0 < prm.qk_cols) {
        // Q or K columns of a QKV projection with qk-norm and / or 2-D RoPE: whole heads
        // (64 columns, two chunks) at a time.
        const bool is_q = pcol0 < (prm.qk_cols >> 1);
        const float* ng = is_q ? prm.qn_g : prm.kn_g;
        const float* nbv = is_q ? prm.qn_b : prm.kn_b;
        int py = 0, px = 0;  // the row's position inside its view
        if (prm.rope_cs) {
          const int tok = prm.tok_index && row_ok ? prm.tok_index[row] : row;
          const int t = tok % prm.tok_per_view - prm.patch_start;
          if (t >= 0) {
            py = t / prm.grid_w + 1;
            px = t - (py - 1) * prm.grid_w + 1;
          }
        }
#pragma unroll 1
        for (int hh = 0; hh < n_grp; ++hh) {
          float x[64];
          tmem_ld32(tcol + 64 * hh, x);
          tmem_ld32(tcol + 64 * hh + 32, x + 32);
          tmem_wait_ld();
          if (hh == n_grp - 1) release_acc();
          const int col0 = pcol0 + 64 * hh;
          bias_fold(x, col0);
          bias_fold(x + 32, col0 + 32);
          if (ng) {  // LayerNorm over the head's 64 channels
            float2 s2 = make_float2(0.f, 0.f);
#pragma unroll
            for (int k = 0; k < 32; ++k) s2 = fadd2(s2, make_float2(x[2 * k], x[2 * k + 1]));
            const float mean = (s2.x + s2.y) * (1.f / 64.f);
            float2 q2 = make_float2(0.f, 0.f);
#pragma unroll
            for (int k = 0; k < 32; ++k) {
              const float2 dd = fadd2(make_float2(x[2 * k], x[2 * k + 1]), make_float2(-mean, -mean));
              q2 = ffma2(dd, dd, q2);
            }
            const float rstd = rsqrtf((q2.x + q2.y) * (1.f / 64.f) + prm.qk_eps);
            const float2 nm = make_float2(-mean * rstd, -mean * rstd), rs = make_float2(rstd, rstd);
#pragma unroll
            for (int q = 0; q < 16; ++q) {
              const float4 g4 = reinterpret_cast<const float4*>(ng)[q];
              const float4 b4 = reinterpret_cast<const float4*>(nbv)[q];
              const float2 a0 = ffma2(ffma2(make_float2(x[4 * q], x[4 * q + 1]), rs, nm),
                                      make_float2(g4.x, g4.y), make_float2(b4.x, b4.y));
              const float2 a1 = ffma2(ffma2(make_float2(x[4 * q + 2], x[4 * q + 3]), rs, nm),
                                      make_float2(g4.z, g4.w), make_float2(b4.z, b4.w));
              x[4 * q] = a0.x;
              x[4 * q + 1] = a0.y;
              x[4 * q + 2] = a1.x;
              x[4 * q + 3] = a1.y;
            }
          }
          if (prm.rope_cs) {  // channels [0, 32) turn with the row, [32, 64) with the column
#pragma unroll
            for (int ax = 0; ax < 2; ++ax) {
              const float4* cs = reinterpret_cast<const float4*>(prm.rope_cs) + (ax ? px : py);
#pragma unroll
              for (int q = 0; q < 8; ++q) {  // frequencies 2q, 2q + 1: (cos, sin) pairs
                const float4 t4 = cs[q * prm.rope_npos];
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                  const int i = 32 * ax + 2 * q + e;
                  const float c = e ? t4.z : t4.x, sn = e ? t4.w : t4.y;
                  const float a = x[i], b = x[i + 16];
                  x[i] = fmaf(a, c, -b * sn);
                  x[i + 16] = fmaf(b, c, a * sn);
                }
              }
            }
          }
          if (col0 < N) {
            unsigned char* brow = block_begin();
            block_put(brow, x, 0);
            block_put(brow, x + 32, 1);
            block_store(col0);
          }
        }
        continue;
      }
      float v[2][32];
      tmem_ld32(tcol, v[0]);
      tmem_wait_ld();
      unsigned char* brow = nullptr;
#pragma unroll
      for (int cc = 0; cc < 2 * kBufs; ++cc) {
        if (cc >= 2 * n_grp) break;
        if (cc + 1 < 2 * n_grp) tmem_ld32(tcol + 32 * (cc + 1), v[(cc + 1) & 1]);  // in flight meanwhile
        float* x = v[cc & 1];
        const int col0 = pcol0 + cc * 32;
        const bool live = pcol0 + 64 * (cc >> 1) < N;  // the 64-column block has columns to store
        if (live) {
          if ((cc & 1) == 0) {
            brow = block_begin();
            if (prm.residual &&
                !mbar_wait_warp(&res_bar[nst % kBufs], (nst / kBufs) & 1, err, abort_flag)) {
              alive = false;
              break;
            }
          }
          // Bias, GELU, LayerScale and residual on column pairs (packed f32x2 arithmetic).
          bias_fold(x, col0);
          if (!kQk && prm.act == VP_ACT_GELU) {
#pragma unroll
            for (int k = 0; k < 16; ++k) {
              const float2 gk = gelu_as2(make_float2(x[2 * k], x[2 * k + 1]));
              x[2 * k] = gk.x;
              x[2 * k + 1] = gk.y;
            }
          }
          if (!kQk && prm.scale) {
#pragma unroll
            for (int q = 0; q < 8; ++q) {
              const float4 s4 = reinterpret_cast<const float4*>(&sm.vec[1][col0 - t.n0])[q];
              const float2 a0 = fmul2(make_float2(x[4 * q], x[4 * q + 1]), make_float2(s4.x, s4.y));
              const float2 a1 = fmul2(make_float2(x[4 * q + 2], x[4 * q + 3]), make_float2(s4.z, s4.w));
              x[4 * q] = a0.x;
              x[4 * q + 1] = a0.y;
              x[4 * q + 2] = a1.x;
              x[4 * q + 3] = a1.y;
            }
          }
          if (!kQk && prm.residual) {  // rows and columns past the edge were filled with zeros
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              const uint4 ru = *reinterpret_cast<const uint4*>(brow + (((4 * (cc & 1) + q) ^ (lane & 7)) << 4));
              const uint32_t uw[4] = {ru.x, ru.y, ru.z, ru.w};
#pragma unroll
              for (int k = 0; k < 4; ++k) {
                const float2 a = fadd2(make_float2(x[8 * q + 2 * k], x[8 * q + 2 * k + 1]),
                                       make_float2(bf16_lo(uw[k]), bf16_hi(uw[k])));
                x[8 * q + 2 * k] = a.x;
                x[8 * q + 2 * k + 1] = a.y;
              }
            }
          }
          if (!kQk && kParts == 2 && prm.part_out) {  // chunk mean and M2 (two passes over registers)
            float2 s2 = make_float2(0.f, 0.f);
#pragma unroll
            for (int k = 0; k < 16; ++k) s2 = fadd2(s2, make_float2(x[2 * k], x[2 * k + 1]));
            const float cm = (s2.x + s2.y) * (1.f / 32.f);
            float2 q2 = make_float2(0.f, 0.f);
#pragma unroll
            for (int k = 0; k < 16; ++k) {
              const float2 dd = fadd2(make_float2(x[2 * k], x[2 * k + 1]), make_float2(-cm, -cm));
              q2 = ffma2(dd, dd, q2);
            }
            cmean[cc] = cm;
            cm2[cc] = q2.x + q2.y;
          }
          block_put(brow, x, cc & 1);
          if (cc & 1) block_store(pcol0 + 64 * (cc >> 1));
        }
        tmem_wait_ld();
        if (cc + 2 == 2 * n_grp) release_acc();  // the last chunk is in registers
      }
      if (!kQk && kParts == 2 && prm.part_out) {  // this row's (mean, M2) of a 128-column block
        float c2 = cmean[2], c3 = cmean[3], q2 = cm2[2], q3 = cm2[3];
        if (kBN == 128) {  // the block's second half is the other warp's of this lane quarter
          float4* st4 = &sm.stats[quarter * 32 + lane];
          if (part == 1) *st4 = make_float4(cmean[0], cmean[1], cm2[0], cm2[1]);
          asm volatile("bar.sync %0, 64;" ::"r"(2 + quarter) : "memory");
          const float4 o = *st4;
          c2 = o.x;
          c3 = o.y;
          q2 = o.z;
          q3 = o.w;
        }
        if (row_ok && pcol0 < N && (kBN == 256 || part == 0)) {
          const float mb = 0.25f * (cmean[0] + cmean[1] + c2 + c3);
          float m2 = cm2[0] + cm2[1] + q2 + q3;
          m2 += 32.f * (cmean[0] - mb) * (cmean[0] - mb);
          m2 += 32.f * (cmean[1] - mb) * (cmean[1] - mb);
          m2 += 32.f * (c2 - mb) * (c2 - mb);
          m2 += 32.f * (c3 - mb) * (c3 - mb);
          prm.part_out[(size_t)row * (N >> 7) + (pcol0 >> 7)] = make_float2(mb, m2);
        }
      }
    }
    if (elect_one()) {
      sm.res_done[(threadIdx.x >> 5) - 2] = nst;
      tma_store_wait_read<0>();  // the staging blocks outlive the reads
    }
    __syncwarp();
  }

  tc_fence_before();
  __syncthreads();
  if (threadIdx.x == 0 && sm.abort_flag) st_cluster_u32(cluster_addr(&sm.peer_abort, cluster_cta_rank() ^ 1), 1u);
  cluster_sync_all();  // neither CTA leaves while the other uses its shared memory or TMEM
  if (sm.abort_flag || sm.peer_abort) drain_pair<kBN, kSkip, kEpiWarps>(prm.N, prm.K, prm.full_units);
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc_pair(tmem, kTmemCols);
  }
}

// RoPE angles in double precision: (cos, sin)(p base^(-i / 16)) at table[i / 2][p][i % 2]: the rows of
// a warp stand at neighbouring positions, so its 16-byte loads of one frequency pair lie side by
// side (with the pairs of a position side by side, a load took 32 cache lines and the epilogue set
// the time: QKV with qk-norm at 43,968 tokens 189 -> 163 us).
__global__ void rope_table_kernel(int max_pos, double base, float2* table) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  const int p = k >> 4, i = k & 15;
  double sn, cs;
  sincos((double)p * pow(base, -(double)i / 16.0), &sn, &cs);
  pdl_wait();
  pdl_launch();
  if (k >= (max_pos + 1) * 16) return;
  table[((i >> 1) * (max_pos + 1) + p) * 2 + (i & 1)] = make_float2((float)cs, (float)sn);
}

}  // namespace

namespace {

// A warp per output column of W_O.
__global__ void wo_mean_fold_kernel(int D, int H, const __nv_bfloat16* w_o, const float* b_o,
                                    const float* mean_v, const int32_t* head_ids,
                                    const int32_t* offsets, float* bias_out) {
  const int n = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
  pdl_wait();
  pdl_launch();
  if (n >= D) return;  // whole warps
  wo_mean_fold_column(n, H, w_o, b_o, mean_v, head_ids, offsets[0], offsets[1], bias_out);
}

}  // namespace

cudaError_t launch_rope_table(int max_pos, float base, float2* table, cudaStream_t st) {
  const int n = (max_pos + 1) * 16;
  return launch_pdl(rope_table_kernel, dim3((n + 255) / 256), 256, 0, st, max_pos, (double)base, table);
}

cudaError_t launch_wo_mean_fold(int D, int H, const __nv_bfloat16* w_o, const float* b_o,
                                const float* mean_v, const int32_t* head_ids,
                                const int32_t* offsets, float* bias_out, cudaStream_t st) {
  const int threads = 256, blocks = (D * 32 + threads - 1) / threads;
  return launch_pdl(wo_mean_fold_kernel, dim3(blocks), threads, 0, st, D, H, w_o, b_o, mean_v, head_ids,
                    offsets, bias_out);
}

cudaError_t launch_linear(const LinearArgs& a, int num_sms, cudaStream_t st) {
  CUtensorMap ta, tb, tb_cut, to, tr;
  cudaError_t e = make_tmap_bf16_2d(&ta, a.A, (uint64_t)a.K, (uint64_t)a.M, (uint64_t)a.K, kBK, kBM / 2);
  if (e != cudaSuccess) return e;
  e = make_tmap_bf16_2d(&to, a.out, (uint64_t)a.N, (uint64_t)a.M, (uint64_t)a.N, 64, 32);
  if (e != cudaSuccess) return e;
  tr = to;
  if (a.residual && a.residual != a.out) {
    e = make_tmap_bf16_2d(&tr, a.residual, (uint64_t)a.N, (uint64_t)a.M, (uint64_t)a.N, 64, 32);
    if (e != cudaSuccess) return e;
  }
  if ((a.ln_part && (a.K % 256 != 0 || !a.ln_c || !a.bias)) ||
      (a.part_out && a.N % 128 != 0))
    return cudaErrorInvalidValue;
  const bool qk = a.qk_cols > 0;
  if (a.skip_ids && (!a.skip_off || a.ln_part || qk || a.K % kBK != 0 || a.K > 32 * kBK))
    return cudaErrorInvalidValue;
  if (qk && (a.qk_cols % 256 != 0 || a.qk_cols > a.N || a.act != VP_ACT_NONE || a.scale ||
             a.residual || a.part_out || (!a.qn_g != !a.qn_b) || (!a.kn_g != !a.kn_b) ||
             (a.rope_cs && (a.tok_per_view < 1 || a.grid_w < 1 || a.patch_start < 0))))
    return cudaErrorInvalidValue;
  // Whole rounds of 256 x 256 tiles over the pairs; a last round that at most half of the pairs
  // would work on is cut into tiles of half the width (10,992 x 1,024 from K = 4,096: 172 tiles
  // on 76 pairs).  Where that is all there is, the instance of 128-wide tiles runs (1,044 rows,
  // K = 4,096: 20 tiles become 40; 28.0 us with 128 x 256 tiles of single CTAs, 16.5 with cut tiles,
  // 14.4 with this instance).
  const int pairs_max = max(1, num_sms / 2);
  const int m_tiles = (a.M + kBM - 1) / kBM;
  const int tiles = m_tiles * ((a.N + 255) / 256);
  const int left = tiles % pairs_max;
  const bool narrow = !qk && 2 * tiles <= pairs_max;
  const int full_units = narrow ? m_tiles * ((a.N + 127) / 128) : 2 * left <= pairs_max ? tiles - left : tiles;
  const int units = narrow ? full_units : full_units + 2 * (tiles - full_units);
  e = make_tmap_bf16_2d(&tb, a.W, (uint64_t)a.K, (uint64_t)a.N, (uint64_t)a.K, kBK, narrow ? 64 : 128);
  if (e != cudaSuccess) return e;
  tb_cut = tb;
  if (full_units < units && !narrow) {
    e = make_tmap_bf16_2d(&tb_cut, a.W, (uint64_t)a.K, (uint64_t)a.N, (uint64_t)a.K, kBK, kTailN / 2);
    if (e != cudaSuccess) return e;
  }
  GemmParams prm{a.M,     a.N,   a.K,   a.bias,      a.act,  a.scale,   a.residual,
                 a.out,   a.err, a.ln_part, a.ln_c, a.ln_eps, a.part_out,
                 qk ? a.qk_cols : 0, a.qn_g, a.qn_b, a.kn_g, a.kn_b, a.qk_eps, a.rope_cs,
                 a.rope_npos, a.tok_per_view, a.patch_start, a.grid_w, a.tok_index, a.skip_ids, a.skip_off,
                 a.w_ready ? 1 : 0, full_units, units};
  const int grid = 2 * min(pairs_max, units);
  auto launch = [&](auto kernel, int epi_warps, size_t smem_bytes = sizeof(GemmSmem<256>)) -> cudaError_t {
    const int smem = (int)smem_bytes;
    cudaError_t le = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (le != cudaSuccess) return le;
    prof_before(VP_KERNEL_GEMM, st);
    le = launch_pdl(kernel, dim3(grid), 64 + 32 * epi_warps, smem, st, ta, tb, tb_cut, to, tr, prm);
    prof_after(st);
    return le;
  };
  if (narrow)
    return a.skip_ids ? launch(gemm_kernel<true, 8, false, 128>, 8, sizeof(GemmSmem<128>))
                      : launch(gemm_kernel<false, 8, false, 128>, 8, sizeof(GemmSmem<128>));
  // Sixteen epilogue warps (64 columns of a row per thread, one staging block each) where the
  // epilogue is what a tile waits for: GELU (137,400 x 4,096 from K = 1,024: 668 us with eight
  // warps, 655 with sixteen), and a single round, whose epilogue no next tile covers (1,044 x
  // 1,024 with residual 15.4 -> 12.2 us).  Eight elsewhere (128 columns, two blocks, so that the
  // next tile's residual loads start earlier: 137,400 x 1,024 with residual 183 us against 189,
  // x 3,072 454 against 462); qk-norm and part_out need a thread to hold whole heads or blocks.
  const bool sixteen = !a.part_out && (a.act == VP_ACT_GELU || units <= pairs_max);
  if (qk) return launch(gemm_kernel<false, 8, true>, 8);
  if (a.skip_ids) return sixteen ? launch(gemm_kernel<true, 16>, 16) : launch(gemm_kernel<true, 8>, 8);
  return sixteen ? launch(gemm_kernel<false, 16>, 16) : launch(gemm_kernel<false, 8>, 8);
}

}  // namespace vp
