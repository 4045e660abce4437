// The routed head outputs Y of one layer (Algorithm 1, step 2): full-mode heads in
// attn_full_kernel, then the surrogate (§4.3) and mean heads queued behind it with
// programmatic dependent launch (heads_cheap_tc.cu).  The full-attention CTAs signal their
// dependents as soon as they start, so cheap-head CTAs take each SM as soon as a
// full-attention CTA retires.  The cheap kernels read only router outputs (bins, C_h, mean of
// V), which were complete before the full-attention kernel started; at their end they wait for
// the full-attention grid (griddepcontrol.wait) and combine the groups it split along the keys
// (combine_split_heads), so work queued after them sees every head's Y.
//
// Two §5 ablations change the cheap heads.  Linear attention replaces the surrogate: its two
// tcgen05 kernels (linear_attn_tc.cu) run before the full-attention kernel.  Without the
// token-wise correction a surrogate head is y_i = C_h, a broadcast like a mean head.  In both
// variants broadcast_heads_kernel writes the broadcast rows (the no-residual surrogate heads and
// the mean heads) behind the full-attention kernel.
#include "attn_plan.cuh"
#include "common.cuh"
#include "internal.h"

namespace vp {

namespace {

constexpr int kThreads = 256;
constexpr int kRows = 256;  // rows per work item

// Y[r0 .. min(N, r0 + kRows))[h][:] = Broadcast(vec[0..63]): 8 threads per row, 16-byte stores.
__device__ __forceinline__ void broadcast_rows(const HeadAttnArgs& a, const float* vec, int h,
                                               int r0, int tid) {
  const int part = tid & 7, rg = tid >> 3;
  const float* mv = vec + 8 * part;
  uint4 val;
  val.x = pack_bf16x2(*(mv + 0), *(mv + 1));
  val.y = pack_bf16x2(*(mv + 2), *(mv + 3));
  val.z = pack_bf16x2(*(mv + 4), *(mv + 5));
  val.w = pack_bf16x2(*(mv + 6), *(mv + 7));
  const int r1 = min(a.N, r0 + kRows);
  for (int row = r0 + rg; row < r1; row += kThreads / 8)
    *reinterpret_cast<uint4*>(a.y + ((size_t)row * a.H + h) * 64 + 8 * part) = val;
}

__global__ void __launch_bounds__(kThreads, 3) broadcast_heads_kernel(HeadAttnArgs a) {
  __shared__ int s_item;
  const int tid = threadIdx.x;
  const int s_first = a.offsets[1], m_first = a.offsets[0];
  const int n_surr = a.offsets[2] - s_first;
  const int n_mean = s_first - m_first;
  const int chunks = (a.N + kRows - 1) / kRows;
  // Surrogate heads are broadcast rows only without the token-wise correction.
  const int s_items = (a.variant & VP_VARIANT_NO_RESIDUAL) ? n_surr * chunks : 0;
  const int items = s_items + (a.skip_mean_y ? 0 : n_mean * chunks);
  pdl_launch();
  // Items (surrogate rows head-major, then mean rows) from a counter, so that CTAs started
  // early (on SMs freed early) do more of them.
  for (;;) {
    __syncthreads();  // s_item is free
    if (tid == 0) s_item = (int)atomicAdd(a.cheap_counter, 1u);
    __syncthreads();
    const int it = s_item;
    if (it >= items) break;
    if (it < s_items) {
      const int slot = it / chunks, chunk = it - slot * chunks;
      const int h = a.head_ids[s_first + slot];
      broadcast_rows(a, a.ctx + h * 64, h, chunk * kRows, tid);
    } else {
      const int it2 = it - s_items;
      const int slot = it2 / chunks, chunk = it2 - slot * chunks;
      const int h = a.head_ids[m_first + slot];
      broadcast_rows(a, a.mean_v + h * 64, h, chunk * kRows, tid);
    }
  }
  // Once the full-attention grid has completed: its split groups.
  pdl_wait();
  combine_split_heads(a, a.attn_ctas, (tid >> 5) * (int)gridDim.x + (int)blockIdx.x, (kThreads / 32) * (int)gridDim.x);
}

}  // namespace

cudaError_t launch_heads(const HeadAttnArgs& a, int num_sms, cudaStream_t st) {
  cudaError_t e = cudaSuccess;
  if (!a.counters_zeroed) {
    e = cudaMemsetAsync(a.counters, 0, sizeof(unsigned int) * kHeadCounters, st);
    if (e != cudaSuccess) return e;
    if (a.s_attn) {  // 0 for the heads that are not in full mode; full heads max into it
      e = cudaMemsetAsync(a.s_attn, 0, sizeof(float) * a.H, st);
      if (e != cudaSuccess) return e;
    }
  }
  if (a.variant & VP_VARIANT_LINEAR_ATTENTION) {
    // The surrogate heads in linear-attention form, state then apply, before the
    // full-attention kernel; the mean heads stay in the cheap-heads kernel behind it.
    e = cudaMemsetAsync(a.lin_state, 0, sizeof(float) * kLinState * a.H, st);
    if (e != cudaSuccess) return e;
    prof_before(VP_KERNEL_SURROGATE, st);
    e = launch_linear_state_tc(a, num_sms, st);
    if (e == cudaSuccess) e = launch_linear_apply_tc(a, num_sms, st);
    prof_extra_launch();
    prof_after(st);
    if (e != cudaSuccess) return e;
  }
  prof_before(VP_KERNEL_ATTN_FULL, st);  // both kernels: no event may separate them
  e = launch_full_heads(a, num_sms, st);
  if (e != cudaSuccess) return e;
  if (!(a.variant & (VP_VARIANT_NO_RESIDUAL | VP_VARIANT_LINEAR_ATTENTION))) {
    e = launch_cheap_heads_tc(a, num_sms, st);
    prof_extra_launch();
    prof_after(st);
    if (e != cudaSuccess) return e;
    return cudaGetLastError();
  }
  e = launch_pdl(broadcast_heads_kernel, dim3(3 * num_sms), kThreads, 0, st, a);
  prof_extra_launch();
  prof_after(st);
  if (e != cudaSuccess) return e;
  return cudaGetLastError();
}

}  // namespace vp
