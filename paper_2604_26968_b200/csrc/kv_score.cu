// Scoring kernels: event reduction, and the fused posterior + EMA + score pass.
//
// The arithmetic itself lives in kv_score_device.cuh.
#include "kv_score_device.cuh"

namespace kvt {

// ---- event reduction ---------------------------------------------------------
// PACKED: touches go to the packed counts, or, while the last epochs' have overflowed them (wide), to the others.
template <bool PACKED>
__global__ void __launch_bounds__(kEventThreads, kEventBlocksPerSm)
event_reduce_kernel(const uint32_t* ev_entry, const uint8_t* ev_hit, uint64_t n_events, const uint8_t* pair,
                    uint32_t* touch, unsigned long long* packed, uint64_t n, unsigned long long* delta,
                    const uint32_t* wide, uint32_t* status) {
  __shared__ uint32_t s_cnt[16 * kEventThreads];   // [pair][thread]: events | hits << 16
#pragma unroll
  for (uint32_t i = 0; i < 16; ++i) s_cnt[i * kEventThreads + threadIdx.x] = 0;   // (the thread's own words)
  wait_for_kernel_ahead();
  const uint64_t gtid = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x, stride = (uint64_t)gridDim.x * blockDim.x;
  EventVec first[kEventVecs];   // (together with *wide: one behind the other is a latency more)
  load_events(ev_entry, ev_hit, n_events / 4, 0, gtid, stride, first);
  const uint32_t bad = reduce_events<PACKED>(PACKED && *wide == 0u, first, ev_entry, ev_hit, n_events, pair, touch,
                                                   packed, n, gtid, stride, s_cnt, delta);
  if (bad) atomicOr(status, bad);
}

// Set up while the kernel ahead finishes, up to this many events: 1.4 M events behind a selection gain
// 2 us that way (46.4 -> 44.1 a pass), 3.3 M still gain, 15.3 M lose 3 us (188.5 -> 191.4).
constexpr uint64_t kEventOverlapMax = 8ull << 20;

cudaError_t launch_event_reduce(const uint32_t* ev_entry, const uint8_t* ev_hit, uint64_t n_events,
                                const EntryState& st, const Workspace& ws, cudaStream_t s) {
  if (n_events == 0) return cudaSuccess;
  uint64_t blocks = (n_events / 4 + kEventThreads - 1) / kEventThreads;
  if (blocks == 0) blocks = 1;
  const uint64_t cap = (uint64_t)sm_count() * kEventBlocksPerSm;
  if (blocks > cap) blocks = cap;
  const uint8_t* pair = st.pair;
  uint32_t* touch = st.touch;
  const uint32_t* wide = &ws.sel->touch_wide;
  unsigned long long* packed = st.packed;
  uint64_t n = st.n;
  unsigned long long* delta = ws.delta;
  uint32_t* status = ws.status;
  void* args[] = {&ev_entry, &ev_hit, &n_events, &pair, &touch, &packed, &n, &delta, &wide, &status};
  const void* fn = packed ? (const void*)event_reduce_kernel<true> : (const void*)event_reduce_kernel<false>;
  const cudaError_t e = launch_scoring_kernel(fn, dim3((unsigned)blocks), dim3(kEventThreads), args, 0, s, false, ws,
                                              n_events <= kEventOverlapMax);
  count_launches(1);
  return e != cudaSuccess ? e : cudaGetLastError();
}

// The touches of a trace whose packed counts nobody takes up, in the 32-bit ones (where they are already while
// *wide says so).
__global__ void __launch_bounds__(kThreads)
event_recount_kernel(const uint32_t* ev_entry, uint64_t n_events, const uint8_t* pair, uint32_t* touch, uint64_t n,
                     const uint32_t* wide) {
  if (*wide) return;
  for (uint64_t e = (uint64_t)blockIdx.x * kThreads + threadIdx.x; e < n_events; e += (uint64_t)gridDim.x * kThreads) {
    const uint32_t i = ev_entry[e];
    if (i < n && !(pair[i] & kPairFree)) atomicAdd(touch + i, 1u);
  }
}

cudaError_t launch_event_recount(const uint32_t* ev_entry, uint64_t n_events, const EntryState& st, const Workspace& ws,
                                 cudaStream_t s) {
  if (n_events == 0) return cudaSuccess;
  const uint64_t blocks = (n_events + kThreads - 1) / kThreads, cap = (uint64_t)sm_count() * 8;
  event_recount_kernel<<<(unsigned)(blocks < cap ? blocks : cap), kThreads, 0, s>>>(ev_entry, n_events, st.pair, st.touch,
                                                                                   st.n, &ws.sel->touch_wide);
  count_launches(1);
  return cudaMemsetAsync(st.packed, 0, (st.n + 3) / 4 * 8, s);
}

// ---- entry pass ----------------------------------------------------------------------
// Every block forms the 16 posteriors itself (32 counters, read-only here), then
// streams its share of the entries: four per thread and iteration, every array
// read and written with 16-byte (for the byte arrays 4-byte) accesses.  The last
// block to finish folds the epoch's counts into the totals, clears them and
// publishes P; by then every block has read them.
constexpr int kUpdateBlocksPerSm = 4;
__global__ void __launch_bounds__(kThreads, kUpdateBlocksPerSm)
entry_update_kernel(const EntryState st, const Predictor pd, const HeadWeights hw, uint32_t epoch) {
  __shared__ float sP[16];
  __shared__ bool s_last;
  const int policy = pd.policy;
  wait_for_kernel_ahead();
  PairStep step;
  if (threadIdx.x < 16) {
    step = pair_step(pd, threadIdx.x);
    sP[threadIdx.x] = step.estimate;
  }
  __syncthreads();
  const uint64_t n4 = st.n / 4;
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  uint64_t v = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  EntryVec cur;
  if (v < n4) cur = entry_load4(st, v, policy);
  for (; v < n4; v += stride) {   // the next vector's loads fly while this one is finished
    EntryVec nxt;
    if (v + stride < n4) nxt = entry_load4(st, v + stride, policy);
    float4 sc;
    entry_finish4<false>(st, v, cur, sP, policy, epoch, hw, nullptr, sc);
    cur = nxt;
  }
  // ragged tail (n not a multiple of 4)
  const uint64_t i = n4 * 4 + (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < st.n) {
    float sc;
    entry_update1(st, i, sP, policy, epoch, hw, 0u, nullptr, sc);
  }
  // commit by the last block to finish
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    s_last = atomicAdd(pd.ticket, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (s_last && threadIdx.x < 16) {
    commit_predictor(pd, threadIdx.x, step);
    if (threadIdx.x == 0) *pd.ticket = 0;
  }
}

__global__ void blend_reset_kernel(BlendState* b) {
  for (uint32_t i = threadIdx.x; i < kMaxWindow * 32; i += blockDim.x) b->win[i] = 0;
  if (threadIdx.x < 32) b->wsum[threadIdx.x] = 0;
  if (threadIdx.x == 0) b->head = 0;
}

cudaError_t launch_blend_reset(const Workspace& ws, cudaStream_t s) {
  blend_reset_kernel<<<1, 256, 0, s>>>(ws.blend);
  count_launches(1);
  return cudaGetLastError();
}

cudaError_t launch_entry_update(const EntryState& st, uint64_t* hits, uint64_t* misses, float* P,
                                float alpha0, float beta0, const Workspace& ws, uint32_t epoch,
                                const ScoreOptions& opt, const HeadWeights& hw, cudaStream_t s) {
  uint64_t blocks = (st.n / 4 + kThreads - 1) / kThreads;
  if (blocks == 0) blocks = 1;
  const uint64_t cap = (uint64_t)sm_count() * kUpdateBlocksPerSm;   // (one wave: a second one forms the posteriors again)
  if (blocks > cap) blocks = cap;
  const Predictor pd{hits,       misses,    P,          alpha0, beta0, ws.delta, &ws.sel->update_ticket,
                     opt.policy, opt.kappa, opt.window, ws.blend};
  EntryState st_arg = st;
  Predictor pd_arg = pd;
  HeadWeights hw_arg = hw;
  void* args[] = {&st_arg, &pd_arg, &hw_arg, &epoch};
  const cudaError_t e = launch_scoring_kernel((const void*)entry_update_kernel, dim3((unsigned)blocks),
                                              dim3(kThreads), args, 0, s, false, ws);
  count_launches(1);
  return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace kvt
