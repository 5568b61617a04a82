// Per-layer prefetch window and the prefetch list of one sequence (RoPE-aware
// prefetching section).
//
// The section states that, with a sequence at position n, promotion requests go out for
// the blocks covering positions [n, n+w] (it also names [n-w, n] as the range likeliest
// to be read next), and that the window w adapts per layer to the observed attention
// pattern: narrow for local-attention layers, wide for global-attention layers.  It
// prints no formula; the form used here, per partition:
//   S[l] <- d*S[l] + (1-d)*x[l]     x[l]: attention span observed in layer l, tokens
//                                   (binary32, each operation rounded once)
//   w[l] = min(w_max, max(1, ceil(S[l] / block_tokens)))    blocks
// and the list of a sequence at position-block pos0 holds, ordered by (distance, layer,
// head), the ring slot of every block of the sequence's block table at distance < w[l]
// that sits in the host tier.
//
// The list is an ordered compaction of at most distance x layers x heads candidates, in one
// launch: a block counts the qualifying candidates of its chunk, publishes the count, adds up
// the counts of the blocks before it as they appear, and writes.  A block waits only for blocks
// of lower index (bounded: one that gives up sets KV_DEV_WAIT_EXPIRED and leaves, and so do the
// blocks behind it; the last one then reports an empty list).  A call is latency: window, table and d_loc are three dependent reads of
// about 0.7 us, the counts one more; a second launch for the writing cost as much again
// (8 lists of 256 x 80 x 8 candidates: 110 -> 56 us).
#include "kvtier_internal.cuh"

namespace kvt {

namespace {

constexpr int kPfThreads = 256;

__device__ __forceinline__ bool span_ok(float v) {
  return v >= 0.0f && v <= 3.402823466e+38f;  // false for NaN, negatives and infinities
}

__device__ __forceinline__ uint32_t window_of(float span, float block_tokens, uint32_t w_max) {
  const float c = ceilf(__fdiv_rn(span, block_tokens));   // exact: the ceiling of a binary32 is one
  double w = (double)c;
  if (w < 1.0) w = 1.0;
  if (w > (double)w_max) w = (double)w_max;
  return (uint32_t)w;
}

// One block.  mode 0: EMA step with observations x; mode 1: every span = tokens.
// A bad observation anywhere leaves the whole partition as it was.
__global__ void prefetch_window_kernel(float* span, uint32_t* win,
                                       const float* x, float d, float tokens, int mode,
                                       uint32_t layers, float block_tokens, uint32_t w_max,
                                       uint32_t* __restrict__ status) {
  wait_for_kernel_ahead();
  int bad = 0;
  if (mode == 0)
    for (uint32_t l = threadIdx.x; l < layers; l += blockDim.x) bad |= !span_ok(x[l]);
  if (__syncthreads_or(bad)) {
    if (threadIdx.x == 0) atomicOr(status, KV_DEV_BAD_SPAN_VALUE);
    return;
  }
  for (uint32_t l = threadIdx.x; l < layers; l += blockDim.x) {
    float s = tokens;
    if (mode == 0) {
      const float t1 = __fmul_rn(d, span[l]);
      const float t2 = __fsub_rn(1.0f, d);
      const float t3 = __fmul_rn(t2, x[l]);
      s = __fadd_rn(t1, t3);
    }
    span[l] = s;
    win[l] = window_of(s, block_tokens, w_max);
  }
}

struct ListArgs {
  const uint32_t* table;   // [n_pos][L][H] block handles
  const uint32_t* win;     // [L]
  const uint32_t* loc;     // [n_tags]
  unsigned long long* out;
  unsigned long long* count;
  unsigned long long* words;    // [gridDim.x] launch number << 32 | count of the chunk
  uint32_t* serial;             // number of the last launch
  uint32_t* status;
  unsigned long long n_items;   // candidates the host can bound: distances x L x H
  unsigned long long chunk;     // candidates per block, a multiple of kPfTile
  unsigned long long pos0, max_out, n_tags;
  uint32_t layers, heads;
  int dir;
  int vector;              // table rows are aligned vectors of four handles
};

constexpr uint32_t kPfPerThread = 4;                        // consecutive candidates of a thread
constexpr uint32_t kPfTile = kPfThreads * kPfPerThread;
constexpr uint32_t kPfWinCache = 1024;                      // layers whose windows a block keeps in shared memory
constexpr uint32_t kPfSpins = 1u << 22;

// Bits of the thread's four candidates i0 .. i0+3 that qualify, and their ring slots; candidates
// are numbered (distance, layer, head).  Index: the type that holds every candidate's number.
template <typename Index>
__device__ __forceinline__ uint32_t candidates(const ListArgs& a, Index i0, Index end, uint32_t row,
                                               const uint32_t* s_win, uint32_t s_wmax,
                                               uint32_t slot[kPfPerThread]) {
  if (i0 >= end) return 0u;
  Index dist = i0 / (Index)row;
  uint32_t r = (uint32_t)(i0 - dist * (Index)row), t[kPfPerThread], m = 0;
  // (all reads go to the L2: the kernel ahead may have written any of the arrays while this
  // block was already set up)
  if (a.vector) {   // rows of a multiple of four handles: the four are one aligned vector
    const unsigned long long pb = a.dir > 0 ? a.pos0 + dist : a.pos0 - dist;
    uint4 v = make_uint4(KV_NONE, KV_NONE, KV_NONE, KV_NONE);
    if (dist < (Index)s_wmax) v = __ldcg(reinterpret_cast<const uint4*>(a.table + pb * row + r));
    t[0] = v.x; t[1] = v.y; t[2] = v.z; t[3] = v.w;
#pragma unroll
    for (uint32_t u = 0; u < kPfPerThread; ++u) {
      const uint32_t layer = (r + u) / a.heads;
      const uint32_t w = layer < kPfWinCache ? s_win[layer] : __ldcg(a.win + layer);
      if (dist >= (Index)w) t[u] = KV_NONE;
    }
  } else {
#pragma unroll
    for (uint32_t u = 0; u < kPfPerThread; ++u) {
      const uint32_t layer = r / a.heads;
      const uint32_t w = layer < kPfWinCache ? s_win[layer] : __ldcg(a.win + layer);
      t[u] = KV_NONE;
      if (i0 + (Index)u < end && dist < (Index)w) {
        const unsigned long long pb = a.dir > 0 ? a.pos0 + dist : a.pos0 - dist;
        t[u] = __ldcg(a.table + pb * row + r);
      }
      if (++r == row) { r = 0; ++dist; }
    }
  }
#pragma unroll
  for (uint32_t u = 0; u < kPfPerThread; ++u) {
    slot[u] = KV_NONE;
    if (t[u] < a.n_tags) slot[u] = __ldcg(a.loc + t[u]);   // (KV_NONE is never a handle)
  }
#pragma unroll
  for (uint32_t u = 0; u < kPfPerThread; ++u) {
    m |= (uint32_t)(slot[u] != KV_NONE && (slot[u] & KV_LOC_HOST)) << u;
    slot[u] &= ~KV_LOC_HOST;
  }
  return m;
}

template <typename Index>
__global__ void __launch_bounds__(kPfThreads) prefetch_list_kernel(const ListArgs a) {
  __shared__ uint32_t s_win[kPfWinCache];
  __shared__ unsigned long long s_before[kPfThreads / 32];
  __shared__ uint32_t s_warp[kPfThreads / 32];
  __shared__ uint32_t s_wmax;
  const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t row = a.layers * a.heads;
  wait_for_kernel_ahead();
  const uint32_t tag = *a.serial + 1u;

  // the widest window bounds the distances any layer wants
  if (tid == 0) s_wmax = 0;
  __syncthreads();
  uint32_t wm = 0;
  for (uint32_t l = tid; l < a.layers; l += kPfThreads) {
    const uint32_t w = __ldcg(a.win + l);
    if (l < kPfWinCache) s_win[l] = w;
    wm = max(wm, w);
  }
  wm = __reduce_max_sync(0xFFFFFFFFu, wm);
  if (lane == 0 && wm) atomicMax(&s_wmax, wm);
  __syncthreads();
  const Index limit = (Index)min(a.n_items, (unsigned long long)s_wmax * row);
  const Index c0 = (Index)blockIdx.x * (Index)a.chunk;
  const Index c1 = (Index)min((unsigned long long)c0 + a.chunk, (unsigned long long)limit);   // (c0 >= c1: nothing)

  uint32_t n = 0, m = 0, slot[kPfPerThread];   // m, slot: the last tile's, all there is of a one-tile chunk
  for (Index i = c0 + (Index)(tid * kPfPerThread), at = c0; at < c1; i += kPfTile, at += kPfTile) {
    m = candidates<Index>(a, i, c1, row, s_win, s_wmax, slot);
    n += (uint32_t)__popc(m);
  }
  n = __reduce_add_sync(0xFFFFFFFFu, n);
  if (lane == 0) s_warp[warp] = n;
  __syncthreads();
  uint32_t mine = 0;
#pragma unroll
  for (int w = 0; w < kPfThreads / 32; ++w) mine += s_warp[w];
  if (tid == 0)
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(a.words + blockIdx.x),
                 "l"((unsigned long long)tag << 32 | mine)
                 : "memory");

  // candidates that qualify before this chunk
  unsigned long long before = 0;
  bool ok = true;
  for (uint32_t b = tid; b < blockIdx.x; b += kPfThreads) {
    unsigned long long v = 0;
    uint32_t it = 0;
    do {
      asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(a.words + b) : "memory");
    } while ((uint32_t)(v >> 32) != tag && ++it < kPfSpins);
    ok = ok && (uint32_t)(v >> 32) == tag;
    before += (uint32_t)v;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) before += __shfl_xor_sync(0xFFFFFFFFu, before, o);
  if (lane == 0) s_before[warp] = before;
  ok = __syncthreads_and(ok) != 0;
  if (!ok) {
    if (tid == 0) {
      atomicOr(a.status, KV_DEV_WAIT_EXPIRED);
      if (blockIdx.x == gridDim.x - 1) {
        *a.count = 0;
        *a.serial = tag;
      }
    }
    return;
  }
  unsigned long long offset = 0;
#pragma unroll
  for (int w = 0; w < kPfThreads / 32; ++w) offset += s_before[w];
  if (blockIdx.x == gridDim.x - 1 && tid == 0) {
    *a.count = offset + mine;
    *a.serial = tag;   // (every block has published its count, so every block has read the number)
  }

  const bool one_tile = c0 < c1 && c1 - c0 <= (Index)kPfTile;
  for (Index i = c0 + (Index)(tid * kPfPerThread), at = c0; at < c1; i += kPfTile, at += kPfTile) {
    if (!one_tile) m = candidates<Index>(a, i, c1, row, s_win, s_wmax, slot);
    uint32_t incl = (uint32_t)__popc(m);
    const uint32_t own = incl;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
      if (lane >= (uint32_t)o) incl += y;
    }
    __syncthreads();                       // s_warp of the tile before has been read
    if (lane == 31) s_warp[warp] = incl;
    __syncthreads();
    uint32_t ahead = 0, total = 0;
#pragma unroll
    for (int w = 0; w < kPfThreads / 32; ++w) {
      const uint32_t c = s_warp[w];
      if (w < (int)warp) ahead += c;
      total += c;
    }
    unsigned long long p = offset + ahead + (incl - own);
#pragma unroll
    for (uint32_t u = 0; u < kPfPerThread; ++u) {
      if ((m >> u) & 1u) {
        if (p < a.max_out) a.out[p] = slot[u];
        ++p;
      }
    }
    offset += total;
  }
}

}  // namespace

cudaError_t launch_prefetch_window(const PrefetchState& pf, int q, int mode, const float* x, float decay,
                                   float tokens, const Workspace& ws, cudaStream_t s) {
  return launch_overlapped(prefetch_window_kernel, 1u, 128u, s, pf.span + pf.off[q], pf.win + pf.off[q], x, decay,
                           tokens, mode, pf.layers[q], (float)pf.block_tokens[q], pf.w_max[q], ws.status);
}

cudaError_t launch_prefetch_list(const PrefetchState& pf, int q, const uint32_t* table, uint64_t n_pos,
                                 uint64_t pos0, int dir, const uint32_t* loc, uint64_t n_tags,
                                 unsigned long long* out, uint64_t max_out, unsigned long long* count,
                                 const Workspace& ws, cudaStream_t s) {
  ListArgs a;
  a.table = table;
  a.win = pf.win + pf.off[q];
  a.loc = loc;
  a.out = out;
  a.count = count;
  a.words = pf.words;
  a.serial = pf.serial;
  a.status = ws.status;
  a.layers = pf.layers[q];
  a.heads = pf.heads[q];
  a.dir = dir;
  a.pos0 = pos0;
  a.max_out = out ? max_out : 0;
  a.n_tags = n_tags;
  // distances inside the table on the chosen side, never more than the cap on the window
  uint64_t dists = n_pos == 0 ? 0 : (dir > 0 ? n_pos - pos0 : pos0 + 1);
  if (dists > pf.w_max[q]) dists = pf.w_max[q];
  a.n_items = dists * a.layers * a.heads;
  a.vector = (a.layers * a.heads) % 4 == 0 && (reinterpret_cast<uintptr_t>(table) & 15u) == 0;
  // One tile of 1,024 candidates per block while two blocks per SM hold them all; beyond that
  // blocks take several (and evaluate their candidates twice, the second time from the caches).
  uint64_t most = (uint64_t)sm_count() * 2;
  if (most > kPrefetchChunks) most = kPrefetchChunks;
  uint64_t chunk = (a.n_items + most - 1) / most;
  chunk = (chunk + kPfTile - 1) / kPfTile * kPfTile;
  if (chunk == 0) chunk = kPfTile;
  a.chunk = chunk;
  uint64_t blocks = (a.n_items + chunk - 1) / chunk;
  if (blocks == 0) blocks = 1;
  // 32-bit numbers divide in a fifth of the instructions
  if (a.n_items < 0x7FFFFFFFull) return launch_overlapped(prefetch_list_kernel<uint32_t>, (unsigned)blocks, kPfThreads, s, a);
  return launch_overlapped(prefetch_list_kernel<unsigned long long>, (unsigned)blocks, kPfThreads, s, a);
}

}  // namespace kvt
