// Device-side pieces of the scoring pass, shared by the stand-alone scoring
// kernels (kv_score.cu) and the fused score + select kernel (kv_select_persist.cu).
//
// All binary32 arithmetic uses the explicitly rounded intrinsics (__fmul_rn,
// __fadd_rn, __fsub_rn, __fdiv_rn), which the compiler never contracts into a
// fused multiply-add, and denormals are kept (no flush-to-zero), so results
// are bit-identical to the same operations done one at a time on a CPU.
#pragma once
#include "kvtier_internal.cuh"

namespace kvt {

// ---- event reduction ---------------------------------------------------------
// Each event adds one to the (pair, hit) counter of its entry's pair -- the
// alpha += 1 / beta += 1 update of the Bayesian reuse section -- and one to
// the entry's touch count.  Counters are integers, so the order of the additions
// does not matter.
//
// Pair counters: every thread owns 16 packed counters in shared memory (one per
// pair: events in the low half, hits in the high half), laid out pair-major so
// that the threads of a warp always fall into 32 different banks.  Counting an
// event is a plain read-add-write of the thread's own word: no vote, no atomic.
// The block adds its columns up once at the end.
//
// Touch counts, in the array that the caller may look at (kv_epoch_events): every update
// is a 64-bit atomic on the aligned pair of 32-bit counts (touch[2i], touch[2i+1]) --
// adding 1, 1 << 32 or both -- so that all atomics on a word have one size.  (A carry out
// of the low count would need 2^32 touches of one entry in one epoch, where the count
// wraps anyway.)  The one exception is the last entry of an array of odd length, whose
// partner would lie outside the array: it takes 32-bit atomics, and only those.
//
// Touch counts that only the fused scoring pass of the same call reads (PACKED): 64 bits
// for four entries, nine for each and the sum of the four in the upper 28, so that one
// atomic counts all events of a vector on the same four entries, and half the bytes are
// scattered over.  A count that overflows carries into the next field and
// takes 511 from the sum of the fields, or, the last one, 512, and adds one to the sum
// kept beside them: the two agree again only after 512 * 2^28 / 513 touches, more than a
// trace that is counted this way has, so the scoring pass sees of every word whether it is
// right.  (Atomics that return the word they found would tell the event reduction of every
// carry, and bytes would do, but they took 37.6 us instead of 28.4 for 15.3 M events, 9.2
// instead of 6.3 for 0.6 M.)
//
// Traces in which a touched block reports all its heads hand every thread four
// consecutive entries (an aligned group of four ids): one 4-byte load then
// fetches their pairs and FREE bits, and one atomic on a packed word, or two on the 32-bit
// counts, counts the four touches.  Those two go out from neighbouring lanes of one instruction, so
// that a 32-byte sector of counts is visited once and not twice.  (A warp's events dealt out again, neighbours to
// neighbouring lanes, where vectors are no runs: 1 us less in 141 where single entries in order follow runs, but
// 12 M events on 18.8 M entries 189 -> 239 us a pass with one broken vector a warp, blocks of two heads 207 -> 245,
// 6 M single entries in order on 3.1 M 53.7 -> 59.8.)
//
// What bounds it: the latency of two dependent scattered reads (event, pair byte) and
// the rate of the atomics.  The next vectors' events are on their way while the current
// ones' pair bytes are fetched.
constexpr uint32_t kEventThreads = 512;
constexpr uint32_t kEventBlocksPerSm = 2;
constexpr uint32_t kEventVecs = 2;          // 4-event vectors a thread handles per iteration
constexpr uint32_t kEventFlushIters = 4096; // iterations between flushes: 8 events each, below 2^16

struct EventVec {
  uint4 id;
  uint32_t hit;    // byte j: hit flag of event j
};

// The calling thread's vectors of iteration it.
__device__ __forceinline__ void load_events(const uint32_t* ev_entry, const uint8_t* ev_hit, uint64_t n4, uint64_t it,
                                            uint64_t gtid, uint64_t stride, EventVec x[kEventVecs]) {
#pragma unroll
  for (uint32_t u = 0; u < kEventVecs; ++u) {
    const uint64_t v = (it * kEventVecs + u) * stride + gtid;
    x[u].id = make_uint4(0xFFFFFFFFu, 0xFFFFFFFFu, 0xFFFFFFFFu, 0xFFFFFFFFu);  // past the end: no entry
    x[u].hit = 0;
    if (v < n4) {
      x[u].id = __ldcs(reinterpret_cast<const uint4*>(ev_entry) + v);
      x[u].hit = __ldcs(reinterpret_cast<const uint32_t*>(ev_hit) + v);
    }
  }
}

// bit 7 of every non-zero byte
__device__ __forceinline__ uint32_t nonzero_bytes(uint32_t x) {
  return (((x & 0x7F7F7F7Fu) + 0x7F7F7F7Fu) | x) & 0x80808080u;
}

__device__ __forceinline__ void touch_add(uint32_t* touch, uint32_t i, uint32_t n32,
                                          unsigned long long inc_pair) {
  // inc_pair: what to add to the aligned pair that contains entry i
  if ((i | 1u) < n32)
    atomicAdd(reinterpret_cast<unsigned long long*>(touch + (i & ~1u)), inc_pair);
  else
    atomicAdd(&touch[i], 1u);   // last entry of an odd-length array (i is even, inc_pair is 1)
}

constexpr uint32_t kFieldBits = 9, kFieldMax = (1u << kFieldBits) - 1u, kSumShift = 4u * kFieldBits;
// Touches of four entries, one byte each (a few of each), as what they add to the entries' packed word.
__device__ __forceinline__ unsigned long long packed_touches(uint32_t b) {
  const uint32_t lo = (b & 0xFFu) | (b & 0xFF00u) << 1 | (b & 0xFF0000u) << 2;
  return ((unsigned long long)(b >> 24) << (3u * kFieldBits) | lo) + ((unsigned long long)__dp4a(b, 0x01010101u, 0u) << kSumShift);
}
// The four counts; false if one of them has overflowed.
__device__ __forceinline__ bool unpack_touches(uint2 w, uint32_t t[4]) {
  t[0] = w.x & kFieldMax;
  t[1] = (w.x >> kFieldBits) & kFieldMax;
  t[2] = (w.x >> (2u * kFieldBits)) & kFieldMax;
  t[3] = __funnelshift_r(w.x, w.y, 3u * kFieldBits) & kFieldMax;
  return t[0] + t[1] + t[2] + t[3] == w.y >> (kSumShift - 32u);
}

// The packed counts w of vector v are added to its 32-bit counts t, and both are cleared.  False, and nothing
// done, if a packed count has overflowed.  (The 32-bit counts are looked at in any case: kv_epoch_events or the
// caller may have left something there.  To have the event reduction look for that took longer, 18.8 M entries
// 158 us a pass instead of 156.)
__device__ __forceinline__ bool take_touches(const EntryState& st, uint64_t v, uint2 w, uint4& t) {
  uint32_t p[4];
  if (!unpack_touches(w, p)) return false;
  if (w.x | w.y) st.packed[v] = 0;
  if (t.x | t.y | t.z | t.w) reinterpret_cast<uint4*>(st.touch)[v] = make_uint4(0, 0, 0, 0);
  t.x += p[0]; t.y += p[1]; t.z += p[2]; t.w += p[3];
  return true;
}

// Four events on entries in a row, all of them in a pool of n: an aligned group, or (packed) one whose words
// of pair bytes lie inside the array.  (From 2^32 - 3 on the sums wrap: the first id has to lie below the
// last one, or an event that is refused would be taken for the neighbour of the pool's first entries.)
__host__ __device__ __forceinline__ bool is_run(const uint32_t id[4], uint32_t n, bool packed) {
  return (packed || !(id[0] & 3u)) && id[0] < id[3] && id[1] == id[0] + 1u && id[2] == id[0] + 2u && id[3] == id[0] + 3u &&
         (id[3] | 3u) < n;
}

// The calling block's share of the events.  s_cnt: kEventThreads * 16 words of shared
// memory, zero on entry; word [p * kEventThreads + t] holds thread t's
// counts for pair p (events | hits << 16) since the last flush.  delta: the 32
// global epoch counters (index 2 * pair + hit).  Returns the KV_DEV_* bits of
// refused events.  nxt: the thread's first vectors, from load_events.  use_packed (PACKED only): where the
// touches go; looked at late, since it comes from memory, and no second template, since a kernel with two copies
// of this takes longer to fetch (4,096 entries: without such a choice 13.05 us a pass, like this 13.2, with two
// copies 13.5).  Every thread of the block must call it.
template <bool PACKED>
__device__ __forceinline__ uint32_t reduce_events(bool use_packed, EventVec nxt[kEventVecs], const uint32_t* ev_entry, const uint8_t* ev_hit,
                                                  uint64_t n_events, const uint8_t* pair, uint32_t* touch,
                                                  unsigned long long* packed, uint64_t n, uint64_t gtid,
                                                  uint64_t stride, uint32_t* s_cnt, unsigned long long* delta) {
  const uint64_t n4 = n_events / 4;
  const uint64_t iters = (n4 + stride * kEventVecs - 1) / (stride * kEventVecs);  // same for every thread
  // ids are 32-bit, so the bound is too (an id can never reach 2^32 - 1 = "no entry")
  const uint32_t n32 = n > 0xFFFFFFFFull ? 0xFFFFFFFFu : (uint32_t)n;
  const uint32_t lane = threadIdx.x & 31u;
  uint32_t* my = s_cnt + threadIdx.x;
  constexpr uint32_t col = kEventThreads;
  const bool to_packed = PACKED && use_packed;
  bool bad_id = false, not_resident = false;

  // adds the block's columns to the global counters and clears them; the 32 sums
  // go out as one warp's 32 neighbouring atomics (a single request per cache line)
  auto flush = [&]() {
    __shared__ uint32_t s_tot[32];
    __syncthreads();
    const uint32_t warp = threadIdx.x >> 5;
    for (uint32_t p = warp; p < 16; p += kEventThreads / 32) {
      uint32_t ev = 0, hi = 0;
#pragma unroll
      for (uint32_t t = 0; t < col; t += 32) {
        const uint32_t c = s_cnt[p * col + t + lane];
        s_cnt[p * col + t + lane] = 0;
        ev += c & 0xFFFFu;
        hi += c >> 16;
      }
      ev = __reduce_add_sync(0xFFFFFFFFu, ev);
      hi = __reduce_add_sync(0xFFFFFFFFu, hi);
      if (lane == 0) {
        s_tot[2 * p + 1] = hi;
        s_tot[2 * p] = ev - hi;
      }
    }
    __syncthreads();
    if (threadIdx.x < 32 && s_tot[threadIdx.x])
      atomicAdd(&delta[threadIdx.x], (unsigned long long)s_tot[threadIdx.x]);
    __syncthreads();
  };
  // counts event j of a vector (pair byte and hit bit already extracted)
  auto count = [&](uint32_t prj, uint32_t hitbit) { my[(prj & 15u) * col] += 1u + (hitbit << 16); };

  auto ids_of = [](const EventVec& x, uint32_t id[4]) { id[0] = x.id.x; id[1] = x.id.y; id[2] = x.id.z; id[3] = x.id.w; };
  auto gather = [&](const uint32_t id[4], bool run) {   // the vector's pair bytes (bit 7 = FREE or out of range)
    uint32_t w = 0;
    if (run) {   // (through the L1: neighbouring blocks share sectors)
      const uint32_t* p = reinterpret_cast<const uint32_t*>(pair) + (id[0] >> 2);
      w = p[0];
      if (PACKED && (id[0] & 3u)) w = __funnelshift_r(w, p[1], 8u * (id[0] & 3u));
    } else {
#pragma unroll
      for (int j = 0; j < 4; ++j) w |= (uint32_t)(id[j] < n32 ? pair[id[j]] : (uint8_t)kPairFree) << (8 * j);
    }
    return w;
  };

  for (uint64_t it = 0; it < iters; ++it) {
    EventVec cur[kEventVecs];
    bool run[kEventVecs];       // ids are a run of four inside the pool
    uint32_t pr4[kEventVecs];   // byte j: pair byte of event j's entry (bit 7 = FREE or out of range)
#pragma unroll
    for (uint32_t u = 0; u < kEventVecs; ++u) cur[u] = nxt[u];
#pragma unroll
    for (uint32_t u = 0; u < kEventVecs; ++u) {  // all gathers before any is used
      uint32_t id[4];
      ids_of(cur[u], id);
      run[u] = is_run(id, n32, PACKED);
      pr4[u] = gather(id, run[u]);
    }
    if (it + 1 < iters) load_events(ev_entry, ev_hit, n4, it + 1, gtid, stride, nxt);
#pragma unroll
    for (uint32_t u = 0; u < kEventVecs; ++u) {
      uint32_t id[4];
      ids_of(cur[u], id);
      const uint32_t pr = pr4[u], hit4 = nonzero_bytes(cur[u].hit);
      // four resident entries in a row (use_packed is looked at as late as this: it comes from memory)
      const bool whole = run[u] && !(pr & 0x80808080u) && (to_packed || !(id[0] & 3u));
      if (to_packed && whole) {
        const uint32_t r = id[0] & 3u;
        atomicAdd(packed + (id[0] >> 2), packed_touches(0x01010101u << (8u * r)));
        if (r) atomicAdd(packed + (id[0] >> 2) + 1u, packed_touches(0x01010101u >> (32u - 8u * r)));
      }
      const uint32_t m = to_packed ? 0u : __ballot_sync(0xFFFFFFFFu, whole);
      if (m) {
#pragma unroll
        for (uint32_t half = 0; half < 2; ++half) {   // 16 vectors' pairs of atomics per instruction
          const uint32_t src = 16u * half + (lane >> 1);
          const uint32_t i0 = __shfl_sync(0xFFFFFFFFu, id[0], src);
          if ((m >> src) & 1u)
            atomicAdd(reinterpret_cast<unsigned long long*>(touch + i0) + (lane & 1u), 0x100000001ull);
        }
      }
      if (whole) {
#pragma unroll
        for (int j = 0; j < 4; ++j) count(pr >> (8 * j), (hit4 >> (8 * j + 7)) & 1u);
      } else if ((it * kEventVecs + u) * stride + gtid < n4) {
        bool ok[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const bool in = id[j] < n32;
          ok[j] = !((pr >> (8 * j)) & kPairFree);   // (out of range gathered nothing: FREE)
          bad_id |= !in;
          not_resident |= in && !ok[j];
        }
        if (to_packed) {   // (the last event on a word adds for those before it)
          uint32_t inc[4];
#pragma unroll
          for (int j = 0; j < 4; ++j) inc[j] = ok[j] ? 1u << (8u * (id[j] & 3u)) : 0u;
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            if (j < 3 && (id[j] >> 2) == (id[j + 1] >> 2)) inc[j + 1] += inc[j];
            else if (inc[j]) atomicAdd(packed + (id[j] >> 2), packed_touches(inc[j]));
          }
        } else {
#pragma unroll
          for (int j = 0; j < 4; j += 2) {
            const uint32_t i0 = id[j], i1 = id[j + 1];
            if (ok[j] && ok[j + 1] && i1 == i0 + 1u && !(i0 & 1u)) {
              atomicAdd(reinterpret_cast<unsigned long long*>(touch + i0), 0x100000001ull);
            } else {
              if (ok[j]) touch_add(touch, i0, n32, (i0 & 1u) ? (1ull << 32) : 1ull);
              if (ok[j + 1]) touch_add(touch, i1, n32, (i1 & 1u) ? (1ull << 32) : 1ull);
            }
          }
        }
#pragma unroll
        for (int j = 0; j < 4; ++j)
          if (ok[j]) count(pr >> (8 * j), (hit4 >> (8 * j + 7)) & 1u);
      }
      __syncwarp();
    }
    if ((it + 1) % kEventFlushIters == 0) flush();   // (uniform over the block)
  }
  uint32_t bad = 0;
  if (bad_id) bad |= KV_DEV_EVENT_BAD_ID;
  if (not_resident) bad |= KV_DEV_EVENT_NOT_RESIDENT;
  // ragged tail (n_events not a multiple of 4): first threads of the grid
  if (gtid < 3) {
    const uint64_t e = n4 * 4 + gtid;
    if (e < n_events) {
      const uint32_t i = __ldcs(ev_entry + e);
      const uint32_t pr = i < n32 ? pair[i] : kPairFree;
      if (i >= n32) {
        bad |= KV_DEV_EVENT_BAD_ID;
      } else if (pr & kPairFree) {
        bad |= KV_DEV_EVENT_NOT_RESIDENT;
      } else {
        count(pr, __ldcs(ev_hit + e) != 0);
        if (to_packed) atomicAdd(packed + (i >> 2), packed_touches(1u << (8u * (i & 3u))));
        else touch_add(touch, i, n32, (i & 1u) ? (1ull << 32) : 1ull);
      }
    }
  }
  flush();
  return bad;
}

// ---- head-granular weight -------------------------------------------------------
// Weight of entry i's (layer, KV head) from the partition's [layer][KV head]
// table (head-granular eviction section); 1 for partitions that are not weighted.
// id = base + (layer * blocks_per_layer + block) * heads + head.
__device__ __forceinline__ float head_weight(const HeadWeights& hw, uint64_t i) {
  int q = 0;
  while (q + 1 < hw.n_parts && i >= hw.base[q + 1]) ++q;
  if (!((hw.on >> q) & 1u)) return 1.0f;
  const uint32_t local = (uint32_t)(i - hw.base[q]);
  const uint32_t layer = hw.by_layer[q](local), head = local - hw.by_heads[q](local) * hw.heads[q];
  return hw.w[hw.w_off[q] + layer * hw.heads[q] + head];
}

// The weights of entries i0 .. i0+3: two divisions for the vector, as multiplications (with the
// divider's own some forty instructions; 3.2 M weighted entries in three calls 54.1 -> 53.4 us),
// then steps along the table.
__device__ __forceinline__ void head_weights4(const HeadWeights& hw, uint64_t i0, float w[4]) {
  int q = 0;
  while (q + 1 < hw.n_parts && i0 >= hw.base[q + 1]) ++q;
  if (q + 1 < hw.n_parts && i0 + 3u >= hw.base[q + 1]) {   // a partition boundary inside the vector
#pragma unroll
    for (int j = 0; j < 4; ++j) w[j] = head_weight(hw, i0 + j);
    return;
  }
#pragma unroll
  for (int j = 0; j < 4; ++j) w[j] = 1.0f;
  if (!((hw.on >> q) & 1u)) return;
  const uint32_t local = (uint32_t)(i0 - hw.base[q]), per_layer = hw.per_layer[q], heads = hw.heads[q];
  const uint32_t layer = hw.by_layer[q](local);
  uint32_t in_layer = local - layer * per_layer, head = in_layer - hw.by_heads[q](in_layer) * heads;
  const float* row = hw.w + hw.w_off[q] + layer * heads;
  const float* const end = hw.w + hw.w_off[q] + hw.layers[q] * heads;
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    if (row < end) w[j] = row[head];   // (a vector at the pool's end may reach past the last layer)
    if (++head == heads) head = 0;
    if (++in_layer == per_layer) { in_layer = 0; row += heads; }   // (a layer is a multiple of heads: head is 0)
  }
}

// ---- per-entry step -----------------------------------------------------------
// One step of the per-entry EMA, then the eviction score of the chosen policy:
// 0 = reuse estimate x EMA importance, 1 = EMA only, 2 = LRU (epoch of the last
// touch, this epoch's touches included) -- the three policies the paper compares.
// w: weight of the entry's (layer, head), which the two importance-based policies
// multiply in (1 = unweighted; x * 1 is exact).
// pair: the entry's pair byte, whose bit 7 says FREE (the state byte is not read: one byte in 22).
__device__ __forceinline__ void entry_step(float& ema, float decay, uint32_t touch, uint32_t pair,
                                           const float* sP, int policy,
                                           uint32_t last_epoch, uint32_t epoch, float w, float& score) {
  if (!(pair & kPairFree)) {
    const float x = __uint2float_rn(touch);
    const float t1 = __fmul_rn(decay, ema);
    const float t2 = __fsub_rn(1.0f, decay);
    const float t3 = __fmul_rn(t2, x);
    ema = __fadd_rn(t1, t3);
    if (policy == 0) score = __fmul_rn(__fmul_rn(sP[pair & 15u], ema), w);
    else if (policy == 1) score = __fmul_rn(ema, w);
    else score = __uint2float_rn(touch ? epoch : last_epoch);
  } else {
    score = __int_as_float(0x7F800000);  // +inf: not a candidate
  }
}

// ---- the predictor ---------------------------------------------------------------
struct Predictor {
  uint64_t* hits;
  uint64_t* misses;
  float* P;
  float alpha0, beta0;
  unsigned long long* delta;   // [32] this epoch's counts, index 2*pair + hit
  unsigned int* ticket;        // blocks that have finished (the last one commits)
  int policy;
  float kappa;                 // confidence saturation constant of the blend
  uint32_t window;             // epochs in the sliding window; 0 = no blending
  BlendState* blend;
};

// Reuse estimate of pair p: the posterior P, or -- when a window is set -- its
// confidence-weighted blend with the hit frequency of the last `window` epochs
// (the current one included).  The paper describes the blend in words (Bayesian
// reuse section: confidence saturates toward 1 as observations accumulate; young
// pairs lean on the windowed frequency); the form used is c = n/(n+kappa),
// estimate = c*P + (1-c)*f, every operation rounded once.  wm/wh receive the
// window's new sums.
__device__ __forceinline__ float reuse_estimate(const Predictor& pd, unsigned p, float P,
                                                unsigned long long h, unsigned long long m,
                                                unsigned long long& wh, unsigned long long& wm) {
  wh = wm = 0;
  if (pd.window == 0) return P;
  const uint32_t head = pd.blend->head;
  wm = pd.blend->wsum[2 * p] - pd.blend->win[head * 32 + 2 * p] + __ldcg(&pd.delta[2 * p]);
  wh = pd.blend->wsum[2 * p + 1] - pd.blend->win[head * 32 + 2 * p + 1] + __ldcg(&pd.delta[2 * p + 1]);
  const float n = __ull2float_rn(h + m);
  const float c = __fdiv_rn(n, __fadd_rn(n, pd.kappa));
  const float fh = __ull2float_rn(wh);
  const float fn = __ull2float_rn(wh + wm);
  const float f = fn > 0.0f ? __fdiv_rn(fh, fn) : P;
  const float t1 = __fmul_rn(c, P);
  const float t2 = __fsub_rn(1.0f, c);
  const float t3 = __fmul_rn(t2, f);
  return __fadd_rn(t1, t3);
}

// Posterior mean of Eq. "reuse" for pair p from the running totals plus this
// epoch's counts: P = alpha / (alpha + beta), alpha = alpha0 + hits, beta =
// beta0 + misses.  The 64-bit counts convert to binary32 with round to nearest
// even; the division is IEEE.  The epoch's counts are read from L2 (other blocks
// of the same launch may have produced them).
__device__ __forceinline__ float posterior(const Predictor& pd, unsigned p, unsigned long long& h,
                                           unsigned long long& m) {
  h = pd.hits[p] + __ldcg(&pd.delta[2 * p + 1]);
  m = pd.misses[p] + __ldcg(&pd.delta[2 * p]);
  const float a = __fadd_rn(pd.alpha0, __ull2float_rn(h));
  const float b = __fadd_rn(pd.beta0, __ull2float_rn(m));
  return __fdiv_rn(a, __fadd_rn(a, b));
}

// What a scoring pass makes of one pair's counters: formed at its start by every block, and
// stored at its end by one of them (from here, without reading the counters again).
struct PairStep {
  unsigned long long h, m, wh, wm;   // totals and window sums with this epoch's counts
  unsigned long long d0, d1;         // this epoch's counts
  float P, estimate;
  uint32_t head;                     // window slot that this epoch takes
};

__device__ __forceinline__ PairStep pair_step(const Predictor& pd, unsigned p) {
  PairStep x;
  x.P = posterior(pd, p, x.h, x.m);
  x.estimate = reuse_estimate(pd, p, x.P, x.h, x.m, x.wh, x.wm);
  x.d0 = __ldcg(&pd.delta[2 * p]);
  x.d1 = __ldcg(&pd.delta[2 * p + 1]);
  x.head = pd.window ? pd.blend->head : 0u;
  return x;
}

// End of an epoch, p = 0..15, once every block has read the counters: folds the epoch's
// counts into the totals, publishes P and the estimate, advances the blend's window and
// clears the counts.
__device__ __forceinline__ void commit_predictor(const Predictor& pd, unsigned p, const PairStep& x) {
  pd.hits[p] = x.h;
  pd.misses[p] = x.m;
  pd.P[p] = x.P;
  pd.blend->estimate[p] = x.estimate;
  if (pd.window > 0) {   // this epoch's counts replace the oldest slot of the window
    pd.blend->win[x.head * 32 + 2 * p] = x.d0;
    pd.blend->win[x.head * 32 + 2 * p + 1] = x.d1;
    pd.blend->wsum[2 * p] = x.wm;
    pd.blend->wsum[2 * p + 1] = x.wh;
    if (p == 0) pd.blend->head = (x.head + 1) % pd.window;
  }
  pd.delta[2 * p] = 0;
  pd.delta[2 * p + 1] = 0;
}

// Four consecutive entries (a 16-byte vector of each array) through the entry step,
// in two halves so that a caller can have the next vector's loads in flight
// while it finishes this one.  v indexes vectors.  The touch counts are read from
// L2: other blocks' atomics made them.  PACKED: take_touches has read and cleared them.  hot:
// where to say that an entry has had more touches than a packed count holds.
struct EntryVec {
  float4 e, d;
  uint4 t, le;         // t: touch counts
  uint32_t pr4;        // pair bytes
};

__device__ __forceinline__ EntryVec entry_load4(const EntryState& st, uint64_t v, int policy) {
  EntryVec x;
  x.e = reinterpret_cast<const float4*>(st.ema)[v];
  x.d = reinterpret_cast<const float4*>(st.decay)[v];
  x.t = __ldcg(reinterpret_cast<const uint4*>(st.touch) + v);
  x.pr4 = reinterpret_cast<const uint32_t*>(st.pair)[v];
  x.le = make_uint4(0, 0, 0, 0);
  if (policy == 2) x.le = reinterpret_cast<const uint4*>(st.last_epoch)[v];  // only LRU reads it
  return x;
}

// The counts and last_epoch are only written where an entry was touched.  kPlain: the caller
// knows that the policy is the Bayesian product and that no partition is weighted (the
// policy and weight tests then fold away at compile time).
template <bool PACKED, bool kPlain = false>
__device__ __forceinline__ void entry_finish4(const EntryState& st, uint64_t v, EntryVec& x, const float* sP,
                                              int policy, uint32_t epoch, const HeadWeights& hw, uint32_t* hot,
                                              float4& sc) {
  float e[4] = {x.e.x, x.e.y, x.e.z, x.e.w}, s[4];
  const float d[4] = {x.d.x, x.d.y, x.d.z, x.d.w};
  const uint32_t t[4] = {x.t.x, x.t.y, x.t.z, x.t.w}, le[4] = {x.le.x, x.le.y, x.le.z, x.le.w};
  // (nearly always all four are RESIDENT: one test then serves them)
  const uint32_t free4 = x.pr4 & (kPairFree * 0x01010101u);
  float w[4] = {1.0f, 1.0f, 1.0f, 1.0f};
  if (!kPlain && hw.on) head_weights4(hw, 4 * v, w);
#pragma unroll
  for (int j = 0; j < 4; ++j)
    entry_step(e[j], d[j], t[j], free4 ? (x.pr4 >> (8 * j)) & 0xFFu : (x.pr4 >> (8 * j)) & 15u, sP,
               kPlain ? 0 : policy, le[j], epoch, w[j], s[j]);
  sc = make_float4(s[0], s[1], s[2], s[3]);
  reinterpret_cast<float4*>(st.ema)[v] = make_float4(e[0], e[1], e[2], e[3]);
  reinterpret_cast<float4*>(st.score)[v] = sc;
  // touch counts of FREE entries are always zero (events on them are refused)
  if (x.t.x | x.t.y | x.t.z | x.t.w) {
    if (!PACKED) reinterpret_cast<uint4*>(st.touch)[v] = make_uint4(0, 0, 0, 0);
    if (hot && max(max(x.t.x, x.t.y), max(x.t.z, x.t.w)) > kFieldMax) *hot = 1u;
    if (x.t.x && x.t.y && x.t.z && x.t.w) {   // a block that reported all its heads: one store
      reinterpret_cast<uint4*>(st.last_epoch)[v] = make_uint4(epoch, epoch, epoch, epoch);
    } else {
      if (x.t.x) st.last_epoch[4 * v + 0] = epoch;
      if (x.t.y) st.last_epoch[4 * v + 1] = epoch;
      if (x.t.z) st.last_epoch[4 * v + 2] = epoch;
      if (x.t.w) st.last_epoch[4 * v + 3] = epoch;
    }
  }
}

// The same for one entry (ragged ends), which has had t touches beside those of the 32-bit count.
__device__ __forceinline__ void entry_update1(const EntryState& st, uint64_t i, const float* sP, int policy,
                                              uint32_t epoch, const HeadWeights& hw, uint32_t t,
                                              uint32_t* hot, float& sc) {
  float e = st.ema[i];
  const uint32_t tw = __ldcg(&st.touch[i]);
  t += tw;
  const float w = hw.on ? head_weight(hw, i) : 1.0f;
  entry_step(e, st.decay[i], t, st.pair[i], sP, policy, policy == 2 ? st.last_epoch[i] : 0u, epoch, w, sc);
  st.ema[i] = e;
  st.score[i] = sc;
  if (tw) st.touch[i] = 0;
  if (hot && t > kFieldMax) *hot = 1u;
  if (t) st.last_epoch[i] = epoch;
}

}  // namespace kvt
