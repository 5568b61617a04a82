// k-lowest selection as ONE cooperative, persistent launch.
//
// The multi-launch selection in kv_select.cu spends most of its time between
// kernels when the pool has a few million entries: ten dependent launches of
// 3-10 us each.  Here one CTA per SM stays resident for the whole selection.
//
// The pool is cut into rows: a full row is one chunk of 4,096 entries per CTA (CTA g
// holds entries (r*G + g)*4096 ...), and what is left after the full rows is one more
// row of equal, shorter pieces (a multiple of 128 entries).  So a region of the pool
// that costs more than others -- many touched entries, many keys near the threshold --
// is spread over all CTAs, and no CTA has a whole chunk more than another.  Inside a
// row a warp owns 128 consecutive entries, a lane four of them.
//
//   A  every score is compared with a bracket around the hinted threshold (tau of the
//      previous selection, or where its trend leads; fused form: the entry pass
//      itself produces the score).  Keys below the bracket set a bit (four ballots per
//      warp and row); keys inside it (typically 4-15 %) enter a histogram of 2,048 bins
//      and are appended to the warp's list of notes.
//   B  when rank k falls inside the bracket, ONE more histogram (the single keys of the
//      bin that holds rank k) finishes it, built from the notes alone; that pass also
//      sets the bits of the notes in lower bins and keeps only the notes of that bin.
//      Otherwise (no hint, or a miss) three digits of a plain radix select, over keys
//      that the first pass leaves in shared memory when they fit.
//   C  tau is known: the kept notes (or the keys) complete the bitmaps "below tau" and
//      "equal to tau", whose population counts go, row by row, into a pool-wide table.
//   D  every CTA sums that table's rows, knows how many victims precede each of its
//      chunks, and writes its own victims in ascending id order straight from the
//      bitmaps.
//
// What bounds it: phase A streams 24 B an entry from HBM, its issue slots half busy; B to D are
// three exchanges between all CTAs (two histograms, one table of counts) of ~2.5 us each, latency of L2
// and of the block barriers around them.  An exchange is a grid barrier (a counter that
// every CTA increments and one of its threads polls).  (Tried for the third one: no
// barrier, every reader polls the table's words for the launch's number.  With 148 CTAs
// the polls of a thousand words each crowd out the stores they wait for: 5.0 us
// where barrier and one reading take 2.5.)  A cooperative launch guarantees that all CTAs
// are resident, so every wait ends; all are bounded nevertheless, and a CTA that gives up
// sets KV_DEV_WAIT_EXPIRED and leaves (every other CTA then runs into the same limit).
// Barrier and histograms come in two sets used in turn; a launch clears the set of the
// next one.  The launch's number, which also says whose turn it is, lives in device
// memory, so that a captured launch can be replayed.  The selection without caller's scratch
// (SHARED = true) cannot rely on the launch before it: it clears its one set itself, while its
// keys are read (a memset ahead of the launch took 3.0 us of a 21.9 us pass over 1,000,003 entries).
// Measured, a pass with the event reduction: 4,096 entries 13.7 us, 0.9 M 26.7, 3.1 M 38.5, 18.8 M 158
// (notes per thread and whole chunks only, 32-bit touch counts: 32.5, 40.3, 59.9, 206).
//
// The same kernel also exists fused with the per-entry scoring pass (FUSED = true):
// every CTA first updates the entries of its own rows (posterior, EMA, score), their
// inputs streamed through shared-memory stages by asynchronous copies.  The touch counts are
// the packed ones of reduce_events, two bytes an entry, beside the caller's (against the caller's alone the
// event reduction of 18.8 M entries takes 32 us instead of 40, a pass 158 instead of 184, of 3.1 M
// entries 38.1 instead of 41.3), or, for a while after a trace that overflowed them, the caller's alone.  The event
// reduction stays a launch of its own ahead of it: its scattered gathers and atomics run slower
// beside this kernel's shared memory (11.5 M entries 101 -> 111 us), and for small traces a
// cooperative launch's own gap of ~3 us takes the place of the one saved (0.9 M 27.3 -> 27.5).
//
// And it exists for paged blocks (BLOCKS = true): an "entry" is then a block, whose score is
// the weighted sum over its heads, formed here from the entries' scores; on a pool of one
// partition the ordered write puts out the ids of all the block's entries.  (A kernel that
// wrote the blocks' scores ahead of this one and one that expanded the blocks behind it took
// 9.2 and 5.2 us of a 64.5 us pass over 393,216 blocks of 8 heads.)
#include <mutex>

#include "kv_score_device.cuh"
#include "kv_select_device.cuh"

namespace kvt {

constexpr uint32_t kPThreads = 1024;
constexpr uint32_t kPWarps = kPThreads / 32;
constexpr uint32_t kPChunk = kPThreads * 4;             // 4096 entries: one 16-byte vector per thread
constexpr uint32_t kPMaxRows = 64;                      // rows the bitmaps and tables are sized for
constexpr uint32_t kBarrierSpins = 1u << 22;
// The bracket reaches 2^17 .. 2^21 keys to either side of the hint; its bins, at most 2,048, are 2^7 ..
// 2^11 keys wide.
constexpr uint32_t kHalfMin = 1u << 17, kHalfMax = 1u << 21;
constexpr uint32_t kBracketShiftMin = 7, kBracketShiftMax = 11;
static_assert((2u * kHalfMax) >> kBracketShiftMax <= kHistBins, "the widest bracket has a bin for every key");
// A note: key - base of the bracket (22 bits), lane (5 bits), position in the lane's vector (2
// bits).  A kept note: key inside its bin (11 bits), lane, position, row (6 bits).
constexpr uint32_t kNoteKeyBits = 22, kKeptKeyBits = 11;
static_assert(2u * kHalfMax <= 1u << kNoteKeyBits && kNoteKeyBits + 7 <= 32, "a note holds any key of the bracket");
static_assert(kBracketShiftMax <= kKeptKeyBits && kPMaxRows <= 64, "a kept note holds any key of a bin, and its row");
// Fused form: the entry pass's inputs of one row in shared memory -- ema, decay and touch counts (4,096 words
// each), pair bytes (1,024 words), for the LRU policy last_epoch (4,096 words), packed touch counts (2,048 words)
__host__ __device__ constexpr uint32_t stage_words(bool packed, bool lru) {
  return 3u * kPChunk + kPThreads + (lru ? kPChunk : 0u) + (packed ? 2u * kPThreads : 0u);
}
constexpr uint64_t kPAlone = 2 * kPChunk;
constexpr uint64_t kPackedMaxEvents = 1ull << 27;       // (reduce_events: no overflow goes unseen)
constexpr unsigned long long kOverflowed = 1ull << 48;  // in SelectTurn::below
// Epochs that go on counting in 32 bits after the last one with a count that the packed ones cannot hold.  18.8 M
// entries: a pass takes 157 us, with 32-bit counts 175, the one that finds such a count out 300.  With 64 no
// trace that is hot now and then costs more than 32-bit counts for all epochs would (184 without packed ones).
constexpr uint32_t kWideEpochs = 64;
constexpr uint32_t kStages = 2;                         // rows in flight ahead of the one being finished
constexpr uint32_t kNoteCapMin = 128;                   // notes a warp keeps in shared memory, at least (the rest spills)

struct PArgs {
  const float* score;     // of the entries, whatever is selected
  const uint8_t* state;
  unsigned long long n;
  unsigned long long k;
  uint32_t* victims;
  SelectScalars* sel;
  SelectTurn* turns;      // [2] barrier and histograms of this launch (zero on entry) and of the next; shared scratch: [1]
  uint32_t* table;        // [n_rows][G] counts of every chunk
  unsigned long long* list;   // shared scratch: [kListMax] keys of the last bin, with their places
  unsigned long long* words;   // shared scratch (nullptr: the pool's own): number of the last call, then words of the first CTAs
  uint32_t* status;
  uint32_t n_full;        // full rows: chunks of 4,096 entries
  uint32_t last_len;      // entries of a CTA's piece of the last, shorter row (multiple of 128; 0: no such row)
  uint32_t n_rows;
  uint32_t note_cap;      // notes per warp in shared memory
  uint32_t stage_words;   // fused form: words of one stage
  uint32_t scratch_words; // words of notes and stages together (the plain path's key cache)
  PartCounts pc;          // partitions of the pool (the victims per partition are a by-product)
  uint32_t* spill;        // global scratch for the notes beyond note_cap: spill_stride words per warp (nullptr: no hints)
  uint32_t spill_stride;
  BlockGeom bg;           // block form: the pool's paged blocks ...
  uint32_t expand;        // ... and, on a pool of one partition, entries per block (0: victims are block indices)
  // the scoring pass of the fused form
  EntryState st;
  Predictor pd;
  HeadWeights hw;
  uint32_t epoch;
  const uint32_t* ev_entry;   // the trace that the packed touch counts hold
  unsigned long long n_events;
};

// The two halves of the bounded grid-wide barrier; work put between them overlaps the wait.
__device__ __forceinline__ void grid_arrive(unsigned int* counter) {
  __syncthreads();
  if (threadIdx.x == 0) asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(counter), "r"(1u) : "memory");
}

// false if the wait ran out
__device__ __forceinline__ bool grid_wait(const unsigned int* counter, unsigned int target) {
  int ok = 1;
  if (threadIdx.x == 0) {
    ok = 0;
    for (uint32_t it = 0; it < kBarrierSpins; ++it) {
      unsigned int v;
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(counter) : "memory");
      if (v >= target) { ok = 1; break; }
    }
  }
  return __syncthreads_and(ok) != 0;
}

// A word that carries the launch's number in its upper half.
__device__ __forceinline__ void publish_word(unsigned long long* p, uint32_t tag, uint32_t value) {
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"((unsigned long long)tag << 32 | value) : "memory");
}
__device__ __forceinline__ unsigned long long peek_word(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
// Waits (bounded) until the word carries the tag; its value, ok = false when the wait ran out.
__device__ __forceinline__ uint32_t await_word(const unsigned long long* p, uint32_t tag, bool& ok) {
  for (uint32_t it = 0; it < kBarrierSpins; ++it) {
    const unsigned long long v = peek_word(p);
    if ((uint32_t)(v >> 32) == tag) return (uint32_t)v;
  }
  ok = false;
  return 0;
}

// What a CTA adds to SelectTurn::below: its keys below the bracket, bit 31 of them kOverflowed.
template <bool FUSED>
__device__ __forceinline__ unsigned long long below_word(uint32_t s_below) {
  return FUSED ? (s_below & 0x7FFFFFFFu) | (s_below >> 31 ? kOverflowed : 0ull) : s_below;
}

// Finds the bin of a histogram (nbins <= 2048, a power of two) that contains rank k_rem (1-based):
// (bin, ranks before the bin, ranks in it, keys of this block in it) to every thread; bin is 0xFFFFFFFF
// when k_rem exceeds the histogram's total.  s_hist, the block's own histogram, is complete (a block
// barrier lies behind the last addition) and is cleared; with local it is the one that is looked at.  A
// block barrier must lie between two calls.
struct Pick { uint32_t bin, before, count, own; };
__device__ __forceinline__ Pick pick_bin(const uint32_t* hist, bool local, uint32_t* s_hist, uint32_t nbins,
                                         uint32_t k_rem, uint32_t* s_warp, uint4* s_pick) {
  const uint32_t t = threadIdx.x, lane = t & 31u, warp = t >> 5;
  const uint2 own = reinterpret_cast<const uint2*>(s_hist)[t];   // (bins from nbins on are empty)
  reinterpret_cast<uint2*>(s_hist)[t] = make_uint2(0u, 0u);
  uint2 c = own;
  if (!local) c = 2u * t < nbins ? __ldcg(reinterpret_cast<const uint2*>(hist) + t) : make_uint2(0u, 0u);
  const uint32_t v = c.x + c.y, all = __reduce_add_sync(0xFFFFFFFFu, v);
  if (lane == 0u) s_warp[warp] = all;
  if (t == 0) *s_pick = make_uint4(0xFFFFFFFFu, 0u, 0u, 0u);
  __syncthreads();
  // (one reduction instead of a second scan, and only the warp that holds the rank looks further)
  const uint32_t ahead = __reduce_add_sync(0xFFFFFFFFu, lane < warp ? s_warp[lane] : 0u);
  if (ahead < k_rem && k_rem - ahead <= all) {
    const uint32_t before = ahead + warp_scan_incl(v, lane) - v, before1 = before + c.x;
    if (before < k_rem && k_rem - before <= c.x) *s_pick = make_uint4(2u * t, before, c.x, own.x);
    if (before1 < k_rem && k_rem - before1 <= c.y) *s_pick = make_uint4(2u * t + 1u, before1, c.y, own.y);
  }
  __syncthreads();
  const uint4 p = *s_pick;
  return Pick{p.x, p.y, p.z, p.w};
}

// Scores of the four paged blocks b0 .. b0+3 (those below b1): the weighted sum over the block's
// heads, added in head order with every operation rounded once; resident bit j: all heads of
// block b0 + j are RESIDENT (the others score +inf).
__device__ __forceinline__ uint32_t block_scores4(const PArgs& a, unsigned long long b0, unsigned long long b1,
                                                  float s[4]) {
  const BlockGeom& bg = a.bg;
  uint32_t resident = 0;
  const int q0 = block_partition(bg, b0 < b1 ? b0 : 0);
  const uint32_t H0 = bg.heads[q0];
  const unsigned long long f0 = bg.entry_base[q0] + (b0 - bg.block_base[q0]) * H0;
#pragma unroll
  for (int j = 0; j < 4; ++j) s[j] = __int_as_float(0x7F800000);
  if (b0 + 4u <= b1 && b0 + 4u <= bg.block_base[q0 + 1] && (f0 & 3u) == 0u && ((H0 & 3u) == 0u || H0 <= 2u)) {
    // the four blocks' entries are aligned vectors
    const float4* sc = reinterpret_cast<const float4*>(a.score + f0);
    const uint32_t* st = reinterpret_cast<const uint32_t*>(a.state + f0);
    constexpr uint32_t kAll = KV_STATE_RESIDENT * 0x01010101u;
    float sum[4] = {0.0f, 0.0f, 0.0f, 0.0f};
    bool all[4] = {true, true, true, true};
    if ((H0 & 3u) == 0u) {
      const uint32_t per = H0 / 4u;   // vectors per block
#pragma unroll 2
      for (uint32_t v = 0; v < per; ++v) {
        float4 x[4];
        uint32_t y[4];
#pragma unroll
        for (uint32_t j = 0; j < 4; ++j) { x[j] = sc[j * per + v]; y[j] = st[j * per + v]; }
#pragma unroll
        for (uint32_t j = 0; j < 4; ++j) {
          sum[j] = __fadd_rn(__fadd_rn(__fadd_rn(__fadd_rn(sum[j], x[j].x), x[j].y), x[j].z), x[j].w);
          all[j] = all[j] && y[j] == kAll;
        }
      }
    } else {
      const float4 x = sc[0];
      const uint32_t y = st[0];
      if (H0 == 1u) {
        sum[0] = __fadd_rn(0.0f, x.x); sum[1] = __fadd_rn(0.0f, x.y);
        sum[2] = __fadd_rn(0.0f, x.z); sum[3] = __fadd_rn(0.0f, x.w);
#pragma unroll
        for (int j = 0; j < 4; ++j) all[j] = ((y >> (8 * j)) & 0xFFu) == KV_STATE_RESIDENT;
      } else {
        const float4 z = sc[1];
        const uint32_t w = st[1];
        sum[0] = __fadd_rn(__fadd_rn(0.0f, x.x), x.y); sum[1] = __fadd_rn(__fadd_rn(0.0f, x.z), x.w);
        sum[2] = __fadd_rn(__fadd_rn(0.0f, z.x), z.y); sum[3] = __fadd_rn(__fadd_rn(0.0f, z.z), z.w);
        all[0] = (y & 0xFFFFu) == (kAll & 0xFFFFu); all[1] = (y >> 16) == (kAll >> 16);
        all[2] = (w & 0xFFFFu) == (kAll & 0xFFFFu); all[3] = (w >> 16) == (kAll >> 16);
      }
    }
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (all[j]) { s[j] = __fmul_rn(bg.weight[q0], sum[j]); resident |= 1u << j; }
    return resident;
  }
  for (uint32_t j = 0; j < 4; ++j) {   // other head counts, partition boundaries, the ragged end
    const unsigned long long gb = b0 + j;
    if (gb >= b1) break;
    const int q = block_partition(bg, gb);
    const uint32_t H = bg.heads[q];
    const unsigned long long first = bg.entry_base[q] + (gb - bg.block_base[q]) * H;
    bool all = true;
    float sum = 0.0f;
    for (uint32_t h = 0; h < H; ++h) {
      all = all && a.state[first + h] == KV_STATE_RESIDENT;
      sum = __fadd_rn(sum, a.score[first + h]);
    }
    if (all) {
      const float x = __fmul_rn(bg.weight[q], sum);
      if (j == 0u) s[0] = x; else if (j == 1u) s[1] = x; else if (j == 2u) s[2] = x; else s[3] = x;
      resident |= 1u << j;
    }
  }
  return resident;
}

// PLAIN (fused form only): the policy is the Bayesian product and no partition is weighted.
// SHARED: on scratch that calls share which know nothing of each other.
template <bool FUSED, bool PLAIN, bool BLOCKS, bool SHARED>
__global__ void __launch_bounds__(kPThreads, 1) select_persistent_kernel(const PArgs a) {
  extern __shared__ __align__(16) uint32_t s_dyn[];
  // offsets in a stage
  constexpr uint32_t kAtTouch = 2u * kPChunk, kAtPair = 3u * kPChunk, kAtLast = kAtPair + kPThreads;
  const uint32_t at_packed = kAtLast + (!PLAIN && a.pd.policy == 2 ? kPChunk : 0u);
  const uint32_t n_words = a.n_rows * 128u;           // bitmap words: 128 per row
  // Bitmaps "below tau" and "equal to tau".  While they are filled, word 4*(row*32 + warp) + q
  // holds position q of the 32 lanes' vectors (a ballot); before they are counted they are
  // turned into natural order (bit j of word w: entry 32*w + j of the CTA).
  uint32_t* const s_bl = s_dyn;
  uint32_t* const s_be = s_bl + n_words;
  uint32_t* const s_nstart = s_be + n_words;          // [32][n_rows + 1] where a warp's notes of a row begin
  uint32_t* const s_note = s_nstart + (a.n_rows + 1u) * 32u;
  uint32_t* const s_stage = s_note + kPWarps * a.note_cap;
  // once phase A is over, notes and stages together are the key cache of the plain path
  __shared__ __align__(16) uint32_t s_hist[kHistBins];
  __shared__ uint32_t s_warp[32];
  __shared__ uint4 s_pick;
  __shared__ uint32_t s_below;
  __shared__ uint32_t s_listed, s_list_at;            // SHARED: keys that this CTA has put on the list, and where they begin
  constexpr uint32_t kListRows = SHARED ? kPMaxRows : 1u;
  __shared__ uint32_t s_less[kListRows], s_equal[kListRows];  // SHARED: listed keys before the CTA's chunk of a row, not of the row before
  __shared__ __align__(16) uint32_t s_wtot[kPMaxRows * 4];   // per 32 bitmap words: below | equal << 16
  __shared__ uint2 s_rowtot[kPMaxRows];               // (below, equal) of a row over all CTAs ...
  __shared__ uint2 s_colpre[kPMaxRows];               // ... and over the CTAs before this one
  __shared__ float sP[16];
  __shared__ PairStep s_pair[FUSED ? 16 : 1];
  const uint32_t t = threadIdx.x, lane = t & 31u, warp = t >> 5;
  const uint32_t lt = (1u << lane) - 1u;
  const uint32_t G = gridDim.x, g = blockIdx.x;
  const bool alone = G == 1u;   // one CTA: nothing is exchanged
  const uint32_t n_rows = a.n_rows;
  // (ids fit 31 bits)
  const uint32_t n = (uint32_t)a.n;
  auto row_base = [&](uint32_t r) -> uint32_t {
    return r < a.n_full ? (r * G + g) * kPChunk : a.n_full * G * kPChunk + g * a.last_len;
  };
  auto row_end = [&](uint32_t r) -> uint32_t {   // (may lie below row_base: an empty piece)
    const uint32_t e = row_base(r) + (r < a.n_full ? kPChunk : a.last_len);
    return e < n ? e : n;
  };
  // Phase boundaries of CTA 0 for timing studies (compiled in with -DKV_PHASE_STAMPS only: a
  // read of the global timer stalls the thread for a few hundred nanoseconds).
  auto stamp = [&](int i) {
#ifdef KV_PHASE_STAMPS
    if (blockIdx.x == 0 && t == 0) {
      unsigned long long ns;
      asm volatile("mov.u64 %0, %globaltimer;" : "=l"(ns));
      a.sel->phase_ns[i] = ns;
    }
#else
    (void)i;
#endif
  };
  wait_for_kernel_ahead();   // (a cooperative launch never starts early: nothing to wait for)
  stamp(0);

  // ---- prologue: the first rows' loads go out before anything else ----
  bool packed = FUSED && a.st.packed != nullptr;   // the trace is in the packed counts (those are zero otherwise)
  auto issue = [&](uint32_t r) {
    if constexpr (FUSED) {
      const uint32_t i0 = row_base(r) + 4u * t;
      if (r < n_rows && i0 + 4u <= row_end(r)) {
        uint32_t* dst = s_stage + (r % kStages) * a.stage_words;
        const uint32_t d0 = (uint32_t)__cvta_generic_to_shared(dst + 4u * t);
        const uint32_t d1 = (uint32_t)__cvta_generic_to_shared(dst + kAtPair + t);
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d0), "l"(a.st.ema + i0) : "memory");
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d0 + 4u * kPChunk), "l"(a.st.decay + i0) : "memory");
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(d1), "l"(a.st.pair + i0) : "memory");
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d0 + 4u * kAtTouch), "l"(a.st.touch + i0) : "memory");
        if (packed) {
          const uint32_t d3 = (uint32_t)__cvta_generic_to_shared(dst + at_packed + 2u * t);
          asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(d3), "l"(a.st.packed + i0 / 4u) : "memory");
        }
        if (!PLAIN && a.pd.policy == 2) {
          const uint32_t d2 = (uint32_t)__cvta_generic_to_shared(dst + kAtLast + 4u * t);
          asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d2), "l"(a.st.last_epoch + i0) : "memory");
        }
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  if constexpr (FUSED) {
#pragma unroll
    for (uint32_t r = 0; r < kStages; ++r) issue(r);
  }
  // Shared scratch: the first CTAs clear the counters, each says so in its word, with a number higher
  // than any a call has ever used there, and none adds to a counter before all have said so.  (The
  // numbers compare equal, so the CTAs of calls that overlap run into the limit instead of finishing
  // with different ones.)
  const unsigned long long call = SHARED ? a.words[0] + 1u : 0u;
  const uint32_t tag = SHARED ? (uint32_t)call : a.sel->serial + 1u;   // this launch's number
  SelectTurn* const turn = a.turns + (SHARED ? 0u : tag & 1u);
  unsigned int* const bar = &turn->bar;
  // (all of these loads together: one behind the answer of another costs 0.3 us)
  const uint32_t hint_valid = a.sel->hint_valid, hint_tau = a.sel->hint_tau;
  const unsigned long long hint_n = a.sel->hint_n;
  uint32_t half = a.sel->hint_half;   // (the bracket's width follows how well the hints have been doing)
  const uint32_t wide = packed ? a.sel->touch_wide : 0u;   // (as the event reduction has found it)
  packed = packed && wide == 0u;
  // where to note counts that the packed ones could not hold (nullptr: they have been tried)
  uint32_t* const hot = wide ? &a.sel->touch_hot : nullptr;
  const bool hint = !SHARED && (a.spill != nullptr) & (hint_valid != 0u) & (hint_n == a.n);
  if constexpr (FUSED) {
    // reuse estimates from the totals plus this epoch's counts (final: the event
    // reduction is an earlier launch)
    if (t < 16) {
      s_pair[t] = pair_step(a.pd, t);
      sP[t] = s_pair[t].estimate;
    }
  }
  for (uint32_t b = t; b < kHistBins; b += kPThreads) s_hist[b] = 0;
  for (uint32_t w = t; w < n_words; w += kPThreads) s_be[w] = 0;
  for (uint32_t w = g * kPThreads + t; w < sizeof(SelectTurn) / 4u; w += G * kPThreads)
    reinterpret_cast<uint32_t*>(a.turns + (SHARED ? 0u : (tag & 1u) ^ 1u))[w] = 0;
  if (t == 0) { s_below = 0; s_listed = 0; }
  if (SHARED && t < kPMaxRows) { s_less[t] = 0; s_equal[t] = 0; }
  half = half < kHalfMin ? kHalfMin : (half > kHalfMax ? kHalfMax : half);
  uint32_t bshift = kBracketShiftMin;                   // bins are 2^bshift keys wide
  while ((2u * half - 1u) >> bshift >= kHistBins) ++bshift;
  // The bracket [base0, base0 + 2 * half) stays between the keys of -inf and of +inf, so that its
  // ends are floats: comparing scores with them is comparing keys (the key order is the float
  // order, and the two zeros share a key).  An entry that is no candidate scores +inf.
  const uint32_t base_max = kKeyPosInf - 2u * half;
  uint32_t base0 = hint_tau > half ? hint_tau - half : 0u;
  base0 = base0 < kKeyNegInf ? kKeyNegInf : (base0 > base_max ? base_max : base0);
  const float neg_inf = __int_as_float(0xFF800000);
  const float lo_f = hint ? key_score(base0) : neg_inf, hi_f = hint ? key_score(base0 + 2u * half) : neg_inf;
  __syncthreads();
  constexpr uint32_t kClearing = (sizeof(SelectTurn) / 4u + kPThreads - 1u) / kPThreads;   // CTAs that clear something
  static_assert(kClearing <= kSharedCtas, "each of them has a word");
  if (SHARED && g < kClearing && t == 0)
    asm volatile("st.release.gpu.global.u64 [%0], %1;" ::"l"(a.words + 1 + g), "l"(call) : "memory");
  auto cleared = [&]() {   // what this thread knows of it; false if its wait ran out
    bool said = !SHARED || t >= kClearing || t >= G;
    if constexpr (SHARED) {
      for (uint32_t it = 0; it < kBarrierSpins && !said; ++it) {
        unsigned long long v;
        asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(a.words + 1 + t) : "memory");
        said = v == call;
      }
    }
    return said;
  };

  // ---- phase A ----
  uint32_t n_noted = 0;     // notes of this warp
  uint32_t n_below = 0;     // keys of this thread below the bracket
  bool overflowed = false;  // a packed count of this thread's has
  uint32_t* const my_nstart = s_nstart + warp * (n_rows + 1u);
  uint32_t* const my_note = s_note + warp * a.note_cap;
  uint32_t* const my_spill = a.spill + (unsigned long long)(g * kPWarps + warp) * a.spill_stride;
  auto note_put = [&](uint32_t at, uint32_t note) {
    if (at < a.note_cap) my_note[at] = note;
    else my_spill[at - a.note_cap] = note;   // (a dense slice: the rest goes to L2)
  };
  auto note_get = [&](uint32_t at) { return at < a.note_cap ? my_note[at] : __ldcg(my_spill + (at - a.note_cap)); };
  // The histograms, the list and the table were written a pass ago and have left the L2 since: fetch their
  // lines while the last rows are worked on (a miss inside an exchange cost 1-4 us).
  auto warm_lines = [&]() {
    constexpr uint32_t kTurnLines = (sizeof(SelectTurn) + 127u) / 128u, kListLines = SHARED ? kListMax * 8u / 128u : 0u;
    const uint32_t lines = kTurnLines + kListLines + (n_rows * G * 4u + 127u) / 128u;
    for (uint32_t l = t * G + g; l < lines; l += kPThreads * G) {
      const char* p = l < kTurnLines ? reinterpret_cast<const char*>(turn) + 128u * l
                      : l < kTurnLines + kListLines ? reinterpret_cast<const char*>(a.list) + 128u * (l - kTurnLines)
                                                    : reinterpret_cast<const char*>(a.table) + 128u * (l - kTurnLines - kListLines);
      asm volatile("prefetch.global.L2 [%0];" ::"l"(p));
    }
  };
  // (row r, the thread's four scores): the below bits, and a note for each key inside the bracket
  auto classify = [&](uint32_t r, const float s[4]) {
    if (lane == 0) my_nstart[r] = n_noted;
    bool in[4];
    uint32_t wl[4], wi[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      // (a NaN is neither below nor inside; the scores that this kernel forms are positive ones, which
      // come behind all numbers, but an array may hold negative ones, which come before)
      bool lo = s[q] < lo_f;
      if constexpr (!FUSED && !BLOCKS) lo = lo || __float_as_uint(s[q]) > 0xFF800000u;
      in[q] = s[q] < hi_f && !lo;
      n_below += lo;
      wl[q] = __ballot_sync(0xFFFFFFFFu, lo);
      wi[q] = __ballot_sync(0xFFFFFFFFu, in[q]);
    }
    if (lane == 0) *reinterpret_cast<uint4*>(s_bl + 4u * (r * 32u + warp)) = make_uint4(wl[0], wl[1], wl[2], wl[3]);
    if (wi[0] | wi[1] | wi[2] | wi[3]) {
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        if (in[q]) {
          const uint32_t d = number_key(s[q]) - base0;   // (inside the bracket: no NaN)
          // (additions of 1 to one bin are merged by the hardware: collecting a thread's equal bins in a
          // register first cost 0.7 of 42.1 us at 3.1 M entries, 1.7 of 20.4 in the plain radix select)
          atomicAdd(&s_hist[d >> bshift], 1u);
          note_put(n_noted + (uint32_t)__popc(wi[q] & lt), d | lane << kNoteKeyBits | (uint32_t)q << (kNoteKeyBits + 5));
        }
        n_noted += (uint32_t)__popc(wi[q]);
      }
    }
  };
  const float inf = __int_as_float(0x7F800000);
  if constexpr (FUSED) {
    const int policy = PLAIN ? 0 : a.pd.policy;
    for (uint32_t r = 0; r < n_rows; ++r) {
      asm volatile("cp.async.wait_group %0;" ::"n"(kStages - 1u) : "memory");   // (that many newer groups may be pending)
      const uint32_t i0 = row_base(r) + 4u * t, i1 = row_end(r);
      float s[4] = {inf, inf, inf, inf};
      if (i0 + 4u <= i1) {
        const uint32_t* src = s_stage + (r % kStages) * a.stage_words;
        EntryVec cur;
        cur.e = *reinterpret_cast<const float4*>(src + 4u * t);
        cur.d = *reinterpret_cast<const float4*>(src + kPChunk + 4u * t);
        cur.pr4 = src[kAtPair + t];
        uint2 counts = make_uint2(0, 0);
        if (packed) counts = *reinterpret_cast<const uint2*>(src + at_packed + 2u * t);
        cur.t = *reinterpret_cast<const uint4*>(src + kAtTouch + 4u * t);
        cur.le = make_uint4(0, 0, 0, 0);
        if (!PLAIN && policy == 2) cur.le = *reinterpret_cast<const uint4*>(src + kAtLast + 4u * t);
        issue(r + kStages);
        if (!take_touches(a.st, i0 / 4, counts, cur.t)) {
          overflowed = true;   // (these entries are left as they are until the trace has been counted again)
        } else {
          float4 sc;
          entry_finish4<true, PLAIN>(a.st, i0 / 4, cur, sP, policy, a.epoch, a.hw, hot, sc);
          s[0] = sc.x; s[1] = sc.y; s[2] = sc.z; s[3] = sc.w;
        }
      } else {
        issue(r + kStages);
        if (i0 < i1) {   // the pool's ragged end
          uint32_t c[4] = {0, 0, 0, 0};
          if (packed && !unpack_touches(__ldcg(reinterpret_cast<const uint2*>(a.st.packed) + i0 / 4u), c)) {
            overflowed = true;
          } else {
            if (packed) a.st.packed[i0 / 4u] = 0;
#pragma unroll
            for (int j = 0; j < 4; ++j)
              if (i0 + j < i1) entry_update1(a.st, i0 + j, sP, policy, a.epoch, a.hw, c[j], hot, s[j]);
          }
        }
      }
      if (r + 2u == n_rows || n_rows == 1u) warm_lines();
      classify(r, s);
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
  } else if (!hint) {
    warm_lines();
  } else {
    constexpr uint32_t kInFlight = BLOCKS ? 1 : 4;   // rows whose loads are in flight
    float4 sc[kInFlight];
    uint32_t st4[kInFlight];
    auto load = [&](uint32_t r, uint32_t u) {
      const uint32_t i0 = row_base(r) + 4u * t;
      if (!BLOCKS && r < n_rows && i0 + 4u <= row_end(r)) {
        sc[u] = __ldcg(reinterpret_cast<const float4*>(a.score + i0));
        st4[u] = __ldcg(reinterpret_cast<const uint32_t*>(a.state + i0));
      }
    };
#pragma unroll
    for (uint32_t u = 0; u < kInFlight; ++u) load(u, u);
    warm_lines();
    for (uint32_t r = 0; r < n_rows; r += kInFlight) {
#pragma unroll
      for (uint32_t u = 0; u < kInFlight; ++u) {
        if (r + u < n_rows) {
          const uint32_t i0 = row_base(r + u) + 4u * t, i1 = row_end(r + u);
          float s[4] = {inf, inf, inf, inf};
          if (BLOCKS) {
            (void)block_scores4(a, i0, i1, s);
          } else if (i0 + 4u <= i1) {
            s[0] = (st4[u] & 0xFFu) == KV_STATE_RESIDENT ? sc[u].x : inf;
            s[1] = ((st4[u] >> 8) & 0xFFu) == KV_STATE_RESIDENT ? sc[u].y : inf;
            s[2] = ((st4[u] >> 16) & 0xFFu) == KV_STATE_RESIDENT ? sc[u].z : inf;
            s[3] = (st4[u] >> 24) == KV_STATE_RESIDENT ? sc[u].w : inf;
          } else {
#pragma unroll
            for (int j = 0; j < 4; ++j)
              if (i0 + j < i1 && a.state[i0 + j] == KV_STATE_RESIDENT) s[j] = a.score[i0 + j];
          }
          load(r + u + kInFlight, u);
          classify(r + u, s);
        }
      }
    }
  }
  stamp(1);
  // (number 0 marks a word never written; the turns alternate across the wrap too)
  auto end_turn = [&]() {
    if (SHARED) atomicMax(a.words, call);
    else a.sel->serial = tag == 0xFFFFFFFFu ? 1u : tag;
  };
  uint32_t nbar = 0;        // grid barriers passed
  bool ok = true, hint_hit = false, recounted = false;
  unsigned long long below = 0;   // keys below the bracket, of all CTAs
  if (FUSED || hint) {
    n_below = __reduce_add_sync(0xFFFFFFFFu, n_below);
    if (lane == 0) {
      my_nstart[n_rows] = n_noted;
      if (n_below) atomicAdd(&s_below, n_below);
    }
    if (FUSED && overflowed) atomicOr(&s_below, 1u << 31);   // (a CTA has fewer entries than that)
    __syncthreads();
    if (!alone) {
      if (hint) add_pair(turn->hist[0] + 2u * t, reinterpret_cast<const uint2*>(s_hist)[t]);
      if (t == 0 && s_below) atomicAdd(&turn->below, below_word<FUSED>(s_below));
      grid_arrive(bar);
      ok = grid_wait(bar, ++nbar * G);
    }
    stamp(2);
    if (!ok) goto fail;
  }
  {
    // ---- phase B: narrow [base, base + 2^shift) around rank k, one histogram per exchange ----
    // Every CTA reads the same global data, so all of them take the same path.
    uint32_t tau = 0;
    uint32_t k_rem = (uint32_t)a.k;   // (k is at most n)
    bool found = true;
    // The CTA's histogram joins the others' in histogram h; false if the wait ran out.
    auto exchange_hist = [&](uint32_t h, uint32_t nbins, bool ready = true) {
      if constexpr (SHARED) {
        if (!__syncthreads_and(ready)) return false;
      } else {
        __syncthreads();
      }
      if (alone) return true;
      if (2u * t < nbins) add_pair(turn->hist[h] + 2u * t, reinterpret_cast<const uint2*>(s_hist)[t]);
      grid_arrive(bar);
      return grid_wait(bar, ++nbar * G);
    };
    // Radix select on shared scratch: as soon as a bin's keys are few, they go on a list with their places,
    // beside the counts of the chunks, and every CTA finds tau on it by itself: one exchange (two, for small
    // arrays) and a pass over the keys less.  1,000,003 entries 18.4 -> 17.0 us.  (Up to 2,048 keys: 17.5, up
    // to 4,096: 18.2.  Behind a hint, where one exchange follows in any case, it gave nothing.)  Every CTA
    // decides alike: the count is the pool's.  `base` is the bin's first key, 2^list_bits its width.
    bool listed = false;
    uint32_t base = 0, list_bits = 0, n_listed = 0;
    Pick pick{0u, 0u, 0u, 0u};
    uint32_t bin_k = 0;
    if (hint) {
      below = alone ? below_word<FUSED>(s_below) : __ldcg(&turn->below);   // (in flight together with the histogram)
      const bool above = a.k > below;   // (false beside kOverflowed)
      pick = pick_bin(turn->hist[0], alone, s_hist, kHistBins, above ? (uint32_t)(a.k - below) : 1u, s_warp, &s_pick);
      hint_hit = above && pick.bin != 0xFFFFFFFFu;
      if (hint_hit) {
        k_rem = (uint32_t)(a.k - below) - pick.before;
        bin_k = pick.bin;
      }
      if (g == 0 && t == 0) atomicAdd(hint_hit ? &a.sel->n_hint_hit : &a.sel->n_hint_miss, 1u);
    }
    if constexpr (FUSED) {
      // A packed count overflowed somewhere.  The words that hold one are the only ones that are not zero by
      // now: the touches of their entries are counted again, in the 32-bit array, these entries get their
      // scoring step, and the selection starts from the scores.  (kWideEpochs epochs are then counted in the
      // 32-bit array from the start.)
      if (!hint) below = alone ? below_word<FUSED>(s_below) : __ldcg(&turn->below);
      recounted = below >= kOverflowed;
      if (recounted) {
        hint_hit = false;
        constexpr uint32_t kAtOnce = 4;   // (two loads behind one another, four of each in flight)
        for (unsigned long long e = g * kPThreads + t; e < a.n_events; e += kAtOnce * G * kPThreads) {
          uint32_t id[kAtOnce];
          unsigned long long w[kAtOnce];
#pragma unroll
          for (uint32_t j = 0; j < kAtOnce; ++j)
            id[j] = e + j * G * kPThreads < a.n_events ? a.ev_entry[e + j * G * kPThreads] : 0xFFFFFFFFu;
#pragma unroll
          for (uint32_t j = 0; j < kAtOnce; ++j) w[j] = id[j] < n ? __ldcg(a.st.packed + id[j] / 4u) : 0ull;
#pragma unroll
          for (uint32_t j = 0; j < kAtOnce; ++j)
            if (w[j] && !(a.st.pair[id[j]] & kPairFree)) atomicAdd(a.st.touch + id[j], 1u);
        }
        if (alone) {
          __syncthreads();
        } else {
          grid_arrive(bar);
          ok = grid_wait(bar, ++nbar * G);
          if (!ok) goto fail;
        }
        for (uint32_t r = 0; r < n_rows; ++r) {
          const uint32_t i0 = row_base(r) + 4u * t, i1 = row_end(r), v = i0 / 4u;
          if (i0 >= i1 || __ldcg(a.st.packed + v) == 0ull) continue;
          a.st.packed[v] = 0;
#pragma unroll 1
          for (uint32_t i = i0; i < i1 && i < i0 + 4u; ++i) {
            float s;
            entry_update1(a.st, i, sP, PLAIN ? 0 : a.pd.policy, a.epoch, a.hw, 0u, nullptr, s);
          }
        }
      }
    }
    // keys of the thread's vector of row r, from the arrays; entries past the row's end or not
    // RESIDENT give kKeyExcluded
    // (scores that the kernel forms itself: a NaN has the one bit pattern that arithmetic gives)
    auto key_of = [](float x) { return FUSED || BLOCKS ? number_key(x) : score_key(x); };
    auto load_keys = [&](uint32_t r, uint32_t key[4]) {
      const uint32_t i0 = row_base(r) + 4u * t, i1 = row_end(r);
      if (BLOCKS) {
        float s[4];
        const uint32_t resident = block_scores4(a, i0, i1, s);
#pragma unroll
        for (int j = 0; j < 4; ++j) key[j] = (resident >> j) & 1u ? key_of(s[j]) : kKeyExcluded;
      } else if (i0 + 4u <= i1) {
        const float4 sc = __ldcg(reinterpret_cast<const float4*>(a.score + i0));
        const uint32_t st4 = __ldcg(reinterpret_cast<const uint32_t*>(a.state + i0));
        key[0] = (st4 & 0xFFu) == KV_STATE_RESIDENT ? key_of(sc.x) : kKeyExcluded;
        key[1] = ((st4 >> 8) & 0xFFu) == KV_STATE_RESIDENT ? key_of(sc.y) : kKeyExcluded;
        key[2] = ((st4 >> 16) & 0xFFu) == KV_STATE_RESIDENT ? key_of(sc.z) : kKeyExcluded;
        key[3] = (st4 >> 24) == KV_STATE_RESIDENT ? key_of(sc.w) : kKeyExcluded;
      } else {
#pragma unroll
        for (int j = 0; j < 4; ++j)
          key[j] = (i0 + j < i1 && a.state[i0 + j] == KV_STATE_RESIDENT) ? key_of(a.score[i0 + j]) : kKeyExcluded;
      }
    };
    // A pass over the CTA's keys, rows in order: body(r, key) sees the thread's four keys of row
    // r, all threads in lock step.  The first rows' keys stay in the key cache (the threads read
    // back only what they wrote); the others are re-read from L2, two rows at a time.
    uint32_t* const cache = s_note;
    const uint32_t cached_rows = a.scratch_words / kPChunk < n_rows ? a.scratch_words / kPChunk : n_rows;
    uint32_t rows_in_cache = 0;
    auto for_keys = [&](auto body) {
      for (uint32_t r = 0; r < rows_in_cache; ++r) {
        const uint4 v = *reinterpret_cast<const uint4*>(cache + r * kPChunk + 4u * t);
        const uint32_t key[4] = {v.x, v.y, v.z, v.w};
        body(r, key);
      }
      for (uint32_t r = rows_in_cache; r < n_rows; r += 2) {
        uint32_t k0[4], k1[4];
        load_keys(r, k0);
        if (r + 1 < n_rows) load_keys(r + 1, k1);
        if (r < cached_rows) *reinterpret_cast<uint4*>(cache + r * kPChunk + 4u * t) = make_uint4(k0[0], k0[1], k0[2], k0[3]);
        if (r + 1 < cached_rows) *reinterpret_cast<uint4*>(cache + (r + 1) * kPChunk + 4u * t) = make_uint4(k1[0], k1[1], k1[2], k1[3]);
        body(r, k0);
        if (r + 1 < n_rows) body(r + 1, k1);
      }
      rows_in_cache = cached_rows;
    };

    if (hint_hit) {
      // One pass over the notes: those of the bins before bin_k set their bits, those of bin_k
      // enter the histogram of its single keys and stay (moved to the front of the list).
      const uint32_t n_bins = 1u << bshift;
      uint32_t row = 0, row_ends = my_nstart[1];   // row of this lane's note (its places ascend)
      uint32_t n_kept = 0;
      for (uint32_t p0 = 0; p0 < n_noted; p0 += 128u) {
        uint32_t v[4];
#pragma unroll
        for (uint32_t u = 0; u < 4u; ++u) {
          const uint32_t p = p0 + 32u * u + lane;
          v[u] = p < n_noted ? note_get(p) : 0xFFFFFFFFu;
        }
        __syncwarp();
#pragma unroll
        for (uint32_t u = 0; u < 4u; ++u) {
          const uint32_t p = p0 + 32u * u + lane;
          const bool in = p < n_noted;
          while (in && p >= row_ends) { ++row; row_ends = my_nstart[row + 1u]; }
          const uint32_t d = v[u] & ((1u << kNoteKeyBits) - 1u), b = d >> bshift, at = v[u] >> kNoteKeyBits;
          if (in && b < bin_k) atomicOr(&s_bl[4u * (row * 32u + warp) + (at >> 5)], 1u << (at & 31u));
          const bool keep = in && b == bin_k;
          const uint32_t m = __ballot_sync(0xFFFFFFFFu, keep);
          if (keep) {
            const uint32_t low = d & (n_bins - 1u);
            atomicAdd(&s_hist[low], 1u);
            note_put(n_kept + (uint32_t)__popc(m & lt), low | at << kKeptKeyBits | row << (kKeptKeyBits + 7));
          }
          n_kept += (uint32_t)__popc(m);
        }
      }
      __syncwarp();
      stamp(8);
      ok = exchange_hist(1, n_bins);
      stamp(3);
      if (!ok) goto fail;
      pick = pick_bin(turn->hist[1], alone, s_hist, n_bins, k_rem, s_warp, &s_pick);
      found = pick.bin != 0xFFFFFFFFu;
      k_rem -= pick.before;
      const uint32_t tau_low = found ? pick.bin : 0u;
      tau = base0 + (bin_k << bshift) + tau_low;
      // phase C from the kept notes: those below tau and equal to it set their bits
      for (uint32_t p = lane; p < n_kept; p += 32u) {
        const uint32_t v = note_get(p), low = v & ((1u << kKeptKeyBits) - 1u), at = (v >> kKeptKeyBits) & 127u;
        const uint32_t w = 4u * ((v >> (kKeptKeyBits + 7)) * 32u + warp) + (at >> 5);
        if (low <= tau_low) atomicOr(low < tau_low ? &s_bl[w] : &s_be[w], 1u << (at & 31u));
      }
    } else {
      // plain radix select: digits of 11, 11 and 10 bits, or until the keys that are left fit the list
      uint32_t h = hint ? 1u : 0u;   // (histogram 0 holds the bracket's counts of this launch)
      k_rem = (uint32_t)a.k;
#pragma unroll 1
      for (int digit = 0; digit < 3 && !(SHARED && listed); ++digit) {
        const uint32_t shift = digit == 0 ? 21u : digit == 1 ? 10u : 0u, top = digit == 2 ? 10u : 11u;
        __syncthreads();   // (the notes are dead: their space becomes the key cache)
        for_keys([&](uint32_t, const uint32_t key[4]) {
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const uint32_t d = (key[q] - base) >> shift;
            if (key[q] != kKeyExcluded && key[q] >= base && (digit == 0 || (d >> top) == 0u)) atomicAdd(&s_hist[d], 1u);
          }
        });
        ok = exchange_hist(h, 1u << top, digit != 0 || alone || cleared());
        if (digit == 1) stamp(3);
        if (!ok) goto fail;
        pick = pick_bin(turn->hist[h], alone, s_hist, 1u << top, k_rem, s_warp, &s_pick);
        ++h;
        found = found && pick.bin != 0xFFFFFFFFu;
        k_rem -= pick.before;
        base += (pick.bin & (kHistBins - 1u)) << shift;
        listed = SHARED && !alone && found && shift != 0u && pick.count <= kListMax;
        list_bits = shift;
      }
      tau = base;
      if (SHARED && listed) {
        n_listed = pick.count;
        if (t == 0 && pick.own) s_list_at = atomicAdd(&turn->listed, pick.own);
        __syncthreads();
      }
      // phase C from the keys
      for_keys([&](uint32_t r, const uint32_t key[4]) {
        uint32_t wl[4], we[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          wl[q] = __ballot_sync(0xFFFFFFFFu, key[q] < tau && key[q] != kKeyExcluded);
          // (equal to tau, or, before tau is known, in the last bin)
          const bool in = (SHARED ? key[q] >= tau && ((key[q] - tau) >> list_bits) == 0u : key[q] == tau) && key[q] != kKeyExcluded;
          we[q] = __ballot_sync(0xFFFFFFFFu, in);
          if (SHARED && listed && we[q]) {
            uint32_t at = 0;
            if (lane == 0) at = s_list_at + atomicAdd(&s_listed, (uint32_t)__popc(we[q]));
            at = __shfl_sync(0xFFFFFFFFu, at, 0);
            at += (uint32_t)__popc(we[q] & lt);
            if (in && at < kListMax) a.list[at] = (unsigned long long)(key[q] - tau) << 28 | r << 22 | g << 12 | (4u * t + (uint32_t)q);
          }
          if (SHARED && listed) we[q] = 0u;
        }
        if (lane == 0) {
          *reinterpret_cast<uint4*>(s_bl + 4u * (r * 32u + warp)) = make_uint4(wl[0], wl[1], wl[2], wl[3]);
          *reinterpret_cast<uint4*>(s_be + 4u * (r * 32u + warp)) = make_uint4(we[0], we[1], we[2], we[3]);
        }
      });
    }
    stamp(10);
    __syncthreads();

    // ---- last exchange: the counts of every chunk, (below | equal << 13), row after row, and the list ----
    for (uint32_t r = warp; r < n_rows; r += kPWarps) {
      const uint4 x = reinterpret_cast<const uint4*>(s_bl)[32u * r + lane], y = reinterpret_cast<const uint4*>(s_be)[32u * r + lane];
      const uint32_t l = (uint32_t)(__popc(x.x) + __popc(x.y) + __popc(x.z) + __popc(x.w));
      const uint32_t e = (uint32_t)(__popc(y.x) + __popc(y.y) + __popc(y.z) + __popc(y.w));
      const uint32_t sum = __reduce_add_sync(0xFFFFFFFFu, l | e << 16);   // at most 4,096 in either half
      if (lane == 0u) {
        if (alone) {
          s_rowtot[r] = make_uint2(sum & 0xFFFFu, sum >> 16);
          s_colpre[r] = make_uint2(0u, 0u);
        } else {
          a.table[r * G + g] = (sum & 0xFFFFu) | (sum >> 16) << 13;
        }
      }
    }
    if (alone) __syncthreads(); else grid_arrive(bar);
    stamp(5);
    if constexpr (FUSED) {
      // every CTA has long formed its estimates: the epoch's counts can be folded in (here, where
      // the CTA waits for the others anyway)
      if (g == 0 && t >= kPThreads - 32u && lane < 16u) {
        commit_predictor(a.pd, lane, s_pair[lane]);
        if (lane == 0u && (wide || recounted)) {
          a.sel->touch_wide = recounted || __ldcg(hot) ? kWideEpochs : wide - 1u;
          a.sel->touch_hot = 0;
        }
      }
    }
    // (while the others arrive: 3.1 M entries 39.3 -> 38.0 us a pass against doing it before) the bitmaps
    // into natural order, and population counts per 32 words.  Thread t owns words t, t + 1024, ...: a
    // row's 128 words belong to four neighbouring warps.
    const uint32_t n_rounds = (n_words + kPThreads - 1u) / kPThreads;
    for (uint32_t rd = 0; rd < n_rounds; ++rd) {
      const uint32_t W = rd * kPThreads + t;
      if (W < n_words) {   // (n_words is a multiple of 128: the whole warp)
        const uint4 x = reinterpret_cast<const uint4*>(s_bl)[W >> 2], y = reinterpret_cast<const uint4*>(s_be)[W >> 2];
        const uint32_t sh = 8u * (W & 3u);
        const uint32_t bl = interleave4(x.x >> sh, x.y >> sh, x.z >> sh, x.w >> sh);
        const uint32_t be = (y.x | y.y | y.z | y.w) ? interleave4(y.x >> sh, y.y >> sh, y.z >> sh, y.w >> sh) : 0u;
        __syncwarp();
        s_bl[W] = bl;
        s_be[W] = be;
        const uint32_t c = __reduce_add_sync(0xFFFFFFFFu, (uint32_t)__popc(bl) | (uint32_t)__popc(be) << 16);
        if (lane == 0) s_wtot[rd * kPWarps + warp] = c;
      }
    }
    if (!alone) ok = grid_wait(bar, ++nbar * G);
    stamp(6);
    if (!ok) goto fail;
    static_assert(kListMax == kPThreads, "a thread looks at one listed key");
    unsigned long long item = ~0ull;
    if (SHARED && listed && t < n_listed) item = __ldcg(a.list + t);
    const uint32_t item_low = (uint32_t)(item >> 28);
    // s_hist gets the digit at bit w of those listed keys that share the digits above it with `low`
    auto list_digit = [&](uint32_t w, uint32_t step, uint32_t low) {
      if (item != ~0ull && ((item_low ^ low) >> (w + step)) == 0u) atomicAdd(&s_hist[(item_low >> w) & ((1u << step) - 1u)], 1u);
    };
    uint32_t list_step = list_bits < 11u ? list_bits : 11u;
    if (SHARED && listed) list_digit(list_bits - list_step, list_step, 0u);
    for (uint32_t r = warp; r < n_rows && !alone; r += kPWarps) {
      uint32_t tl = 0, te = 0, pl = 0, pe = 0;
      for (uint32_t c0 = 0; c0 < G; c0 += 160u) {
        uint32_t v[5];   // (loads in flight together)
#pragma unroll
        for (uint32_t u = 0; u < 5u; ++u) {
          const uint32_t c = c0 + 32u * u + lane;
          v[u] = c < G ? __ldcg(&a.table[r * G + c]) : 0u;
        }
#pragma unroll
        for (uint32_t u = 0; u < 5u; ++u) {
          const uint32_t l = v[u] & 0x1FFFu, e = v[u] >> 13;
          tl += l; te += e;
          if (c0 + 32u * u + lane < g) { pl += l; pe += e; }
        }
      }
      tl = __reduce_add_sync(0xFFFFFFFFu, tl);
      te = __reduce_add_sync(0xFFFFFFFFu, te);
      pl = __reduce_add_sync(0xFFFFFFFFu, pl);
      pe = __reduce_add_sync(0xFFFFFFFFu, pe);
      if (lane == 0) { s_rowtot[r] = make_uint2(tl, te); s_colpre[r] = make_uint2(pl, pe); }
    }
    __syncthreads();
    uint32_t list_less = 0, list_equal = 0;   // listed keys below tau, and equal to it
    if (SHARED && listed) {
      // Every CTA finds tau among the listed keys, counts those that come before its chunks and sets the
      // bits of its own.
      list_less = k_rem;
      uint32_t low = 0;
      for (uint32_t w = list_bits - list_step;;) {
        pick = pick_bin(nullptr, true, s_hist, 1u << list_step, k_rem, s_warp, &s_pick);
        found = found && pick.bin != 0xFFFFFFFFu;
        k_rem -= pick.before;
        low |= (pick.bin & ((1u << list_step) - 1u)) << w;
        if (w == 0u) break;
        list_step = w;   // (21 bits: 11 and 10)
        w = 0u;
        list_digit(w, list_step, low);
        __syncthreads();
      }
      tau = base + low;
      list_less -= k_rem;
      list_equal = pick.count;
      if (item != ~0ull && item_low <= low) {
        const bool less = item_low < low;
        const uint32_t where = (uint32_t)item, row = (where >> 22) & 63u, of = (where >> 12) & 1023u;
        const uint32_t W = row * 128u + ((where >> 5) & 127u);
        const uint32_t from = row + (of >= g ? 1u : 0u);   // the first row whose chunk comes behind the key
        if (from < n_rows) atomicAdd(less ? &s_less[from] : &s_equal[from], 1u);
        if (of == g && row < n_rows) {
          atomicOr(less ? &s_bl[W] : &s_be[W], 1u << (where & 31u));
          atomicAdd(&s_wtot[W >> 5], less ? 1u : 1u << 16);
        }
      }
      __syncthreads();
    }
    const uint32_t need_eq = k_rem;
    // ---- phase D: where this CTA's chunks start, and the ordered write ----
    // Lane r of every warp: what the pool holds before this CTA's chunk of row r (and of row r + 32).
    uint32_t all_l, all_e, rl0, re0, rl1 = 0, re1 = 0;
    {
      const uint2 v0 = lane < n_rows ? s_rowtot[lane] : make_uint2(0u, 0u);
      const uint32_t i0 = warp_scan_incl(v0.x, lane), j0 = warp_scan_incl(v0.y, lane);
      all_l = __shfl_sync(0xFFFFFFFFu, i0, 31);
      all_e = __shfl_sync(0xFFFFFFFFu, j0, 31);
      const uint2 p0 = lane < n_rows ? s_colpre[lane] : make_uint2(0u, 0u);
      rl0 = i0 - v0.x + p0.x;
      re0 = j0 - v0.y + p0.y;
      if (n_rows > 32u) {
        const uint2 v1 = lane + 32u < n_rows ? s_rowtot[lane + 32u] : make_uint2(0u, 0u);
        const uint32_t i1 = warp_scan_incl(v1.x, lane), j1 = warp_scan_incl(v1.y, lane);
        const uint2 p1 = lane + 32u < n_rows ? s_colpre[lane + 32u] : make_uint2(0u, 0u);
        rl1 = all_l + i1 - v1.x + p1.x;
        re1 = all_e + j1 - v1.y + p1.y;
        all_l += __shfl_sync(0xFFFFFFFFu, i1, 31);
        all_e += __shfl_sync(0xFFFFFFFFu, j1, 31);
      }
      if (SHARED && listed) {
        const uint32_t l0 = warp_scan_incl(s_less[lane], lane), e0 = warp_scan_incl(s_equal[lane], lane);
        rl0 += l0;
        re0 += e0;
        if (n_rows > 32u) {
          rl1 += __shfl_sync(0xFFFFFFFFu, l0, 31) + warp_scan_incl(s_less[lane + 32u], lane);
          re1 += __shfl_sync(0xFFFFFFFFu, e0, 31) + warp_scan_incl(s_equal[lane + 32u], lane);
        }
        all_l += list_less;
        all_e += list_equal;
      }
    }
    const uint32_t eq_room = need_eq;
    const unsigned long long got = (unsigned long long)all_l + (all_e < eq_room ? all_e : eq_room);
    // (block form, one partition: the entries of block gb, the pos-th of the selected ones)
    auto write_block = [&](uint32_t pos, uint32_t gb) {
      const uint32_t H = a.expand, first = gb * H;
      uint32_t* const out = a.victims + (unsigned long long)pos * H;
      if ((H & 3u) == 0u) {
        for (uint32_t h = 0; h < H; h += 4u)
          *reinterpret_cast<uint4*>(out + h) = make_uint4(first + h, first + h + 1u, first + h + 2u, first + h + 3u);
      } else {
        for (uint32_t h = 0; h < H; ++h) out[h] = first + h;
      }
    };
    // (the notes are dead: their space holds a warp's ids on their way out)
    const uint32_t room = a.scratch_words / kPWarps;
    uint32_t* const ids = s_note + warp * room;
    // With L entries below tau and E entries equal to tau before it in id order, an entry below
    // tau goes to L + min(E, need_eq) and an entry equal to tau, taken while E < need_eq, to L + E.
    for (uint32_t rd = 0; rd < n_rounds; ++rd) {
      const uint32_t W = rd * kPThreads + t, row = W >> 7;   // (one row per warp)
      if (row >= n_rows) break;
      const uint32_t bl = s_bl[W], be = s_be[W];
      const uint32_t c = (uint32_t)__popc(bl) | (uint32_t)__popc(be) << 16;
      uint32_t ex = warp_scan_incl(c, lane) - c;
      const uint4 wt = reinterpret_cast<const uint4*>(s_wtot)[row];
      const uint32_t quarter = warp & 3u;
      ex += (quarter > 0u ? wt.x : 0u) + (quarter > 1u ? wt.y : 0u) + (quarter > 2u ? wt.z : 0u);
      uint32_t L = __shfl_sync(0xFFFFFFFFu, row < 32u ? rl0 : rl1, row & 31u) + (ex & 0xFFFFu);
      uint32_t E = __shfl_sync(0xFFFFFFFFu, row < 32u ? re0 : re1, row & 31u) + (ex >> 16);
      const uint32_t id0 = row_base(row) + 32u * (W & 127u);
      // a partition boundary at one of this word's entries: the victims before it
      for (uint32_t q = 1; (int)q < a.pc.n_parts; ++q) {
        const uint32_t b = (uint32_t)a.pc.base[q] - id0;
        if (a.pc.base[q] < a.n && b < 32u && id0 + b < row_end(row)) {
          const uint32_t m = (1u << b) - 1u;
          const uint32_t l = L + (uint32_t)__popc(bl & m), e = E + (uint32_t)__popc(be & m);
          publish_word(&a.sel->bound[q - 1], tag, l + (e < eq_room ? e : eq_room));
        }
      }
      if (!found) continue;
      uint32_t bits = (E >= eq_room) ? bl : (bl | be);
      const uint32_t p0 = L + (E < eq_room ? E : eq_room);
      // Where the warp has no entry equal to tau that is taken (nearly everywhere), a victim is a bit
      // and a place: half the work of the general loop below.  The warp's ids are neighbours.  Where they
      // are many they leave together through shared memory (a store of 32 lanes' next ids touches a dozen
      // sectors, each of them again for the ids that follow: 3.2 M entries of which 15 % leave, three
      // calls, 55.0 -> 53.7 us); with 10 % and less the detour costs what it saves (18.8 M entries even,
      // 1.0 M in the radix select 17.0 -> 17.6).
      const uint32_t p1 = p0 + (uint32_t)__popc(bits);
      if (!BLOCKS && __all_sync(0xFFFFFFFFu, (be == 0u || E >= eq_room) && p1 <= (uint32_t)a.k)) {
        const uint32_t from = __shfl_sync(0xFFFFFFFFu, p0, 0), n_ids = __shfl_sync(0xFFFFFFFFu, p1, 31) - from;
        if (!SHARED && n_ids > 128u && n_ids <= room) {
          uint32_t* out = ids + (p0 - from);
          while (bits) {
            *out++ = id0 + (uint32_t)__ffs(bits) - 1u;
            bits &= bits - 1u;
          }
          __syncwarp();
          for (uint32_t i = lane; i < n_ids; i += 32u) a.victims[from + i] = ids[i];
          __syncwarp();
        } else {
          uint32_t* out = a.victims + p0;
          while (bits) {
            *out++ = id0 + (uint32_t)__ffs(bits) - 1u;
            bits &= bits - 1u;
          }
        }
        continue;
      }
      while (bits) {
        const uint32_t b = (uint32_t)__ffs(bits) - 1u;
        bits &= bits - 1u;
        uint32_t pos = L + (E < eq_room ? E : eq_room);
        if ((be >> b) & 1u) {
          if (E >= eq_room) pos = 0xFFFFFFFFu;
          ++E;
        } else {
          ++L;
        }
        if (pos < a.k) {
          if (BLOCKS && a.expand) write_block(pos, id0 + b);
          else a.victims[pos] = id0 + b;
        }
      }
    }
    stamp(4);
    if (g == G - 1u && t == 0) {
      // (together: one behind the answer of another is latency at the launch's end)
      const uint32_t last = a.sel->hint_last, trend = a.sel->hint_trend;
      const uint32_t was_off_last = a.sel->hint_off_last, was_off_trend = a.sel->hint_off_trend;
      // every entry has been counted: the selection must hold exactly k ids
      if (!found || got != a.k) atomicOr(a.status, KV_DEV_SELECT_MISMATCH);
      if (a.pc.n_parts > 1 && a.pc.d_counts) {
        unsigned long long prev = 0;
        for (int q = 1; q <= 4; ++q) {
          unsigned long long upto = prev;
          if (q < a.pc.n_parts && a.pc.base[q] < a.n) upto = await_word(&a.sel->bound[q - 1], tag, ok);
          else if (q <= a.pc.n_parts) upto = got;
          a.pc.d_counts[q - 1] = upto - prev;
          if (a.pc.h_counts) a.pc.h_counts[q - 1] = upto - prev;
          prev = upto;
        }
        if (!ok) atomicOr(a.status, KV_DEV_WAIT_EXPIRED);
      } else if (BLOCKS && a.expand && a.pc.h_counts) {   // what a demotion will want to know
        a.pc.h_counts[0] = got * a.expand;
        for (int q = 1; q < 4; ++q) a.pc.h_counts[q] = 0;
      }
      end_turn();   // (every CTA has read the number long ago)
      if constexpr (SHARED) return;   // (nobody comes after it who could use what follows)
      a.sel->tau = tau;
      a.sel->need_eq = need_eq;
      a.sel->n_select += 1;
      // Hint for the next selection over the same keys: this tau, or this tau moved on by as much as it moved
      // since the selection before, whichever has been the better guess lately (scores that grow epoch after
      // epoch, and LRU's, follow a trend; others scatter about a level, and a trend doubles their error).
      // The bracket reaches two and a half times a slowly decaying maximum of that guess's errors to either
      // side: fewer keys in the bracket are fewer notes, a miss costs two or three passes over the keys.
      // 30 pools, 30 passes each: 10 misses and a mean reach of 920 K keys, where the trend alone, five times
      // a faster decaying maximum and full width after a miss gave 25 misses and 1,181 K.
      auto worn = [tau](uint32_t off, uint32_t guess) {
        const uint32_t now = tau > guess ? tau - guess : guess - tau;
        off -= off / 10u;
        return now > off ? now : off;
      };
      const uint32_t off_last = hint ? worn(was_off_last, last) : 1u << 18;
      const uint32_t off_trend = hint ? worn(was_off_trend, trend) : 1u << 18;
      long long guess = hint ? 2ll * (long long)tau - (long long)last : (long long)tau;
      if (guess < 0) guess = 0;
      if (guess > 0xFFFFFFFEll) guess = 0xFFFFFFFEll;
      const uint32_t off = off_last <= off_trend ? off_last : off_trend;
      const uint32_t new_half = off < kHalfMax / 5u * 2u ? off * 2u + off / 2u : kHalfMax;
      a.sel->hint_off_last = off_last;
      a.sel->hint_off_trend = off_trend;
      a.sel->hint_trend = (uint32_t)guess;
      a.sel->hint_half = new_half < kHalfMin ? kHalfMin : new_half;
      a.sel->hint_last = tau;
      a.sel->hint_tau = off_last <= off_trend ? tau : (uint32_t)guess;
      a.sel->hint_n = a.n;
      a.sel->hint_valid = (found && got == a.k) ? 1u : 0u;
    }
  }
  stamp(7);
  return;

fail:
  if (t == 0) {
    atomicOr(a.status, KV_DEV_WAIT_EXPIRED);
    end_turn();   // (the next launch finds the other set, which every CTA of this one has cleared)
  }
}

// What one device can do with the persistent kernels, probed once per device
// (with that device current) under a lock.
namespace {
struct PersistDevice {
  int state = 0;   // 0 = not probed, 1 = usable, -1 = not usable
  int n_sm = 0;
  size_t smem_max = 0;   // dynamic shared memory the kernels were opted in for
};
constexpr int kPMaxDevices = 64;
std::mutex g_persist_mutex;
PersistDevice g_persist[kPMaxDevices];

// Dynamic shared memory of a launch: two bitmaps, where the warps' notes of each row begin, the
// notes, and the entry pass's stages.
inline size_t persist_smem(uint32_t n_rows, uint32_t note_cap, uint32_t stages_words) {
  return 4u * ((size_t)n_rows * 256u + (n_rows + 1u) * 32u + (size_t)note_cap * kPWarps + (size_t)stages_words);
}
}  // namespace

// Launches the persistent selection (fused with the entry pass when fs is given)
// if the device can hold one CTA per SM of it co-resident and the rows fit the
// bitmaps; *used = false (and nothing launched) otherwise.
cudaError_t launch_select_persistent(const EntryState& st, uint64_t k, uint32_t* d_victims,
                                     const Workspace& ws, cudaStream_t s, bool* used, const FusedScore* fs,
                                     const PartCounts* pc, const BlockGeom* bg) {
  *used = false;
  const uint64_t n = bg ? bg->block_base[bg->n_parts] : st.n;   // what is selected from
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return cudaGetLastError();
  if (dev < 0 || dev >= kPMaxDevices) return cudaSuccess;
  PersistDevice pd;
  {
    std::lock_guard<std::mutex> lock(g_persist_mutex);
    PersistDevice& d = g_persist[dev];
    if (d.state == 0) {
      int coop = 0, blocks = 1, optin = 0;
      cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
      cudaDeviceGetAttribute(&d.n_sm, cudaDevAttrMultiProcessorCount, dev);
      cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
      void* fns[5] = {(void*)select_persistent_kernel<false, false, false, false>, (void*)select_persistent_kernel<true, false, false, false>,
                      (void*)select_persistent_kernel<true, true, false, false>, (void*)select_persistent_kernel<false, false, true, false>,
                      (void*)select_persistent_kernel<false, false, false, true>};
      cudaError_t e = cudaSuccess;
      size_t fixed = 0;
      for (void* fn : fns) {
        cudaFuncAttributes fa{};
        if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, fn);
        if (fa.sharedSizeBytes > fixed) fixed = fa.sharedSizeBytes;
      }
      // the most a launch may ask for: everything a block can opt in to beyond the kernels' static share
      const size_t want = (size_t)optin > fixed ? ((size_t)optin - fixed) / 1024 * 1024 : 0;
      if (want < persist_smem(kPMaxRows, kNoteCapMin, kStages * stage_words(true, false))) e = cudaErrorInvalidValue;
      d.smem_max = want;
      for (void* fn : fns) {
        int b = 0;
        if (e == cudaSuccess) e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)want);
        if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, fn, (int)kPThreads, want);
        if (b < blocks) blocks = b;
      }
      d.state = (e == cudaSuccess && coop && blocks >= 1 && d.n_sm > 0) ? 1 : -1;
      (void)cudaGetLastError();
    }
    pd = d;
  }
  if (pd.state != 1) return cudaSuccess;
  // One CTA per SM, but none with less than 1,024 entries (more CTAs only make the exchanges wider);
  // up to kPAlone entries one CTA, which exchanges nothing and needs no cooperative launch.
  uint64_t ctas = n <= kPAlone ? 1 : (n + kPChunk / 4 - 1) / (kPChunk / 4);
  if (ctas > (uint64_t)pd.n_sm) ctas = (uint64_t)pd.n_sm;
  if (ctas > kPThreads) ctas = kPThreads;
  const uint32_t G = ctas ? (uint32_t)ctas : 1u;
  PArgs a;
  const uint64_t row = (uint64_t)G * kPChunk;
  a.n_full = (uint32_t)(n / row);
  const uint64_t rest = n - a.n_full * row;
  a.last_len = (uint32_t)((rest + G * 128ull - 1) / (G * 128ull) * 128ull);
  a.n_rows = a.n_full + (rest ? 1u : 0u);
  if (a.n_rows > kPMaxRows) return cudaSuccess;   // more than the bitmaps hold: the multi-launch selection runs
  if ((uint64_t)a.n_rows * G > ws.table_words) return cudaSuccess;
  a.score = st.score;
  a.state = st.state;
  a.n = n;
  a.k = k;
  a.victims = d_victims;
  a.sel = ws.sel;
  a.turns = ws.turns;
  a.table = ws.table;
  a.list = ws.list;
  a.words = ws.shared_words;
  a.status = ws.status;
  const bool lru = fs && fs->opt.policy == 2;
  // (the LRU policy's stages leave no room for the packed counts on pools of more than 41 rows)
  const bool packed = fs && fs->n_events < kPackedMaxEvents &&
                      persist_smem(a.n_rows, kNoteCapMin, kStages * stage_words(true, lru)) <= pd.smem_max;
  a.stage_words = fs ? stage_words(packed, lru) : 0u;
  const uint32_t stages_words = kStages * a.stage_words;
  // Notes: the bracket typically holds 4-15 % of a warp's keys, in some traces several times
  // that.  A quarter of them stays in shared memory (what does not fit goes to the global scratch);
  // the form without the entry pass takes room for every key, which the plain path fills.
  uint32_t cap = fs ? a.n_rows * 32u : a.n_rows * 128u;
  if (cap < kNoteCapMin) cap = kNoteCapMin;
  while (cap > kNoteCapMin && persist_smem(a.n_rows, cap, stages_words) > pd.smem_max) cap -= 4;
  const size_t smem = persist_smem(a.n_rows, cap, stages_words);
  if (smem > pd.smem_max) return cudaSuccess;
  a.note_cap = cap;
  a.scratch_words = cap * kPWarps + stages_words;
  a.pc = pc ? *pc : PartCounts{};
  // (scratch of promotions and admissions: idle while a selection runs.  It has N + 4,096 words;
  // n_rows * 4,096 * G is at most N + 4,096 * G, and every warp keeps at least 128 notes itself)
  a.spill = ws.free_list;
  a.spill_stride = a.n_rows * 128u > cap ? a.n_rows * 128u - cap : 0u;
  a.bg = bg ? *bg : BlockGeom{};
  a.expand = bg && bg->n_parts == 1 ? bg->heads[0] : 0u;
  a.st = st;
  if (!packed) a.st.packed = nullptr;
  a.pd = Predictor{};
  a.hw = HeadWeights{};
  const Workspace lws = packed ? ws.for_packed() : ws;
  a.epoch = 0;
  a.ev_entry = nullptr;
  a.n_events = 0;
  if (fs) {
    a.pd = Predictor{fs->hits,       fs->misses,    fs->P,          fs->alpha0, fs->beta0, ws.delta, nullptr,
                     fs->opt.policy, fs->opt.kappa, fs->opt.window, ws.blend};
    a.hw = fs->hw;
    a.epoch = fs->epoch;
    const cudaError_t e = launch_event_reduce(fs->ev_entry, fs->ev_hit, fs->n_events, a.st, lws, s);
    if (e != cudaSuccess) return e;
    a.ev_entry = fs->ev_entry;
    a.n_events = fs->n_events;
  }
  void* args[] = {&a};
  const bool plain = fs && fs->opt.policy == 0 && fs->hw.on == 0;
  void* fn = bg ? (void*)select_persistent_kernel<false, false, true, false>
             : ws.shared_words ? (void*)select_persistent_kernel<false, false, false, true>
             : !fs ? (void*)select_persistent_kernel<false, false, false, false>
                   : plain ? (void*)select_persistent_kernel<true, true, false, false>
                           : (void*)select_persistent_kernel<true, false, false, false>;
  cudaError_t e = launch_scoring_kernel(fn, dim3(G), dim3(kPThreads), args, smem, s, G > 1, lws);
  if (e != cudaSuccess) {
    if (packed) (void)launch_event_recount(fs->ev_entry, fs->n_events, a.st, ws, s);
    return e;
  }
  count_launches(1);
  *used = true;
  return cudaSuccess;
}

}  // namespace kvt
