// Internal declarations shared by the kvtier translation units.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>

#include "kvtier.h"

namespace kvt {

constexpr int kThreads = 256;
constexpr uint32_t kRadixBits1 = 11, kRadixBits2 = 11, kRadixBits3 = 10;
constexpr uint32_t kHistBins = 2048;  // bins of the widest digit
constexpr uint32_t kTileEntries = 2048;  // entries per compaction tile (256 threads x 8)
// Bit 7 of an entry's pair byte is set while the entry is FREE, so that the event
// reduction learns both the pair and the state from one gathered byte.
constexpr uint32_t kPairFree = 0x80u;

// Kernels launched by this library in this process (all pools).
extern std::atomic<uint64_t> g_kernel_launches;
inline void count_launches(uint64_t n) { g_kernel_launches.fetch_add(n, std::memory_order_relaxed); }

// Streaming multiprocessors of the current device (148 on a B200); grids are sized in
// multiples of it.  Asked of the runtime at every launch: the answer belongs to the
// device that is current, not to the process.
inline int sm_count() {
  int dev = 0, n = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0) {
    (void)cudaGetLastError();
    return 1;
  }
  return n;
}

// Geometry of one partition, as the kernels need it.
struct PartGeom {
  uint8_t* slab;         // device
  uint64_t base;         // first global id
  uint64_t n;            // entries
  uint32_t heads;        // KV heads per block (1 for MLA)
  uint32_t n_chunks;     // 2 (K, V) or 1 (MLA)
  uint32_t chunk_bytes;  // bytes of one contiguous chunk in the slab
  uint32_t entry_bytes;  // n_chunks * chunk_bytes
  uint32_t ring_slots;
  // device mirror of per-ring-slot metadata
  uint32_t* r_tag;
  uint32_t* r_last_epoch;
  float* r_ema;
  float* r_decay;
  uint8_t* r_pair;
  uint32_t* r_depoch;    // epoch in which the slot's block was demoted
  uint32_t epoch_now;    // epoch of the pool's last scoring pass (set by the host before a launch)
  uint32_t lazy_decay;   // promotion applies the EMA steps missed on the host
};

// EMA of a block that sat out `missed` scoring passes untouched: every pass is
// ema <- decay*ema + (1 - decay)*0 = decay*ema, one rounded multiply.  Stops early
// at a fixed point (0, decay 1, or a denormal that no longer shrinks), where
// further steps change nothing.
__device__ __forceinline__ float ema_catch_up(float ema, float decay, uint32_t missed) {
  for (uint32_t s = 0; s < missed; ++s) {
    const float nx = __fmul_rn(decay, ema);
    if (nx == ema) break;
    ema = nx;
  }
  return ema;
}

// Per-entry state arrays.
//
struct EntryState {
  float* ema;
  float* decay;
  uint32_t* touch;
  uint32_t* last_epoch;
  uint8_t* pair;
  uint8_t* state;
  uint32_t* tag;
  float* score;
  uint64_t n;
  // Touches that only the fused scoring pass of the same call reads, a word for four entries, zero
  // between calls (nullptr: touches are counted in `touch`).  See reduce_events in kv_score_device.cuh.
  unsigned long long* packed = nullptr;
};

// Small block of device scalars used by selection and compaction.
struct SelectScalars {
  uint32_t prefix;        // key bits fixed so far
  uint32_t tau;           // key of the k-th smallest entry
  unsigned long long k_rem;    // rank still to resolve inside the current bucket
  unsigned long long need_eq;  // how many entries with key == tau are taken
  uint32_t serial;             // number of the last persistent selection
  unsigned int update_ticket;  // blocks of the entry pass that have finished (the last one commits)
  unsigned int hint_valid;     // the persistent selection left a usable hint
  uint32_t hint_tau;           // where the next persistent selection centres its bracket ...
  uint32_t hint_last;          // (tau of the last one)
  unsigned long long hint_n;   // ... and the number of keys it ran over
  unsigned long long phase_ns[16]; // %globaltimer at the phase boundaries of the last persistent selection (CTA 0)
  // how the persistent selections went so far (kv_selection_stats)
  unsigned int n_select;       // selections run
  unsigned int n_hint_hit;     // ... whose hint's bracket held rank k
  unsigned int n_hint_miss;    // ... whose hint's bracket did not
  unsigned int n_reread;       // reserved (kv_selection_stats reports it), 0
  // persistent selection on a pool of several partitions: launch number | victims before
  // partition boundary q + 1, written by the CTA that holds it
  unsigned long long bound[3];
  // how far the next selection's bracket reaches to either side of the hint, in keys; slowly decaying
  // maxima of how far tau landed from the last one and from where the trend of the last two put it
  uint32_t hint_half;
  uint32_t hint_off_last, hint_off_trend;
  uint32_t hint_trend;         // where the trend puts the next tau
  uint32_t touch_wide;         // so many epochs to come of the fused pass count their touches in `touch` ...
  uint32_t touch_hot;          // ... and one of them has met an entry with more than a packed count holds
};

// What the CTAs of one persistent selection share while it runs.  A pool has two of these, used in
// turn: a launch finds its own zeroed and clears the next launch's.
struct SelectTurn {
  unsigned int bar;             // arrivals at the grid barrier
  unsigned int listed;          // keys in the list
  unsigned long long below;     // keys below the bracket (and kOverflowed for CTAs that met an overflowed count)
  uint32_t hist[4][kHistBins];  // the bracket's bins, then its last bin's keys or the radix select's digits
};

// Sliding window of per-epoch (pair, hit) counts for the confidence-weighted
// blend of the reuse estimate, and the estimates themselves.
constexpr uint32_t kMaxWindow = 64;
struct BlendState {
  unsigned long long wsum[32];              // sums over the window, index 2*pair + hit
  unsigned long long win[kMaxWindow * 32];  // ring of per-epoch counts
  float estimate[16];                       // reuse estimate used by the Bayesian score
  uint32_t head;                            // ring slot the next epoch overwrites
  uint32_t pad;
};

// Host-chosen options of the scoring pass.
struct ScoreOptions {
  int policy = 0;       // 0 Bayesian, 1 EMA only, 2 LRU
  float kappa = 0.0f;   // confidence saturation constant
  uint32_t window = 0;  // epochs in the sliding window; 0 = no blending
};

// Paged blocks (layer, block) of all partitions in one index space, for
// block-granular selection.
struct BlockGeom {
  uint64_t block_base[5];   // first global block index of each partition; [n_parts] = total
  uint64_t entry_base[4];   // first global entry id of each partition
  uint32_t heads[4];        // KV-head entries per block
  float weight[4];          // query heads per KV-head entry
  int n_parts;
};

__device__ __forceinline__ int block_partition(const BlockGeom& bg, uint64_t gb) {
  int q = 0;
  while (q + 1 < bg.n_parts && gb >= bg.block_base[q + 1]) ++q;
  return q;
}

// Division of numbers below 2^31 by d, as a multiplication: with 2^s the power of two from d on and
// mul = ceil(2^(31+s) / d), the product exceeds x * 2^(31+s) / d by less than x * 2^s / d < 2^(31+s) / d,
// too little to reach the next quotient (Granlund and Montgomery, "Division by invariant integers using
// multiplication", 1994).
struct Divisor {
  uint32_t mul = 0, shift = 0;   // mul 0: d is 1
  Divisor() = default;
  explicit Divisor(uint32_t d) {
    if (d < 2u) return;
    uint32_t s = 0;
    while ((1ull << s) < d) ++s;
    mul = (uint32_t)(((1ull << (31u + s)) + d - 1u) / d);
    shift = s - 1u;
  }
  __device__ __forceinline__ uint32_t operator()(uint32_t x) const { return mul ? __umulhi(x, mul) >> shift : x; }
};

// Head-granular importance (head-granular eviction section): per partition a
// [layer][query head] importance matrix, [layer][KV head] multipliers and the
// resulting [layer][KV head] score weights, each partition's block at its offset.
struct HeadWeights {
  float* imp;              // importance matrices, partition q at imp_off[q]
  float* mult;             // multipliers, partition q at w_off[q]
  float* w;                // weights, partition q at w_off[q]
  uint64_t base[5];        // first global entry id of each partition; [n_parts] = N
  uint32_t per_layer[4];   // entries per layer: blocks per layer x KV heads
  uint32_t heads[4];       // KV heads (1 for MLA)
  Divisor by_layer[4], by_heads[4];   // the same, to divide by
  uint32_t q_heads[4];     // tracked query heads per layer (1 for MLA)
  uint32_t layers[4];
  uint32_t imp_off[4], w_off[4];
  uint32_t on;             // bit q: scores of partition q are weighted
  int n_parts;
};

// Per-layer prefetch windows (RoPE-aware prefetching section): per partition the EMA of
// the observed attention span in tokens and the window in blocks derived from it.
constexpr uint32_t kPrefetchChunks = 1024;   // most blocks of one prefetch-list launch
struct PrefetchState {
  float* span;             // [layers] per partition, partition q at off[q]
  uint32_t* win;           // same layout
  unsigned long long* words;   // [kPrefetchChunks] scratch of the list kernel: counts tagged with the launch's number
  uint32_t* serial;            // number of the last list launch
  uint32_t off[4], layers[4], heads[4];
  uint32_t block_tokens[4];
  uint32_t w_max[4];       // cap on the window, blocks
};

struct Workspace {
  BlendState* blend;
  float* block_score;       // [blocks] aggregate score per paged block
  uint8_t* block_state;     // [blocks] RESIDENT iff every head of the block is
  uint32_t* block_victims;  // [blocks] selected global block indices
  unsigned long long* delta;   // [32] per-epoch (pair, hit) counts: index pair*2+hit
  uint32_t* hist;              // [3][kHistBins], zero between selections
  SelectScalars* sel;
  uint32_t* status;            // device status word
  uint2* tile_counts;          // [n_tiles] (less, equal) or (free, 0)
  uint2* tile_offsets;         // [n_tiles] exclusive prefix of tile_counts
  uint32_t* free_list;         // [max(N, ..)] ascending ids of FREE entries
  uint32_t* slot_list[8];      // [max_promote] promote lists (ring slots), used in turn
  unsigned long long* part_counts;  // [4] victims per partition
  uint32_t n_tiles;
  // persistent selection
  SelectTurn* turns;                // [2], used in turn
  uint32_t* table;                  // [table_words] counts per chunk
  unsigned long long* list = nullptr;   // shared scratch: [kListMax] the keys of the last bin, and where they are
  uint64_t table_words;
  // Scratch that calls share which know nothing of each other (nullptr: it is the pool's own): the
  // number of the last call, then a word for each CTA that clears (up to kSharedCtas).  Each call
  // clears its set of counters itself, whatever the one before has left.
  unsigned long long* shared_words = nullptr;
  // One of the state arrays kept in the persisting part of the L2 (kv_set_l2_residency):
  // the scoring kernels are launched with this access-policy window.  bytes == 0: none.
  const void* l2_base = nullptr;
  size_t l2_bytes = 0;
  float l2_ratio = 0.0f;
  // ... or this one, for the launches that count touches in EntryState::packed
  const void* l2_packed = nullptr;
  size_t l2_packed_bytes = 0;
  Workspace for_packed() const {
    Workspace w = *this;
    if (l2_packed) { w.l2_base = l2_packed; w.l2_bytes = l2_packed_bytes; w.l2_ratio = 1.0f; }
    return w;
  }
};

// Launches fn (kernel taking the arguments in args) with the workspace's L2 window, if it has
// one, as a launch attribute; cooperative launches carry that attribute too.
inline cudaError_t launch_scoring_kernel(const void* fn, dim3 grid, dim3 block, void** args, size_t smem,
                                         cudaStream_t s, bool cooperative, const Workspace& ws,
                                         bool overlap = true) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  unsigned n = 0;
  if (cooperative) {
    attr[n].id = cudaLaunchAttributeCooperative;
    attr[n].val.cooperative = 1;
    ++n;
  } else if (overlap) {   // (see wait_for_kernel_ahead)
    attr[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[n].val.programmaticStreamSerializationAllowed = 1;
    ++n;
  }
  if (ws.l2_bytes) {
    attr[n].id = cudaLaunchAttributeAccessPolicyWindow;
    attr[n].val.accessPolicyWindow.base_ptr = const_cast<void*>(ws.l2_base);
    attr[n].val.accessPolicyWindow.num_bytes = ws.l2_bytes;
    attr[n].val.accessPolicyWindow.hitRatio = ws.l2_ratio;
    attr[n].val.accessPolicyWindow.hitProp = cudaAccessPropertyPersisting;
    attr[n].val.accessPolicyWindow.missProp = cudaAccessPropertyNormal;
    ++n;
  }
  cfg.attrs = attr;
  cfg.numAttrs = n;
  return cudaLaunchKernelExC(&cfg, fn, args);
}

// A kernel launched with launch_overlapped (or launch_scoring_kernel, if not cooperative) may be
// set up while the kernel ahead of it in the stream is still finishing (programmatic dependent
// launch).  It calls this before it touches memory, which waits until everything ahead of it is
// complete and visible, and then lets the kernel behind it be set up in turn.  Such a kernel reads
// nothing through the read-only (non-coherent) path: the kernel ahead may have written it while this
// one was already resident.  About 1 us per kernel of a chain.
__device__ __forceinline__ void wait_for_kernel_ahead() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

template <typename... Params, typename... Args>
inline cudaError_t launch_overlapped_smem(void (*kernel)(Params...), unsigned grid, unsigned block, size_t smem,
                                          cudaStream_t s, Args... args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  count_launches(1);
  return cudaLaunchKernelEx(&cfg, kernel, Params(args)...);
}

template <typename... Params, typename... Args>
inline cudaError_t launch_overlapped(void (*kernel)(Params...), unsigned grid, unsigned block, cudaStream_t s,
                                     Args... args) {
  return launch_overlapped_smem(kernel, grid, block, 0, s, args...);
}

// ---- kv_score.cu ----
// With st.packed the touches go there, for the fused scoring pass.
cudaError_t launch_event_reduce(const uint32_t* ev_entry, const uint8_t* ev_hit, uint64_t n_events,
                                const EntryState& st, const Workspace& ws, cudaStream_t s);
// Behind a launch_event_reduce into st.packed whose scoring pass could not be launched: the touches go where
// kv_epoch_events leaves them, beside the epoch counters, which hold the trace already.
cudaError_t launch_event_recount(const uint32_t* ev_entry, uint64_t n_events, const EntryState& st, const Workspace& ws,
                                 cudaStream_t s);
// posterior (from hits/misses plus the epoch counters in ws.delta) + EMA + score in one launch;
// folds ws.delta into hits/misses, clears it and writes P
cudaError_t launch_entry_update(const EntryState& st, uint64_t* hits, uint64_t* misses, float* P,
                                float alpha0, float beta0, const Workspace& ws, uint32_t epoch,
                                const ScoreOptions& opt, const HeadWeights& hw, cudaStream_t s);
// kv_heads.cu: mode 0 = EMA step of partition q's importance matrix with observations
// src [L][QH]; mode 1 = multipliers of q from src [L][H] (nullptr: all 1).  Both then
// recompute q's weights.  Values that are negative or not finite are skipped and flagged.
cudaError_t launch_head_update(const HeadWeights& hw, int q, int mode, const float* src, float decay,
                               const Workspace& ws, cudaStream_t s);
cudaError_t launch_head_init(const HeadWeights& hw, uint32_t n_imp, uint32_t n_w, cudaStream_t s);
// kv_prefetch.cu: mode 0 = EMA step of partition q's per-layer span with observations x [L]
// (any negative or non-finite value: nothing changes, flagged); mode 1 = every span = tokens.
// Both recompute the windows.
cudaError_t launch_prefetch_window(const PrefetchState& pf, int q, int mode, const float* x, float decay,
                                   float tokens, const Workspace& ws, cudaStream_t s);
// ring slots of the host-tier blocks of table [n_pos][L][H] inside the windows around
// position-block pos0, ordered by (distance, layer, head); *count = how many qualified
cudaError_t launch_prefetch_list(const PrefetchState& pf, int q, const uint32_t* table, uint64_t n_pos,
                                 uint64_t pos0, int dir, const uint32_t* loc, uint64_t n_tags,
                                 unsigned long long* out, uint64_t max_out, unsigned long long* count,
                                 const Workspace& ws, cudaStream_t s);
// empties the sliding window of the blend (the estimates stay as they are)
cudaError_t launch_blend_reset(const Workspace& ws, cudaStream_t s);

// ---- kv_select.cu ----
// Where the victims of a selection fall: partition bases (global entry ids; [n_parts] = N),
// and where the per-partition victim counts go (device, and host memory the device can
// write, or nullptr).
struct PartCounts {
  unsigned long long base[5] = {0, 0, 0, 0, 0};
  int n_parts = 1;
  unsigned long long* d_counts = nullptr;   // [4]
  unsigned long long* h_counts = nullptr;   // [4] device-visible address of pinned host memory
};
// Words of the persistent selection's table of counts for n entries: one per chunk of 4,096 entries
// of every CTA, the last row's pieces counted as chunks (at most 1,024 CTAs).
inline uint64_t select_table_words(uint64_t n) { return n / 4096 + 1024; }
// The scratch of selections for callers that have none to give (kv_select.cu).
constexpr uint64_t kStaticMaxEntries = 1ull << 22;  // 4,194,304 entries
constexpr uint64_t kStaticMaxTiles = kStaticMaxEntries / kTileEntries + 2;
constexpr uint32_t kSharedCtas = 16;
// Keys of one bin that the persistent selection on shared scratch puts on a list which every CTA reads,
// instead of another exchange: at most these.
constexpr uint32_t kListMax = 1024;
struct StaticScratch {
  uint32_t hist[3 * kHistBins];
  SelectTurn turn;
  SelectScalars sel;
  unsigned long long words[1 + kSharedCtas];
  uint32_t status[4];
  uint2 tile_counts[kStaticMaxTiles];
  uint2 tile_offsets[kStaticMaxTiles];
  uint32_t table[kStaticMaxEntries / 4096 + 1024];
  unsigned long long list[kListMax];
};
// n <= kStaticMaxEntries; status may be nullptr
cudaError_t launch_select_static(const float* score, const uint8_t* state, uint64_t n, uint64_t k, uint32_t* d_victims,
                                 StaticScratch* scratch, uint32_t* status, cudaStream_t s, int variant = 1);
// variant 1 = one persistent cooperative launch (falls back to 0 where the device cannot run
// it or the slices are too long), 0 = one launch per phase of the radix select
cudaError_t launch_select(const EntryState& st, uint64_t k, uint32_t* d_victims, const Workspace& ws,
                          cudaStream_t s, int variant = 1, const PartCounts* pc = nullptr);
// kv_select_persist.cu: the same selection as one cooperative launch; *used tells
// whether it was launched (false: the device cannot co-schedule it, nothing was enqueued)
// With fs a launch of the event reduction goes ahead (touches into st.packed), and the launch also
// does the entry pass first (posterior, EMA, score).
struct FusedScore {
  uint64_t* hits;
  uint64_t* misses;
  float* P;
  float alpha0, beta0;
  uint32_t epoch;
  ScoreOptions opt;
  HeadWeights hw;
  const uint32_t* ev_entry;      // the epoch's trace, whose reduction is launched ahead
  const uint8_t* ev_hit;
  uint64_t n_events;
};
cudaError_t launch_select_persistent(const EntryState& st, uint64_t k, uint32_t* d_victims,
                                     const Workspace& ws, cudaStream_t s, bool* used,
                                     const FusedScore* fs = nullptr, const PartCounts* pc = nullptr,
                                     const BlockGeom* bg = nullptr);   // bg: from paged blocks
// kv_blocks.cu: k_blocks lowest blocks by weighted aggregate score; writes all their entries
// (ascending) to d_victims, the per-partition block counts to ws.part_counts and the
// per-partition ENTRY counts to h_entry_counts (host memory the device can write; may be nullptr)
cudaError_t launch_select_blocks(const EntryState& st, const BlockGeom& bg, uint64_t k_blocks,
                                 uint32_t* d_victims, const Workspace& ws, cudaStream_t s,
                                 unsigned long long* h_entry_counts);
// ascending ids of FREE entries in [lo, hi), at most `limit` of them, into ws.free_list + out_offset
cudaError_t launch_free_list(const EntryState& st, uint64_t lo, uint64_t hi, uint64_t limit,
                             const Workspace& ws, cudaStream_t s, uint64_t out_offset = 0);
// victims per partition of an ascending list into pc.d_counts (and pc.h_counts)
cudaError_t launch_partition_counts(const uint32_t* d_victims, uint64_t m, const PartCounts& pc,
                                    cudaStream_t s);

// ---- kv_dedup.cu ----
// SHA-256 of the images of entries ids[0..m) (ids == nullptr: entries 0..m-1), 32 bytes each
cudaError_t launch_hash_entries(const PartGeom* parts, int n_parts, const uint32_t* ids, uint64_t m,
                                uint8_t* digests, uint64_t n_entries, const Workspace& ws, cudaStream_t s);
// first position per digest and reference counts; table_slots is a power of two >= 2*m
cudaError_t launch_dedup(const uint8_t* digests, uint64_t m, uint32_t* canon, uint32_t* refcount,
                         uint32_t* table, uint64_t table_slots, uint32_t* n_unique, uint32_t* status,
                         cudaStream_t s);

// ---- kv_move.cu ----
cudaError_t launch_init(const EntryState& st, uint64_t* hits, uint64_t* misses, float* P, float p0,
                        uint32_t* loc, uint64_t n_tags, const PartGeom* parts, int n_parts,
                        const Workspace& ws, cudaStream_t s);
// ---- kv_move_tma.cu: gather (demotion) and scatter (promotion) on the bulk asynchronous copy engine ----
// pack: victims[0 .. count) of one partition into staging (images back to back); also moves the
// metadata.  The kv_slot_meta records go straight to the pinned mirror (host_meta: the address at
// which the device sees it), or behind the images at meta_offset (~0: none).  free_out: receives
// the victims' ids, i.e. the slots they leave, in order.
// mode: 0 = metadata and payload, 1 = metadata only (staging unused), 2 = payload only
// (the metadata moved earlier; host-mirror records are rebuilt from the ring mirror)
cudaError_t launch_pack_tma(const PartGeom& g, const EntryState& st, uint32_t* loc, const uint32_t* victims,
                            uint64_t count, uint64_t ring_start, uint8_t* staging, uint64_t meta_offset,
                            const Workspace& ws, cudaStream_t s, uint32_t mode = 0, uint32_t* free_out = nullptr,
                            uint8_t* host_meta = nullptr);
// pack of a few entries without staging: images (and records) straight into the pinned ring
// (ring_dev, host_meta: the addresses at which the device sees them)
cudaError_t launch_pack_direct(const PartGeom& g, const EntryState& st, uint32_t* loc, const uint32_t* victims,
                               uint64_t count, uint64_t ring_start, uint8_t* ring_dev, const Workspace& ws,
                               cudaStream_t s, uint32_t* free_out, uint8_t* host_meta);
// Longest promote list that travels in a launch's arguments (2 KB of them).
constexpr uint32_t kInlineSlots = 512;
// unpack: staging images [0, count) into the listed free slots of the partition; the ring slots they
// come from are listed in h_slots (host, count <= kInlineSlots) or, without it, in slots (device)
cudaError_t launch_unpack_tma(const PartGeom& g, const EntryState& st, uint32_t* loc, const uint32_t* slots,
                              const uint64_t* h_slots, const uint32_t* free_ids, uint64_t count,
                              const uint8_t* staging, const Workspace& ws, cudaStream_t s);
// the same scatter with the entries fetched by the kernel itself from the pinned ring (ring_dev:
// the address at which the device sees it): for lists of short runs
cudaError_t launch_gather_promote(const PartGeom& g, const EntryState& st, uint32_t* loc, const uint32_t* slots,
                                  const uint64_t* h_slots, const uint32_t* free_ids, uint64_t count,
                                  const uint8_t* ring_dev, const Workspace& ws, cudaStream_t s);
// admits free_ids[0 .. count) of one partition, which are the pool's free slots number first ...
cudaError_t launch_admit(const PartGeom& g, const EntryState& st, uint32_t* loc, const uint32_t* free_ids,
                         uint64_t first, uint64_t count, uint64_t first_tag, const uint8_t* new_pairs,
                         uint32_t epoch, float decay, int fill_pattern, const Workspace& ws,
                         cudaStream_t s);

}  // namespace kvt
