// What the library's host side (kvtier_host.cu) enqueues, checked for order.  The runtime's calls and
// the kernel launches are stand-ins: streams and events are vector clocks, every operation is noted
// with the ring slots, staging buffers, slab entries, ring metadata and list words it reads and
// writes, and an access that is not ordered behind the last write of the same thing (a write also
// behind the reads since) is an error.  List contents are kept in order, so slots and ids are real.
// usage: enqueued_order <seed> <deferred 0|1> <ring slots> <gather threshold in bytes> [scenario]
// exit status 1 and a line for the first access out of order.
#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <random>
#include <string>
#include <vector>

#include "kvtier.h"
#include "kvtier_internal.cuh"

namespace {

constexpr int kStreams = 4;   // 1: compute, 2: D2H, 3: H2D
constexpr uint64_t kEntry = 65536, kPinned = 1ull << 44, kSlab = 1ull << 45, kStage = 1ull << 46;
using Clock = uint64_t[kStreams];
struct Event { uint64_t at[kStreams] = {}; };
Clock g_clock[kStreams];
std::string g_bad, g_what;

struct Cell { int by = 0; uint64_t at = 0; std::string what; uint64_t read[kStreams] = {}; };
std::map<std::string, std::vector<Cell>> g_cells;

int sid(cudaStream_t s) { return (int)(intptr_t)s; }
int op(cudaStream_t s, const std::string& what) { g_what = what; ++g_clock[sid(s)][sid(s)]; return sid(s); }

void touch(int s, const std::string& kind, uint64_t i, bool write) {
  std::vector<Cell>& v = g_cells[kind];
  if (v.size() <= i) v.resize(i + 1);
  Cell& c = v[i];
  bool ok = c.at <= g_clock[s][c.by];
  for (int r = 0; write && r < kStreams; ++r) ok = ok && c.read[r] <= g_clock[s][r];
  if (!ok && g_bad.empty())
    g_bad = g_what + " on stream " + std::to_string(s) + (write ? " writes " : " reads ") + kind + " " + std::to_string(i) +
            " last written by " + c.what + " on stream " + std::to_string(c.by) + " without being ordered behind all that came before";
  if (write) {
    c.by = s; c.at = g_clock[s][s]; c.what = g_what;
    for (uint64_t& r : c.read) r = 0;
  } else {
    c.read[s] = g_clock[s][s];
  }
}

std::vector<uint8_t> g_state;   // FREE or RESIDENT, per entry, in the order of the calls
uint32_t* g_list = nullptr;     // the list scratch
int part_of(uint64_t slot_address) { return (int)((slot_address - kPinned) >> 40); }
std::string ring_of(const kvt::PartGeom& g) { return "ring " + std::to_string(g.base ? 1 : 0) + " slot"; }
std::string meta_of(const kvt::PartGeom& g) { return "ring metadata " + std::to_string(g.base ? 1 : 0) + " slot"; }
std::string stage_of(uint64_t a) { return "staging " + std::to_string((a - kStage) >> 32); }
bool pinned(const void* p) { return (uint64_t)p >= kPinned && (uint64_t)p < kSlab; }
void list_words(int s, const uint32_t* from, uint64_t n, bool write) {
  for (uint64_t i = 0; i < n; ++i) touch(s, "list word", (uint64_t)(from + i - g_list), write);
}

}  // namespace

// ---- the runtime ----
extern "C" {
// (under names of their own, with the symbols of the runtime: its header declares some of them for the device)
cudaError_t stand_in_cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) __asm__("cudaEventCreateWithFlags");
cudaError_t stand_in_cudaEventCreate(cudaEvent_t* e) __asm__("cudaEventCreate");
cudaError_t stand_in_cudaEventDestroy(cudaEvent_t e) __asm__("cudaEventDestroy");
cudaError_t stand_in_cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) __asm__("cudaEventElapsedTime");
cudaError_t stand_in_cudaEventQuery(cudaEvent_t) __asm__("cudaEventQuery");
cudaError_t stand_in_cudaEventRecord(cudaEvent_t e, cudaStream_t s) __asm__("cudaEventRecord");
cudaError_t stand_in_cudaEventSynchronize(cudaEvent_t) __asm__("cudaEventSynchronize");
cudaError_t stand_in_cudaStreamSynchronize(cudaStream_t) __asm__("cudaStreamSynchronize");
cudaError_t stand_in_cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned) __asm__("cudaStreamWaitEvent");
cudaError_t stand_in_cudaGetDevice(int* d) __asm__("cudaGetDevice");
cudaError_t stand_in_cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) __asm__("cudaDeviceGetAttribute");
cudaError_t stand_in_cudaDeviceSetLimit(cudaLimit, size_t) __asm__("cudaDeviceSetLimit");
cudaError_t stand_in_cudaCtxResetPersistingL2Cache() __asm__("cudaCtxResetPersistingL2Cache");
cudaError_t stand_in_cudaGetLastError() __asm__("cudaGetLastError");
cudaError_t stand_in_cudaHostGetDevicePointer(void** d, void* h, unsigned) __asm__("cudaHostGetDevicePointer");
cudaError_t stand_in_cudaMemsetAsync(void* p, int v, size_t n, cudaStream_t s) __asm__("cudaMemsetAsync");
cudaError_t stand_in_cudaMemcpyAsync(void* d, const void* h, size_t n, cudaMemcpyKind, cudaStream_t s_) __asm__("cudaMemcpyAsync");
void** __cudaRegisterFatBinary(void*) { static void* h; return &h; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
char __cudaInitModule(void**) { return 1; }
cudaError_t stand_in_cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { *e = (cudaEvent_t) new Event; return cudaSuccess; }
cudaError_t stand_in_cudaEventCreate(cudaEvent_t* e) { return stand_in_cudaEventCreateWithFlags(e, 0); }
cudaError_t stand_in_cudaEventDestroy(cudaEvent_t e) { delete (Event*)e; return cudaSuccess; }
cudaError_t stand_in_cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { *ms = 0.f; return cudaSuccess; }
cudaError_t stand_in_cudaEventQuery(cudaEvent_t) { return cudaSuccess; }
cudaError_t stand_in_cudaEventRecord(cudaEvent_t e, cudaStream_t s) { std::memcpy(((Event*)e)->at, g_clock[sid(s)], sizeof(Clock)); return cudaSuccess; }
cudaError_t stand_in_cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t stand_in_cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t stand_in_cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned) {
  for (int r = 0; r < kStreams; ++r) g_clock[sid(s)][r] = std::max(g_clock[sid(s)][r], ((Event*)e)->at[r]);
  return cudaSuccess;
}
cudaError_t stand_in_cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t stand_in_cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { *v = 148; return cudaSuccess; }
cudaError_t stand_in_cudaDeviceSetLimit(cudaLimit, size_t) { return cudaSuccess; }
cudaError_t stand_in_cudaCtxResetPersistingL2Cache() { return cudaSuccess; }
cudaError_t stand_in_cudaGetLastError() { return cudaSuccess; }
cudaError_t stand_in_cudaHostGetDevicePointer(void** d, void* h, unsigned) { *d = h; return cudaSuccess; }
cudaError_t stand_in_cudaMemsetAsync(void* p, int v, size_t n, cudaStream_t s) { op(s, "memset"); std::memset(p, v, n); return cudaSuccess; }
cudaError_t stand_in_cudaMemcpyAsync(void* d, const void* h, size_t n, cudaMemcpyKind, cudaStream_t s_) {
  const int s = op(s_, pinned(d) ? "copy D2H" : "copy H2D");
  if (pinned(d) || pinned(h)) {
    const uint64_t a = pinned(d) ? (uint64_t)d : (uint64_t)h, q = part_of(a), first = (a - kPinned - (q << 40)) / kEntry;
    for (uint64_t i = 0; i < n / kEntry; ++i) touch(s, "ring " + std::to_string(q) + " slot", first + i, pinned(d));
    const uint64_t b = pinned(d) ? (uint64_t)h : (uint64_t)d;
    for (uint64_t i = 0; i < n / kEntry; ++i) touch(s, stage_of(b), ((b & 0xFFFFFFFFull) / kEntry) + i, !pinned(d));
  } else {
    std::memcpy(d, h, n);
  }
  return cudaSuccess;
}
}  // extern "C"

// ---- the kernels ----
namespace kvt {

static cudaError_t pack(const PartGeom& g, const uint32_t* victims, uint64_t count, uint64_t ring_start, uint8_t* staging, cudaStream_t s_,
                        uint32_t mode, uint32_t* free_out, bool direct) {
  if (count == 0) return cudaSuccess;
  const int s = op(s_, direct ? "pack to the ring" : mode == 1 ? "pack (metadata)" : "pack");
  if (free_out) list_words(s, free_out, count, true);
  for (uint64_t j = 0; j < count; ++j) {
    const uint64_t slot = (ring_start + j) % g.ring_slots;
    if (mode != 2) {
      touch(s, meta_of(g), slot, true);
      touch(s, "entry state", victims[j], true);
      g_state[victims[j]] = KV_STATE_FREE;
      if (free_out) free_out[j] = victims[j];
    }
    if (mode != 1) {
      touch(s, "slab entry", victims[j], false);
      if (direct) touch(s, ring_of(g), slot, true);
      else touch(s, stage_of((uint64_t)staging), j, true);
    }
  }
  return cudaSuccess;
}

static cudaError_t fill(const PartGeom& g, const uint32_t* slots, const uint64_t* h_slots, const uint32_t* free_ids, uint64_t count,
                        const uint8_t* staging, cudaStream_t s_) {
  const int s = op(s_, staging ? "unpack" : "gather from the ring");
  list_words(s, free_ids, count, false);
  for (uint64_t j = 0; j < count; ++j) {
    const uint64_t slot = h_slots ? h_slots[j] : slots[j];
    if (staging) touch(s, stage_of((uint64_t)staging), j, false);
    else touch(s, ring_of(g), slot, false);
    touch(s, meta_of(g), slot, true);
    touch(s, "slab entry", free_ids[j], true);
    touch(s, "entry state", free_ids[j], true);
    if (g_state[free_ids[j]] != KV_STATE_FREE && g_bad.empty()) g_bad = "an entry lands in a slot that is not FREE";
    g_state[free_ids[j]] = KV_STATE_RESIDENT;
  }
  return cudaSuccess;
}

static void whole_pool(int s, const EntryState& st, bool write) {
  for (uint64_t i = 0; i < st.n; ++i) touch(s, "entry state", i, write);
}

cudaError_t launch_pack_tma(const PartGeom& g, const EntryState&, uint32_t*, const uint32_t* victims, uint64_t count, uint64_t ring_start,
                            uint8_t* staging, uint64_t, const Workspace&, cudaStream_t s, uint32_t mode, uint32_t* free_out, uint8_t*) {
  return pack(g, victims, count, ring_start, staging, s, mode, free_out, false);
}
cudaError_t launch_pack_direct(const PartGeom& g, const EntryState&, uint32_t*, const uint32_t* victims, uint64_t count, uint64_t ring_start,
                               uint8_t*, const Workspace&, cudaStream_t s, uint32_t* free_out, uint8_t*) {
  return pack(g, victims, count, ring_start, nullptr, s, 0, free_out, true);
}
cudaError_t launch_unpack_tma(const PartGeom& g, const EntryState&, uint32_t*, const uint32_t* slots, const uint64_t* h_slots,
                              const uint32_t* free_ids, uint64_t count, const uint8_t* staging, const Workspace&, cudaStream_t s) {
  return fill(g, slots, h_slots, free_ids, count, staging, s);
}
cudaError_t launch_gather_promote(const PartGeom& g, const EntryState&, uint32_t*, const uint32_t* slots, const uint64_t* h_slots,
                                  const uint32_t* free_ids, uint64_t count, const uint8_t*, const Workspace&, cudaStream_t s) {
  return fill(g, slots, h_slots, free_ids, count, nullptr, s);
}
cudaError_t launch_free_list(const EntryState&, uint64_t lo, uint64_t hi, uint64_t limit, const Workspace& ws, cudaStream_t s_, uint64_t at) {
  const int s = op(s_, "free list");
  uint64_t n = 0;
  for (uint64_t i = lo; i < hi; ++i) touch(s, "entry state", i, false);
  for (uint64_t i = lo; i < hi && n < limit; ++i)
    if (g_state[i] == KV_STATE_FREE) ws.free_list[at + n++] = (uint32_t)i;
  list_words(s, ws.free_list + at, n, true);
  return cudaSuccess;
}
cudaError_t launch_admit(const PartGeom&, const EntryState&, uint32_t*, const uint32_t* free_ids, uint64_t, uint64_t count, uint64_t,
                         const uint8_t*, uint32_t, float, int, const Workspace&, cudaStream_t s_) {
  const int s = op(s_, "admit");
  list_words(s, free_ids, count, false);
  for (uint64_t j = 0; j < count; ++j) {
    touch(s, "slab entry", free_ids[j], true);
    touch(s, "entry state", free_ids[j], true);
    if (g_state[free_ids[j]] != KV_STATE_FREE && g_bad.empty()) g_bad = "a block is admitted to a slot that is not FREE";
    g_state[free_ids[j]] = KV_STATE_RESIDENT;
  }
  return cudaSuccess;
}
cudaError_t launch_select(const EntryState& st, uint64_t, uint32_t*, const Workspace& ws, cudaStream_t s_, int, const PartCounts*) {
  const int s = op(s_, "select");   // (its notes overflow into the list scratch)
  whole_pool(s, st, false);
  list_words(s, ws.free_list, st.n, true);
  for (uint64_t i = 0; i < st.n; ++i) ws.free_list[i] = 0xDEADBEEFu;
  return cudaSuccess;
}
cudaError_t launch_select_persistent(const EntryState& st, uint64_t k, uint32_t* v, const Workspace& ws, cudaStream_t s, bool* used,
                                     const FusedScore* fs, const PartCounts* pc, const BlockGeom*) {
  *used = true;
  if (fs) {
    whole_pool(op(s, "events"), st, true);
    whole_pool(op(s, "entry pass"), st, true);
  }
  return launch_select(st, k, v, ws, s, 1, pc);
}
cudaError_t launch_select_blocks(const EntryState& st, const BlockGeom&, uint64_t k, uint32_t* v, const Workspace& ws, cudaStream_t s, unsigned long long*) {
  return launch_select(st, k, v, ws, s, 1, nullptr);
}
cudaError_t launch_hash_entries(const PartGeom* parts, int n_parts, const uint32_t*, uint64_t, uint8_t*, uint64_t n, const Workspace& ws, cudaStream_t s_) {
  const int s = op(s_, "hash");
  (void)parts; (void)n_parts;
  for (uint64_t i = 0; i < n; ++i) touch(s, "slab entry", i, false);
  list_words(s, ws.free_list, n, true);
  for (uint64_t i = 0; i < n; ++i) ws.free_list[i] = 0xDEADBEEFu;
  return cudaSuccess;
}
cudaError_t launch_entry_update(const EntryState& st, uint64_t*, uint64_t*, float*, float, float, const Workspace&, uint32_t, const ScoreOptions&,
                                const HeadWeights&, cudaStream_t s) {
  whole_pool(op(s, "entry pass"), st, true);
  return cudaSuccess;
}
cudaError_t launch_event_reduce(const uint32_t*, const uint8_t*, uint64_t, const EntryState& st, const Workspace&, cudaStream_t s) {
  whole_pool(op(s, "events"), st, true);
  return cudaSuccess;
}
cudaError_t launch_partition_counts(const uint32_t* v, uint64_t m, const PartCounts& pc, cudaStream_t s) {
  op(s, "counts");
  for (int q = 0; q < 4; ++q) pc.d_counts[q] = 0;
  for (uint64_t j = 0; j < m; ++j)
    for (int q = 0; q < pc.n_parts; ++q) pc.d_counts[q] += v[j] >= pc.base[q] && v[j] < pc.base[q + 1];
  return cudaSuccess;
}
cudaError_t launch_init(const EntryState&, uint64_t*, uint64_t*, float*, float, uint32_t*, uint64_t, const PartGeom*, int, const Workspace& ws, cudaStream_t) {
  g_list = ws.free_list;
  return cudaSuccess;
}
cudaError_t launch_dedup(const uint8_t*, uint64_t, uint32_t*, uint32_t*, uint32_t*, uint64_t, uint32_t*, uint32_t*, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_head_init(const HeadWeights&, uint32_t, uint32_t, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_head_update(const HeadWeights&, int, int, const float*, float, const Workspace&, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_blend_reset(const Workspace&, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_prefetch_list(const PrefetchState&, int, const uint32_t*, uint64_t, uint64_t, int, const uint32_t*, uint64_t, unsigned long long*,
                                 uint64_t, unsigned long long*, const Workspace&, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_prefetch_window(const PrefetchState&, int, int, const float*, float, float, const Workspace&, cudaStream_t) { return cudaSuccess; }

}  // namespace kvt

// ---- the calls ----
static int fail(const char* what) { std::printf("%s\n", what); return 2; }

int main(int argc, char** argv) {
  if (argc < 5) return fail("arguments");
  std::mt19937_64 rng(std::atoi(argv[1]));
  const uint64_t ring = std::atoi(argv[3]);
  const std::string scenario = argc > 5 ? argv[5] : "";
  kv_pool_desc d{};
  d.n_partitions = 2;
  const uint64_t n_part[2] = {2 * 2 * 200, 2 * 2 * 150}, n = n_part[0] + n_part[1];   // 2 layers of 200 and 150 blocks, 2 heads
  for (int q = 0; q < 2; ++q) {
    kv_partition_desc& p = d.part[q];
    p.model = kv_model_desc{KV_AUTO, 2, 4, 2, 128, 0, 0, 16};
    p.block_tokens = 128;   // 64 KB entries
    p.blocks_per_layer = q == 0 ? 200 : 150;
    p.d_slab = (void*)(kSlab + ((uint64_t)q << 40));
    p.h_ring = (void*)(kPinned + ((uint64_t)q << 40));
    p.ring_slots = ring;
  }
  std::vector<std::vector<uint64_t>> arrays;
  auto real = [&](uint64_t bytes) { arrays.emplace_back(bytes / 8 + 4); return (void*)(((uintptr_t)arrays.back().data() + 15) & ~15ull); };
  d.n_tags = 1 << 20;
  d.d_ema = (float*)real(n * 4); d.d_decay = (float*)real(n * 4); d.d_touch = (uint32_t*)real(n * 4);
  d.d_last_epoch = (uint32_t*)real(n * 4); d.d_pair = (uint8_t*)real(n); d.d_state = (uint8_t*)real(n);
  d.d_tag = (uint32_t*)real(n * 4); d.d_score = (float*)real(n * 4); d.d_hits = (uint64_t*)real(128);
  d.d_misses = (uint64_t*)real(128); d.d_P = (float*)real(64); d.d_loc = (uint32_t*)real(d.n_tags * 4);
  d.alpha0 = d.beta0 = 1.0f;
  const uint64_t batch = 4u << 20;
  d.staging_bytes = batch + 4096;
  for (int b = 0; b < 4; ++b) d.d_staging[b] = (void*)(kStage + ((uint64_t)b << 32));
  d.max_promote = 1024;
  uint64_t dev = 0, host = 0;
  if (kv_workspace_bytes(&d, &dev, &host) != KV_OK) return fail("kv_workspace_bytes");
  d.d_workspace = real(dev); d.workspace_bytes = dev;
  d.h_workspace = real(host); d.h_workspace_bytes = host;
  g_state.assign(n, KV_STATE_FREE);
  const kv_stream_t compute = (void*)1, d2h = (void*)2, h2d = (void*)3;
  kv_pool* p = nullptr;
  if (kv_pool_create(&d, compute, &p) != KV_OK) return fail("kv_pool_create");
  if (kv_set_deferred_packing(p, std::atoi(argv[2])) != KV_OK) return fail("deferred");
  if (kv_set_gather_threshold(p, std::strtoull(argv[4], nullptr, 10)) != KV_OK) return fail("gather threshold");
  std::vector<uint8_t> pairs(n + 16);
  std::vector<std::vector<uint32_t>> keep;   // (deferred packing reads the lists later)
  uint32_t epoch = 0;
  auto ids = [&](int q, bool resident) {
    std::vector<uint32_t> v;
    for (uint64_t i = q ? n_part[0] : 0; i < (q ? n : n_part[0]); ++i)
      if ((g_state[i] == KV_STATE_RESIDENT) == resident) v.push_back((uint32_t)i);
    return v;
  };
  auto demote = [&](const uint64_t want[2]) -> int32_t {
    std::vector<uint32_t> v;
    uint64_t counts[4] = {0, 0, 0, 0};
    for (int q = 0; q < 2; ++q) {
      std::vector<uint32_t> have = ids(q, true);
      std::shuffle(have.begin(), have.end(), rng);
      have.resize(std::min<uint64_t>({have.size(), want[q], ring}));
      counts[q] = have.size();
      v.insert(v.end(), have.begin(), have.end());
    }
    std::sort(v.begin(), v.end());
    const uint64_t m = v.size();
    v.resize(m + 8);
    keep.push_back(std::move(v));
    uint32_t* a = (uint32_t*)(((uintptr_t)keep.back().data() + 15) & ~15ull);
    std::memmove(a, keep.back().data(), m * 4);
    return m ? kv_demote_counted(p, a, m, counts, batch, compute, d2h) : KV_OK;
  };
  auto live = [&](int q) {
    std::vector<uint8_t> l(ring);
    kv_ring_query(p, q, nullptr, nullptr, l.data());
    std::vector<uint64_t> v;
    for (uint64_t i = 0; i < ring; ++i) if (l[i]) v.push_back(i);
    return v;
  };
  auto promote = [&](int q, std::vector<uint64_t> slots) -> int32_t {
    slots.resize(std::min(slots.size(), ids(q, false).size()));
    return slots.empty() ? KV_OK : kv_promote(p, q, slots.data(), slots.size(), batch, compute, h2d);
  };
  auto check = [&](int32_t rc, const char* what) {
    if (rc != KV_OK && g_bad.empty()) g_bad = std::string(what) + " returned " + std::to_string(rc);
  };
  check(kv_admit(p, 0, 0.9f, pairs.data(), pairs.size(), 0, nullptr, compute), "kv_admit");

  const uint64_t small[2] = {8, 0}, large[2] = {ring * 5 / 8, 0};
  if (scenario == "both") {          // large, small, then a promotion of slots of both (the last transfer's)
    check(demote(large), "kv_demote"); check(demote(small), "kv_demote");
    check(promote(0, {large[0] - 2, large[0] - 1, large[0], large[0] + 1}), "kv_promote");
  } else if (scenario == "behind") {   // large, small, small, then a promotion of the large one's slots
    check(demote(large), "kv_demote"); check(demote(small), "kv_demote"); check(demote(small), "kv_demote");
    check(promote(0, {large[0] - 2, large[0] - 1}), "kv_promote");
  } else if (scenario == "wrap") {     // small demotions follow a large one around the ring
    check(demote(large), "kv_demote");
    for (uint64_t i = 0; i < ring / 8 && g_bad.empty(); ++i) check(demote(small), "kv_demote");
  } else {
    for (int step = 0; step < 120 && g_bad.empty(); ++step) {
      const uint64_t what = rng() % 16;
      if (what < 7) {
        uint64_t k[2];
        for (uint64_t& x : k) x = rng() % 3 == 0 ? 0 : rng() % 2 ? 1 + rng() % 8 : 1 + rng() % (ring / 2);
        check(demote(k), "kv_demote");
      } else if (what < 13) {
        const int q = rng() % 2;
        std::vector<uint64_t> l = live(q);
        if (l.empty()) continue;
        if (rng() % 2) std::shuffle(l.begin(), l.end(), rng);
        const uint64_t from = rng() % l.size();
        l.erase(l.begin(), l.begin() + from);
        l.resize(std::min<uint64_t>(l.size(), 1 + rng() % (rng() % 2 ? 8 : 300)));
        check(promote(q, l), "kv_promote");
      } else if (what == 13) {
        uint64_t resident = ids(0, true).size() + ids(1, true).size();
        if (resident) check(kv_select_victims(p, 1 + rng() % resident, (uint32_t*)d.d_score, compute), "kv_select_victims");
      } else if (what == 14) {
        check(kv_hash_entries(p, nullptr, n, (uint8_t*)d.d_loc, compute), "kv_hash_entries");
      } else if (rng() % 2) {
        check(kv_admit(p, ++epoch, 0.9f, pairs.data(), pairs.size(), 0, nullptr, compute), "kv_admit");
      } else if (rng() % 2) {
        check(kv_epoch_score(p, ++epoch, nullptr, nullptr, 0, compute), "kv_epoch_score");
      } else {
        const uint64_t resident = ids(0, true).size() + ids(1, true).size();
        check(kv_epoch_score_select(p, ++epoch, nullptr, nullptr, 0, resident ? 1 + rng() % resident : 0, (uint32_t*)d.d_score, compute),
              "kv_epoch_score_select");
      }
    }
  }
  check(kv_flush(p), "kv_flush");
  kv_pool_destroy(p);
  if (!g_bad.empty()) { std::printf("%s\n", g_bad.c_str()); return 1; }
  return 0;
}
