// The line in which chains of messages wait for a warp (kv_dedup.cu), as rules without memory or
// threads: how long it can get, what a place in it stands for, and which words in it are good.  Plain
// C++, so that they are the same in the kernel and where its arithmetic is checked.
#pragma once
#include <cstdint>

#ifdef __CUDACC__
#define KV_QUEUE_FN __host__ __device__ __forceinline__
#else
#define KV_QUEUE_FN inline
#endif

namespace kvt {

constexpr uint32_t kHashSlices = 7;

struct HashShape {
  uint32_t n_chains = 0;
  uint32_t slice_blocks = 0;   // blocks of a slice: a seventh of the longest message
  uint32_t longest = 0;        // blocks of the longest message
  uint32_t ring_places = 0;    // times that chains can be queued again, all together
};

// A chain's first slice has 1 to slice_blocks blocks, each further one has slice_blocks until the
// message ends.  After the first block at most (longest - 1) / slice_blocks, rounded up, slices are
// left, which is at most kHashSlices: so often is a chain queued again, at most.
KV_QUEUE_FN HashShape hash_shape(uint32_t n_chains, uint32_t longest) {
  HashShape s;
  s.n_chains = n_chains;
  s.longest = longest;
  s.slice_blocks = (longest + kHashSlices - 1u) / kHashSlices;
  s.ring_places = n_chains * kHashSlices;
  return s;
}

KV_QUEUE_FN uint32_t hash_first_slice(const HashShape& s, uint32_t chain) {
  return 1u + (chain * 2654435761u >> 8) % s.slice_blocks;
}

// Place number pos in the line: a chain that nobody has begun (at: which), a place of the ring of
// chains queued again (at: which), or one behind all of these, for which nothing can ever come.
// Every warp takes one place more than it gets work from, so such places are taken.
enum HashPlace { kHashChain, kHashRing, kHashNothing };
KV_QUEUE_FN HashPlace hash_place(const HashShape& s, uint32_t pos, uint32_t& at) {
  at = pos;
  if (pos < s.n_chains) return kHashChain;
  at = pos - s.n_chains;
  return at < s.ring_places ? kHashRing : kHashNothing;
}

// A word of the ring: bit 63 | the chain's next block << 32 | the chain; 0 until it is written.
KV_QUEUE_FN uint64_t hash_word(uint32_t chain, uint32_t block) { return 1ull << 63 | (uint64_t)block << 32 | chain; }
KV_QUEUE_FN uint32_t hash_word_chain(uint64_t w) { return (uint32_t)w; }
KV_QUEUE_FN uint32_t hash_word_block(uint64_t w) { return (uint32_t)(w >> 32) & 0x7FFFFFFFu; }
KV_QUEUE_FN bool hash_word_good(const HashShape& s, uint64_t w) {
  return (w >> 63) != 0u && hash_word_chain(w) < s.n_chains && hash_word_block(w) < s.longest;
}

}  // namespace kvt
