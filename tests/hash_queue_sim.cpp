// The line of kv_dedup.cu's hash kernel played through on the CPU, with the kernel's own rules
// (kv_hash_queue.h): warps of random speed take places, do slices and queue chains again, in memory
// that holds the words of an earlier, longer call behind the part that is cleared.
// usage: hash_queue_sim <messages> <blocks of a message> <warps> <seed>
// prints: places polled at most, the ring's length, chains queued again; exit status 1 and a line on
// the first wrong step.
#include <cstdio>
#include <cstdlib>
#include <queue>
#include <random>
#include <vector>

#include "kv_hash_queue.h"

using namespace kvt;

static int wrong(const char* what) {
  std::printf("wrong: %s\n", what);
  return 1;
}

int main(int argc, char** argv) {
  if (argc != 5) return 2;
  const uint32_t m = std::atoi(argv[1]), longest = std::atoi(argv[2]), warps = std::atoi(argv[3]);
  std::mt19937_64 rng(std::atoi(argv[4]));
  const HashShape s = hash_shape((m + 31) / 32, warps, longest);
  std::vector<uint64_t> ring(2u * s.ring_places + 2u * warps + 64u);
  for (size_t i = s.ring_places; i < ring.size(); ++i) ring[i] = hash_word((uint32_t)(rng() % s.n_chains), 1u + (uint32_t)(rng() % longest));
  std::vector<uint32_t> done(s.n_chains, 0);
  std::vector<char> busy(s.n_chains, 0);

  struct Warp { uint32_t chain, b0, len, at; bool waits, gone; double speed; };
  std::vector<Warp> w(warps);
  using Event = std::pair<double, uint32_t>;
  std::priority_queue<Event, std::vector<Event>, std::greater<Event>> events;
  auto begin = [&](uint32_t i, double now) {
    const uint32_t left = s.longest - w[i].b0, n = w[i].len < left ? w[i].len : left;
    events.push({now + n * w[i].speed, i});
  };
  uint32_t head = 0, tail = 0, finished = 0, most = 0, requeued = 0;
  for (uint32_t i = 0; i < warps; ++i) {
    w[i] = Warp{i, 0u, hash_first_slice(s, i), 0u, false, false, 1.0 + (rng() % 1000) / 500.0};
    if (i >= s.n_chains) return wrong("fewer chains than warps");
    busy[i] = 1;
    begin(i, 0.0);
  }
  while (!events.empty()) {
    const double now = events.top().first;
    const uint32_t i = events.top().second;
    events.pop();
    Warp& x = w[i];
    if (!x.waits) {   // a slice has ended
      const uint32_t left = s.longest - x.b0, n = x.len < left ? x.len : left;
      if (done[x.chain] != x.b0 || !busy[x.chain]) return wrong("a chain goes on from another block than it was left at");
      done[x.chain] += n;
      busy[x.chain] = 0;
      if (done[x.chain] < s.longest) {
        const uint32_t p = tail++;
        ++requeued;
        if (p >= s.ring_places) return wrong("a chain is queued behind the ring's end");
        ring[p] = hash_word(x.chain, done[x.chain]);
      } else {
        ++finished;
      }
      uint32_t at;
      switch (hash_place(s, s.n_warps + head++, at)) {
        case kHashNothing: x.gone = true; continue;
        case kHashRing:
          if (at > most) most = at;
          x.waits = true;
          x.at = at;
          break;
        case kHashChain:
          x.chain = at; x.b0 = 0; x.len = s.slice_blocks;
          if (busy[at] || done[at]) return wrong("a chain is begun twice");
          busy[at] = 1;
          begin(i, now);
          continue;
      }
    }
    const uint64_t v = ring[x.at];
    if (v != 0) {
      if (!hash_word_good(s, v)) return wrong("a word that no warp has written is taken");
      x.chain = hash_word_chain(v); x.b0 = hash_word_block(v); x.len = s.slice_blocks; x.waits = false;
      if (busy[x.chain]) return wrong("a chain is taken twice");
      busy[x.chain] = 1;
      begin(i, now);
    } else if (finished >= s.n_chains) {
      x.gone = true;
    } else {
      events.push({now + 0.7, i});   // looks again
    }
  }
  for (uint32_t c = 0; c < s.n_chains; ++c)
    if (done[c] != s.longest) return wrong("a chain is not finished");
  std::printf("%u %u %u\n", most, s.ring_places, requeued);
  return 0;
}
