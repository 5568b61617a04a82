// The line of kv_dedup.cu's hash kernel played through on the CPU, with the kernel's own rules
// (kv_hash_queue.h): blocks of warps of random speed start as others leave, take places, do slices
// and queue chains again, in memory that holds the words of an earlier, longer call behind the part
// that is cleared.
// usage: hash_queue_sim <messages> <blocks of a message> <thread blocks> <warps of one> <of these resident> <seed>
// prints: place polled at most, the ring's length, chains queued again; exit status 1 and a line on
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
  if (argc != 7) return 2;
  const uint32_t m = std::atoi(argv[1]), longest = std::atoi(argv[2]), blocks = std::atoi(argv[3]);
  const uint32_t per_block = std::atoi(argv[4]), resident = std::atoi(argv[5]);
  std::mt19937_64 rng(std::atoi(argv[6]));
  const HashShape s = hash_shape((m + 31) / 32, longest);
  std::vector<uint64_t> ring(2u * s.ring_places + 2u * blocks * per_block + 64u);
  for (size_t i = s.ring_places; i < ring.size(); ++i) ring[i] = hash_word((uint32_t)(rng() % s.n_chains), 1u + (uint32_t)(rng() % longest));
  std::vector<uint32_t> done(s.n_chains, 0);
  std::vector<char> busy(s.n_chains, 0);

  struct Warp { uint32_t chain, b0, len, at; bool waits; double speed; };
  std::vector<Warp> w(blocks * per_block);
  std::vector<uint32_t> left_in(blocks, per_block);
  using Event = std::pair<double, uint32_t>;
  std::priority_queue<Event, std::vector<Event>, std::greater<Event>> events;
  uint32_t head = 0, tail = 0, finished = 0, most = 0, requeued = 0, started = 0, running = 0, queued = 0;
  const char* bad = nullptr;

  auto begin = [&](uint32_t i, double now, uint32_t chain, uint32_t b0, uint32_t len) {
    if (busy[chain] || done[chain] != b0) bad = "a chain is taken twice, or not where it was left";
    busy[chain] = 1;
    w[i].chain = chain; w[i].b0 = b0; w[i].waits = false;
    w[i].len = len < longest - b0 ? len : longest - b0;
    events.push({now + w[i].len * w[i].speed, i});
    ++running;
  };
  auto leave = [&](uint32_t i) { --left_in[i / per_block]; };
  // warp i looks at ring place w[i].at
  auto look = [&](uint32_t i, double now) {
    const uint64_t v = ring[w[i].at];
    if (v != 0) {
      --queued;
      if (!hash_word_good(s, v)) bad = "a word that no warp has written is taken";
      else begin(i, now, hash_word_chain(v), hash_word_block(v), s.slice_blocks);
    } else if (finished >= s.n_chains) {
      leave(i);
    } else {
      w[i].waits = true;
      events.push({now + 0.7, i});
    }
  };
  auto take = [&](uint32_t i, double now, uint32_t pos, bool first) {
    uint32_t at;
    switch (hash_place(s, pos, at)) {
      case kHashNothing: leave(i); break;
      case kHashChain: begin(i, now, at, 0u, first ? hash_first_slice(s, at) : s.slice_blocks); break;
      case kHashRing:
        if (at > most) most = at;
        w[i].at = at;
        look(i, now);
    }
  };
  double now = 0.0;
  auto start_blocks = [&]() {
    uint32_t here = 0;
    for (uint32_t b = 0; b < started; ++b) here += left_in[b] != 0;
    while (here < resident && started < blocks) {
      const uint32_t b = started++, pos = head;
      head += per_block;
      for (uint32_t k = 0; k < per_block; ++k) {
        w[b * per_block + k].speed = 1.0 + (rng() % 1000) / 500.0;
        take(b * per_block + k, now, pos + k, true);
      }
      here += left_in[b] != 0;
    }
  };
  start_blocks();
  while (!events.empty() && !bad) {
    now = events.top().first;
    const uint32_t i = events.top().second;
    events.pop();
    if (w[i].waits) {
      if (running == 0 && queued == 0 && finished < s.n_chains) return wrong("the warps that run wait for a block that cannot start");
      look(i, now);
    } else {   // a slice has ended
      --running;
      const uint32_t c = w[i].chain;
      done[c] += w[i].len;
      busy[c] = 0;
      if (done[c] < longest) {
        const uint32_t p = tail++;
        ++requeued;
        ++queued;
        if (p >= s.ring_places) return wrong("a chain is queued behind the ring's end");
        ring[p] = hash_word(c, done[c]);
      } else {
        ++finished;
      }
      take(i, now, head++, false);
    }
    if (left_in[i / per_block] == 0) start_blocks();
  }
  if (bad) return wrong(bad);
  if (started != blocks) return wrong("a block has not started");
  for (uint32_t c = 0; c < s.n_chains; ++c)
    if (done[c] != longest) return wrong("a chain is not finished");
  std::printf("%u %u %u\n", most, s.ring_places, requeued);
  return 0;
}
