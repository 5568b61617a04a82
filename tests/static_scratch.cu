// The selection without caller's scratch, on scratch that the test hands over (in any state).
#include "kvtier_internal.cuh"

extern "C" uint64_t scratch_bytes() { return sizeof(kvt::StaticScratch); }
extern "C" uint64_t scratch_words_at() { return offsetof(kvt::StaticScratch, words); }
extern "C" uint64_t scratch_words() { return 1 + kvt::kSharedCtas; }
extern "C" int select_on(const float* score, const uint8_t* state, uint64_t n, uint64_t k, uint32_t* victims, void* scratch,
                         uint32_t* status, void* stream, int variant) {
  return (int)kvt::launch_select_static(score, state, n, k, victims, static_cast<kvt::StaticScratch*>(scratch), status,
                                        static_cast<cudaStream_t>(stream), variant);
}
