// One call of a copy of the prefetch list (LIST_SOURCE) on buffers that the test hands over.
#include LIST_SOURCE

extern "C" int prefetch_list(uint32_t* win, unsigned long long* words, uint32_t* serial, uint32_t* status, uint32_t layers,
                             uint32_t heads, uint32_t w_max, const uint32_t* table, uint64_t n_pos, const uint32_t* loc,
                             uint64_t n_tags, unsigned long long* out, uint64_t max_out, unsigned long long* count, void* stream) {
  kvt::PrefetchState pf{};
  pf.win = win;
  pf.words = words;
  pf.serial = serial;
  pf.layers[0] = layers;
  pf.heads[0] = heads;
  pf.w_max[0] = w_max;
  kvt::Workspace ws{};
  ws.status = status;
  return (int)kvt::launch_prefetch_list(pf, 0, table, n_pos, 0, 1, loc, n_tags, out, max_out, count, ws,
                                        static_cast<cudaStream_t>(stream));
}
