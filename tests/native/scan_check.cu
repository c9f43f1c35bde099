// Calls the library's exclusive scan of counts (csrc/tree.cu) on arrays of the
// caller (tests/test_gpu_scan_range.py builds this against libsph.so).
#include "sph_internal.cuh"

namespace sph {
void scan_counts(sph_ctx *c, const int32_t *in, int32_t *out, int64_t m, cudaStream_t st);
void scan_counts(sph_ctx *c, const int32_t *in, int64_t *out, int64_t m, cudaStream_t st);
}  // namespace sph

// look: look_words(m, m) words of scratch; err: a zeroed device word
template <class O>
static int run(const int32_t *in, O *out, int64_t m, uint32_t *look, int32_t *err, void *stream) {
  sph_ctx c;
  memset(&c, 0, sizeof(c));
  c.tree.look = look;
  c.d_err = err;
  sph::scan_counts(&c, in, out, m, (cudaStream_t)stream);
  return (int)cudaGetLastError();
}

extern "C" int64_t scan_look_words(int64_t m) { return sph::look_words(m, m); }
extern "C" int scan32(const int32_t *in, int32_t *out, int64_t m, uint32_t *look, int32_t *err, void *stream) {
  return run(in, out, m, look, err, stream);
}
extern "C" int scan64(const int32_t *in, int64_t *out, int64_t m, uint32_t *look, int32_t *err, void *stream) {
  return run(in, out, m, look, err, stream);
}
