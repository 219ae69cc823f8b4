// The host side of the library (csrc/c2t_api.cu) over a CUDA runtime that does nothing but write down what it is asked, for
// tests without a GPU: in which order copies, clears, waits and launches are issued, and what becomes of a call that fails.
#include <cuda_runtime.h>
#include <math.h>
#include <stdarg.h>
#include <stdio.h>
#include <string.h>

#include <string>

inline unsigned __float_as_uint(float x) { unsigned u; memcpy(&u, &x, 4); return u; }
inline float __uint_as_float(unsigned u) { float x; memcpy(&x, &u, 4); return x; }

namespace fake {
std::string log, fail_name;
int fail_at = 0, device = 0, events = 0, streams = 0;
size_t next_handle = 0x100;

cudaError_t call(const char *name, const char *fmt, ...) {
  char args[256];
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(args, sizeof args, fmt, ap);
  va_end(ap);
  const bool fails = fail_at > 0 && fail_name == name && --fail_at == 0;
  log += std::string(name) + " " + args + (fails ? " FAILED\n" : "\n");
  return fails ? cudaErrorUnknown : cudaSuccess;
}
}  // namespace fake

extern "C" {
const char *fake_log() { return fake::log.c_str(); }
void fake_reset() { fake::log.clear(); fake::fail_at = 0; fake::device = 0; }
void fake_fail(const char *name, int at) { fake::fail_name = name; fake::fail_at = at; }
int fake_events() { return fake::events; }
int fake_streams() { return fake::streams; }

cudaError_t cudaSetDevice(int d) { fake::device = d; return cudaSuccess; }
cudaError_t cudaGetDevice(int *d) { *d = fake::device; return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr, int) { *v = 148; return cudaSuccess; }
cudaError_t cudaMemcpy(void *d, const void *, size_t n, cudaMemcpyKind) { return fake::call("memcpy", "%p %zu", d, n); }
cudaError_t cudaMemset(void *d, int, size_t n) { return fake::call("memset", "%p %zu", d, n); }
cudaError_t cudaMemsetAsync(void *d, int, size_t n, cudaStream_t s) { return fake::call("memset_async", "%p %zu %p", d, n, (void *)s); }
cudaError_t cudaMemcpyAsync(void *d, const void *, size_t n, cudaMemcpyKind k, cudaStream_t s) {
  return fake::call(k == cudaMemcpyHostToDevice ? "copy" : "copy_back", "%p %zu %p", d, n, (void *)s);
}
cudaError_t cudaMemcpy2DAsync(void *d, size_t dp, const void *, size_t, size_t, size_t h, cudaMemcpyKind, cudaStream_t s) {
  return fake::call("copy", "%p %zu %p", d, dp * h, (void *)s);
}
cudaError_t cudaStreamSynchronize(cudaStream_t s) { return fake::call("sync", "%p", (void *)s); }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) {
  *s = (cudaStream_t)fake::next_handle++;
  const cudaError_t e = fake::call("create_stream", "%p device %d", (void *)*s, fake::device);
  fake::streams += e == cudaSuccess;
  return e;
}
cudaError_t cudaStreamDestroy(cudaStream_t s) { --fake::streams; return fake::call("destroy_stream", "%p", (void *)s); }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *ev, unsigned) {
  *ev = (cudaEvent_t)fake::next_handle++;
  const cudaError_t e = fake::call("create_event", "%p device %d", (void *)*ev, fake::device);
  fake::events += e == cudaSuccess;
  return e;
}
cudaError_t cudaEventDestroy(cudaEvent_t ev) { --fake::events; return fake::call("destroy_event", "%p", (void *)ev); }
cudaError_t cudaEventRecord(cudaEvent_t ev, cudaStream_t s) { return fake::call("record", "%p %p", (void *)ev, (void *)s); }
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t ev, unsigned) { return fake::call("wait", "%p %p", (void *)s, (void *)ev); }
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes *a, const void *p) {       // (every host buffer is pinned here)
  memset(a, 0, sizeof *a);
  a->type = cudaMemoryTypeHost;
  a->hostPointer = a->devicePointer = const_cast<void *>(p);
  return cudaSuccess;
}
}

#include "../paper_2502_13652_b200/csrc/c2t_api.cu"

namespace c2t {
cudaError_t prepare_expand_pass() { return cudaSuccess; }
cudaError_t prepare_topm_pass() { return cudaSuccess; }
cudaError_t prepare_tree_kernels() { return cudaSuccess; }
cudaError_t prepare_accept_lazy() { return cudaSuccess; }
int row_chunks(int vocab, int elem_bytes) { return (vocab * elem_bytes + 4095) / 4096; }
int topm_floor_place(int vocab, int, int M) { return 4 * M > vocab ? 0 : 24; }
size_t topm_pool_vectors(size_t batch, size_t rows, int vocab, int elem_bytes) { return batch * rows * vocab * elem_bytes / 48; }

static cudaError_t launched(const char *name, cudaStream_t s, const void *reads = nullptr) { return fake::call(name, "%p %p", (void *)s, reads); }
cudaError_t launch_expand_pass(PassParams p, int, int, cudaStream_t s) { return launched("expand", s, p.logits); }
cudaError_t launch_expand_prune(PassParams p, const TreeState &, int, const c2t_frontier *, int, int, cudaStream_t s) { return launched("expand", s, p.logits); }
cudaError_t launch_argmax_pass(const PassParams &p, int, int, cudaStream_t s) { return launched("argmax", s, p.logits); }
cudaError_t launch_accept_lazy(const TreeState &, const void *l, int64_t, int64_t, const c2t_accept_out *, int, int, cudaStream_t s) { return launched("accept_lazy", s, l); }
cudaError_t launch_topm_entropy(const void *l, int64_t, int64_t, int, int, int, int, const int32_t *, const TreeState &, double2 *, const int32_t *,
                                int, int, cudaStream_t s) { return launched("topm_entropy", s, l); }
cudaError_t launch_topm_finish(int, int, int, const int32_t *, const TreeState &, double2 *, int, cudaStream_t s) { return launched("topm_finish", s); }
cudaError_t launch_begin_step(const TreeState &, const int32_t *, const int32_t *, cudaStream_t s) { return launched("begin", s); }
cudaError_t launch_prune_level(const TreeState &, int, const c2t_frontier *, const c2t_row_record *, int, cudaStream_t s) { return launched("prune", s); }
cudaError_t launch_export_rows(const TreeState &, int, int, c2t_row_record *, cudaStream_t s) { return launched("export_rows", s); }
cudaError_t launch_final_prune(const TreeState &, cudaStream_t s) { return launched("final_prune", s); }
cudaError_t launch_build_verify(const TreeState &, const c2t_verify *, cudaStream_t s) { return launched("build_verify", s); }
cudaError_t launch_dense_mask(const TreeState &, void *, int, int64_t, cudaStream_t s) { return launched("dense_mask", s); }
cudaError_t launch_accept_walk(const TreeState &, const c2t_accept_out *, const unsigned long long *, int, cudaStream_t s) { return launched("accept_walk", s); }
cudaError_t launch_export_best(const TreeState &, int, unsigned long long *, cudaStream_t s) { return launched("export_best", s); }
cudaError_t launch_lazy_walk_round(const TreeState &, int, const c2t_accept_out *, const unsigned long long *, int, cudaStream_t s) { return launched("lazy_walk", s); }
cudaError_t launch_export_lazy_best(const TreeState &, int, unsigned long long *, cudaStream_t s) { return launched("export_lazy_best", s); }
}  // namespace c2t

extern "C" void fake_row_plan(int vocab, int elem_bytes, long long rows, int K, int sms, int *cluster, int *threads) {
  const c2t::RowPlan plan = c2t::row_pass_plan(vocab, elem_bytes, rows, K, sms);
  *cluster = plan.cluster;
  *threads = plan.threads;
}
