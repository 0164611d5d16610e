// Stand-in for the CUDA runtime and the kernel launchers, for tests of the C ABI's host side
// (csrc/api.cu, compiled as plain C++) on a machine without a GPU.  "Device" memory is host memory;
// every call leaves its name in a log; copies are made at once; the launchers launch nothing.
#include <cstdlib>
#include <cstring>
#include <new>
#include <string>
#include <vector>

#include "common.cuh"

namespace {
cudaError_t g_error = cudaSuccess;         // what cudaGetDevice returns
size_t g_limit = SIZE_MAX;                 // C++ allocations above this many bytes fail
std::string g_log;
void note(const char *what) { g_log += what; g_log += ' '; }
struct { const void *p[5]; } g_workers;    // what launch_workers_build was last given
}  // namespace

void *operator new(size_t n) {
  void *p = n > g_limit ? nullptr : malloc(n);
  if (!p) throw std::bad_alloc();
  return p;
}
void *operator new[](size_t n) { return operator new(n); }
void *operator new(size_t n, const std::nothrow_t &) noexcept { return n > g_limit ? nullptr : malloc(n); }
void *operator new[](size_t n, const std::nothrow_t &) noexcept { return n > g_limit ? nullptr : malloc(n); }
void operator delete(void *p) noexcept { free(p); }
void operator delete[](void *p) noexcept { free(p); }
void operator delete(void *p, size_t) noexcept { free(p); }
void operator delete[](void *p, size_t) noexcept { free(p); }

extern "C" {
const char *host_log() { return g_log.c_str(); }
void host_log_clear() { g_log.clear(); }
void host_allocation_limit(size_t n) { g_limit = n; }
void host_device_error(int on) { g_error = on ? cudaErrorNoDevice : cudaSuccess; }
const void *host_workers_table(int i) { return g_workers.p[i]; }
int host_split(uint32_t max_task_variants) {
  infaas::DeviceCatalog c{};
  c.max_task_variants = max_task_variants;
  return infaas::split_for(c);
}
void host_task_share(uint32_t V, uint32_t K, uint32_t share, uint32_t *out) {
  const infaas::TaskShare s = infaas::task_share(V, K, share);
  const uint32_t v[8] = {s.cs, s.ng, s.rows, s.y0, s.lo, s.hi, s.w0, s.w1};
  memcpy(out, v, sizeof(v));
}

cudaError_t cudaGetDevice(int *d) { *d = 0; return g_error; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr, int) { *v = 148; return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
const char *cudaGetErrorName(cudaError_t) { return "an error name that does not fit into a short string"; }
const char *cudaGetErrorString(cudaError_t) { return "of the stand-in"; }
cudaError_t cudaMalloc(void **p, size_t n) {
  note("malloc");
  *p = malloc(n);
  return *p ? cudaSuccess : cudaErrorMemoryAllocation;
}
cudaError_t cudaFree(void *p) { note("free"); free(p); return cudaSuccess; }
cudaError_t cudaMemset(void *p, int v, size_t n) { note("memset"); memset(p, v, n); return cudaSuccess; }
cudaError_t cudaMemsetAsync(void *p, int v, size_t n, cudaStream_t) { return cudaMemset(p, v, n); }
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, cudaMemcpyKind) { note("copy"); memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind k, cudaStream_t) { return cudaMemcpy(d, s, n, k); }
cudaError_t cudaStreamSynchronize(cudaStream_t) { note("wait"); return cudaSuccess; }
cudaError_t cudaDeviceSynchronize() { note("wait"); return cudaSuccess; }
}

namespace infaas {
cudaError_t prepare_select_kernel() { return cudaSuccess; }
cudaError_t prepare_tally_kernel() { return cudaSuccess; }
cudaError_t prepare_rebuild_kernel() { return cudaSuccess; }
uint32_t select_image_smem(uint32_t n) { return n; }
cudaError_t launch_layout(const CatalogLayout &, uint32_t, uint32_t, cudaStream_t) { note("layout"); return cudaSuccess; }
cudaError_t rebuild_clusters_at_once(uint32_t, uint32_t *n) { *n = 33; return cudaSuccess; }
cudaError_t launch_rebuild(const DeviceCatalog &c, bool, uint32_t, cudaStream_t) {
  note(c.rebuild_ctas == 1 ? "rebuild" : "rebuild_by_clusters");
  return cudaSuccess;
}
cudaError_t launch_tally(const DeviceCatalog &, const uint32_t *, uint64_t, int, cudaStream_t) { note("tally"); return cudaSuccess; }
cudaError_t launch_select(const DeviceCatalog &, const uint16_t *, const uint32_t *, const uint16_t *, uint64_t, uint32_t *, int,
                          uint32_t, uint32_t, bool, cudaStream_t) { note("select"); return cudaSuccess; }
cudaError_t launch_autoscale(const DeviceCatalog &, const uint32_t *, const uint16_t *, const unsigned long long *,
                             const uint32_t *, uint32_t, uint32_t, uint32_t, uint32_t *, uint32_t *, cudaStream_t) {
  note("autoscale");
  return cudaSuccess;
}
cudaError_t launch_load_state(const DeviceCatalog &, const uint32_t *, LoadStateTail *tail, unsigned long long *, uint32_t *,
                              uint32_t *, cudaStream_t) {
  note("load_state");
  memset(tail, 0, sizeof(*tail));
  return cudaSuccess;
}
cudaError_t launch_states(const DeviceCatalog &, const uint32_t *, unsigned char *, cudaStream_t) { note("states"); return cudaSuccess; }
cudaError_t launch_scatter(const DeviceCatalog &, const uint32_t *, uint32_t *, const unsigned char *, const uint32_t *, uint32_t *,
                           cudaStream_t) { note("scatter"); return cudaSuccess; }
cudaError_t launch_workers_build(uint32_t, const unsigned char *, const uint32_t *iv, const uint32_t *iw, const uint32_t *il, uint32_t,
                                 const unsigned char *wh, const uint32_t *wu, uint32_t, unsigned long long *, unsigned long long *,
                                 uint32_t *, cudaStream_t) {
  note("workers_build");
  g_workers = {iv, iw, il, wh, wu};
  return cudaSuccess;
}
cudaError_t launch_assign_workers(const uint32_t *, uint64_t, uint32_t, const uint32_t *, uint32_t *, int, int, cudaStream_t) {
  note("assign");
  return cudaSuccess;
}
cudaError_t launch_intpipe_probe(uint32_t, uint32_t, uint32_t *, int, unsigned long long *, cudaStream_t) { return cudaSuccess; }
}  // namespace infaas
