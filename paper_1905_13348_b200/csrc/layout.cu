// Slot order of a catalog (once per load): one CTA per task sorts the task's rows by (cost,
// 10000-acc, id), scatters their attributes into the per-slot arrays and writes down everything
// about the list order that does not hang on the predicted latency.
#include "common.cuh"

namespace infaas {
namespace {

constexpr uint32_t LAYOUT_THREADS = 512;

// Bitonic sort of P (a power of two) keys in shared memory, ascending.  All threads; ends in a barrier.
template <class T>
__device__ __forceinline__ void sort_shared(T *k, uint32_t P) {
  for (uint32_t size = 2; size <= P; size <<= 1)
    for (uint32_t j = size >> 1; j > 0; j >>= 1) {
      __syncthreads();
      for (uint32_t x = threadIdx.x; x < (P >> 1); x += blockDim.x) {
        const uint32_t i = ((x & ~(j - 1u)) << 1) | (x & (j - 1u)), l = i | j;   // lower and upper index of the pair
        const T a = k[i], b = k[l];
        if (((i & size) == 0u) == (b < a)) { k[i] = b; k[l] = a; }
      }
    }
  __syncthreads();
}

// Number of sorted keys below x.
__device__ __forceinline__ uint32_t lower_bound(const unsigned long long *k, uint32_t n, unsigned long long x) {
  uint32_t lo = 0;
  while (n) {
    const uint32_t half = n >> 1;
    if (k[lo + half] < x) { lo += half + 1u; n -= half + 1u; } else n = half;
  }
  return lo;
}

__global__ void __launch_bounds__(LAYOUT_THREADS)
layout_kernel(CatalogLayout o) {
  extern __shared__ __align__(16) unsigned char dyn[];
  __shared__ uint32_t warp_cnt[LAYOUT_THREADS / 32];
  const uint32_t t = blockIdx.x, tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5;
  const uint32_t base = o.task_off[t], V = o.task_off[t + 1] - base;
  uint32_t P = 1;
  while (P < V) P <<= 1;
  unsigned long long *key = reinterpret_cast<unsigned long long *>(dyn);   // cost | 10000 - acc (14 bits) | index (13 bits)
  uint32_t *by_acc = reinterpret_cast<uint32_t *>(key + P);                // 10000 - acc | local index (13 bits)
  uint32_t *head = by_acc + P;                                             // order word without the position
  for (uint32_t i = tid; i < P; i += LAYOUT_THREADS) {
    unsigned long long k = ~0ull;
    if (i < V) {
      const infaas_variant &r = o.rows[o.members[base + i]];
      k = ((unsigned long long)r.cost << 27) | ((unsigned long long)(10000u - r.acc_bp) << 13) | i;
    }
    key[i] = k;
  }
  sort_shared(key, P);
  for (uint32_t p = tid; p < P; p += LAYOUT_THREADS) {
    if (p >= V) { by_acc[p] = 0xFFFFFFFFu; continue; }
    const unsigned long long k = key[p];
    const uint32_t slot = base + p, id = o.members[base + (uint32_t)(k & 0x1FFFu)];
    const infaas_variant r = o.rows[id];
    o.s_lat[slot] = r.lat_us; o.s_batch[slot] = r.batch; o.s_acc[slot] = r.acc_bp; o.s_cost[slot] = r.cost;
    o.s_id[slot] = id; o.s_queued[slot] = r.queued; o.s_arch[slot] = r.arch;
    o.s_qps[slot] = 1000000000ull * r.batch / r.lat_us;                    // floor(10^9 * batch / lat_us)
    o.slot_of_id[id] = slot; o.hw_by_id[id] = r.hw;
    o.s_cost_run[slot] = lower_bound(key, V, (unsigned long long)r.cost << 27) |
                         (lower_bound(key, V, ((unsigned long long)r.cost + 1ull) << 27) << 16);
    const uint32_t first = lower_bound(key, V, k & ~0x1FFFull);
    const bool many = first != p || (p + 1u < V && (key[p + 1u] >> 13) == (k >> 13));
    head[p] = (first << 13) | (many ? 0x80000000u : 0u);
    by_acc[p] = ((10000u - r.acc_bp) << 13) | p;
  }
  sort_shared(by_acc, P);
  uint32_t classes = 0;                                                     // distinct accuracies so far
  for (uint32_t p0 = 0; p0 < V; p0 += LAYOUT_THREADS) {                     // uniform trip count
    const uint32_t p = p0 + tid;
    const uint32_t e = p < V ? by_acc[p] : 0u;
    const bool fresh = p < V && (p == 0u || (by_acc[p - 1u] >> 13) != (e >> 13));
    const unsigned m = __ballot_sync(0xFFFFFFFFu, fresh);
    __syncthreads();
    if (lane == 0u) warp_cnt[warp] = __popc(m);
    __syncthreads();
    uint32_t before = classes;
    for (uint32_t w = 0; w < LAYOUT_THREADS / 32; ++w) {
      before += w < warp ? warp_cnt[w] : 0u;
      classes += warp_cnt[w];
    }
    if (p < V) {
      const uint32_t local = e & 0x1FFFu, k = before + __popc(m & ((2u << lane) - 1u)) - 1u;
      o.s_order[base + local] = p | head[local];
      o.s_class[base + local] = (uint16_t)k;
      if (fresh) o.class_acc[base + k] = (uint16_t)(10000u - (e >> 13));
      uint32_t before_too = 0;
      for (uint32_t q = p & ~31u; q < p; ++q) before_too |= (uint32_t)((by_acc[q] & 0x1FFFu) < local) << (q & 31u);
      o.by_acc[base + p] = make_uint2(local, before_too);
    }
  }
  if (tid == 0u) o.n_class[t] = classes;
}

}  // namespace

cudaError_t launch_layout(const CatalogLayout &o, uint32_t n_tasks, uint32_t max_task_variants, cudaStream_t stream) {
  uint32_t P = 1;
  while (P < max_task_variants) P <<= 1;
  const size_t smem = (size_t)P * 16;                                       // 128 KB at the limit of 8192
  cudaError_t e = cudaFuncSetAttribute(layout_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)(INFAAS_MAX_TASK_VARIANTS * 16u));
  if (e != cudaSuccess) return e;
  layout_kernel<<<n_tasks, LAYOUT_THREADS, smem, stream>>>(o);
  return cudaGetLastError();
}

}  // namespace infaas
