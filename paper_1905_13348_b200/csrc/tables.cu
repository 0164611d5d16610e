// Between the caller's tables, which are ordered by variant id, and the per-slot arrays: the
// permutations run here, so that a table crosses PCIe once, in one piece, and the host neither
// permutes nor waits in between.
#include "common.cuh"

namespace infaas {
namespace {

constexpr uint32_t TABLE_THREADS = 256;
inline uint32_t blocks_for(uint32_t n) { return (n + TABLE_THREADS - 1) / TABLE_THREADS; }

__global__ void __launch_bounds__(TABLE_THREADS)
load_state_kernel(DeviceCatalog c, const uint32_t *slot_of_id, LoadStateTail *tail, unsigned long long *served,
                  uint32_t *queued, uint32_t *pred) {
  const uint32_t v = blockIdx.x * TABLE_THREADS + threadIdx.x;
  const uint32_t s = v < c.n_variants ? slot_of_id[v] : 0u;
  chain_wait();
  chain_next();
  if (v < c.n_variants) {
    served[v] = c.s_served[s];
    queued[v] = c.s_queued[s];
    pred[v] = c.s_pred[s];
  }
  if (v == 0u) {
    for (int i = 0; i < 3; ++i) tail->counters[i] = c.counters[i];
    tail->err = *c.err;
    tail->image_bytes = c.image_hdr[0];
  }
}

__global__ void __launch_bounds__(TABLE_THREADS)
states_kernel(DeviceCatalog c, const uint32_t *slot_of_id, unsigned char *state) {
  const uint32_t v = blockIdx.x * TABLE_THREADS + threadIdx.x;
  const uint32_t s = v < c.n_variants ? slot_of_id[v] : 0u;
  chain_wait();
  chain_next();
  if (v < c.n_variants) state[v] = c.s_state[s];
}

// Per-slot u32 (and, with state_by_id, state) from tables by id; a u32 table per task is copied.
__global__ void __launch_bounds__(TABLE_THREADS)
scatter_kernel(DeviceCatalog c, const uint32_t *value_by_id, uint32_t *s_value, const unsigned char *state_by_id,
               const uint32_t *by_task, uint32_t *task_value) {
  const uint32_t i = blockIdx.x * TABLE_THREADS + threadIdx.x;
  const uint32_t id = i < c.n_variants ? c.s_id[i] : 0u;
  chain_wait();
  chain_next();
  if (i < c.n_variants) {
    s_value[i] = value_by_id ? value_by_id[id] : 0u;
    if (state_by_id) c.s_state[i] = state_by_id[id];
  }
  if (by_task && i < c.n_tasks) task_value[i] = by_task[i];
}

}  // namespace

cudaError_t launch_load_state(const DeviceCatalog &c, const uint32_t *slot_of_id, LoadStateTail *tail,
                              unsigned long long *served, uint32_t *queued, uint32_t *pred, cudaStream_t stream) {
  return launch_chained(load_state_kernel, blocks_for(c.n_variants), TABLE_THREADS, 0, split_for(c), stream, c, slot_of_id, tail, served,
                        queued, pred);
}

cudaError_t launch_states(const DeviceCatalog &c, const uint32_t *slot_of_id, unsigned char *state, cudaStream_t stream) {
  return launch_chained(states_kernel, blocks_for(c.n_variants), TABLE_THREADS, 0, split_for(c), stream, c, slot_of_id, state);
}

cudaError_t launch_scatter(const DeviceCatalog &c, const uint32_t *value_by_id, uint32_t *s_value,
                           const unsigned char *state_by_id, const uint32_t *by_task, uint32_t *task_value,
                           cudaStream_t stream) {
  const uint32_t n = c.n_variants > c.n_tasks ? c.n_variants : c.n_tasks;
  return launch_chained(scatter_kernel, blocks_for(n), TABLE_THREADS, 0, split_for(c), stream, c, value_by_id, s_value, state_by_id,
                        by_task, task_value);
}

}  // namespace infaas
