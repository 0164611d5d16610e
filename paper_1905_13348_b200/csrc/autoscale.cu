// Scaling-up step of the Model-Autoscaler on the window's tallies (Section 4.2.2, "A Greedy
// Heuristic"; cost function and constraints (1), (2), (4) of Section 4.2.1): one CTA per
// task compares the running variants' saturation throughput with the load they served and,
// if the headroom is too small, prices "replicate the running variant" against "add a faster
// variant of the same architecture".  All arithmetic is unsigned integer arithmetic with
// explicit saturation; the cost is compared as a 128-bit product.
#include "common.cuh"

namespace infaas {
namespace {

constexpr uint32_t AUTOSCALE_THREADS = 256;
constexpr unsigned long long U64_MAX_ = ~0ull;

__device__ __forceinline__ unsigned long long sat_add(unsigned long long a, unsigned long long b) {
  const unsigned long long s = a + b;
  return s < a ? U64_MAX_ : s;
}
__device__ __forceinline__ unsigned long long sat_mul(unsigned long long a, unsigned long long b) {
  return __umul64hi(a, b) ? U64_MAX_ : a * b;
}
// ceil(x * m / 100), saturating at 2^64-1.
__device__ unsigned long long scale_pct_ceil(unsigned long long x, uint32_t m) {
  unsigned long long hi = __umul64hi(x, (unsigned long long)m), lo = x * m;
  const unsigned long long lo99 = lo + 99ull;
  hi += lo99 < lo;
  lo = lo99;
  if (hi >= 100ull) return U64_MAX_;
  // (hi * 2^64 + lo) / 100 by two 64-bit divisions; hi < 100 keeps each quotient below 2^32
  const unsigned long long t1 = (hi << 32) | (lo >> 32);
  const unsigned long long q1 = t1 / 100ull, r1 = t1 % 100ull;
  const unsigned long long t0 = (r1 << 32) | (lo & 0xFFFFFFFFull);
  return (q1 << 32) | (t0 / 100ull);
}

// A candidate: its cost as four words from the top, kind << 31 | id, instances to add.  `any` = false: none.
struct Action {
  uint32_t w[5], delta;
  bool any;
};
// The smallest (cost, kind, id) of the warp, in all lanes: one reduction per word among the lanes that were
// smallest so far; ids differ, so one lane is left.
__device__ __forceinline__ Action smallest(const Action &a) {
  bool in = a.any;
  Action r;
  r.any = __any_sync(0xFFFFFFFFu, in);
#pragma unroll
  for (int k = 0; k < 5; ++k) {
    r.w[k] = __reduce_min_sync(0xFFFFFFFFu, in ? a.w[k] : 0xFFFFFFFFu);
    in = in && a.w[k] == r.w[k];
  }
  r.delta = __reduce_max_sync(0xFFFFFFFFu, in ? a.delta : 0u);
  return r;
}

// What a variant brings to the decision: fixed, and what earlier kernels of the stream have written.
struct Variant {
  uint32_t id, lat, cost, arch, count, instances, load_lat;
  unsigned long long q;                          // saturation throughput, milli-queries/s
};

// Bound by latency: two rounds of loads (the count is found by id), two 64-bit divisions, and three passes of
// reductions.  A thread keeps its first variant in registers, fetched as far as it is fixed before the wait;
// every warp combines all warps' sums and divides for itself, which saves a barrier and a broadcast.  64 tasks x
// 256 variants, one call in a graph of 50: 4.5 -> 3.0 us.
__global__ void __launch_bounds__(AUTOSCALE_THREADS)
autoscale_kernel(DeviceCatalog c, const uint32_t *s_inst, const uint16_t *s_arch,
                 const unsigned long long *s_qps, const uint32_t *task_slo,
                 uint32_t window_us, uint32_t slack_pct, uint32_t lambda_milli, uint32_t *out_variant,
                 uint32_t *out_delta) {
  constexpr uint32_t WARPS = AUTOSCALE_THREADS / 32;
  __shared__ unsigned long long w_served[WARPS], w_cap[WARPS], w_key[WARPS];
  __shared__ uint32_t w_slot[WARPS];
  __shared__ Action w_best[WARPS];
  const uint32_t t = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t lo = c.task_off[t], hi = c.task_off[t + 1];
  auto load_fixed = [&](uint32_t s, Variant &v) {
    v.id = c.s_id[s]; v.lat = c.s_lat[s]; v.cost = c.s_cost[s]; v.arch = s_arch[s]; v.q = s_qps[s];
  };
  auto load_rest = [&](uint32_t s, Variant &v) {
    v.count = c.count_by_id[v.id]; v.instances = s_inst[s]; v.load_lat = c.s_load_lat[s];
  };
  Variant v0{};
  if (lo + tid < hi) load_fixed(lo + tid, v0);
  chain_wait();
  chain_next();
  const uint32_t slo = task_slo[t];

  // load served, capacity of what runs, and which running variant served most (ties: lower id)
  unsigned long long served = 0, cap = 0, key = 0;
  uint32_t r = 0xFFFFFFFFu;                      // slot of the running variant, ~0 if none
  Variant v = v0;
#pragma unroll 1
  for (uint32_t s = lo + tid; s < hi; s += AUTOSCALE_THREADS) {
    if (s != lo + tid) load_fixed(s, v);
    load_rest(s, v);
    if (s == lo + tid) v0 = v;
    served += v.count;
    if (v.instances) {
      cap = sat_add(cap, sat_mul(v.instances, v.q));
      const unsigned long long k = ((unsigned long long)v.count << 32) | (0xFFFFFFFFu - v.id);
      if (k > key) { key = k; r = s; }
    }
  }
  auto combine = [&](uint32_t from) {
    for (uint32_t o = from; o; o >>= 1) {
      served += __shfl_xor_sync(0xFFFFFFFFu, served, o);
      cap = sat_add(cap, __shfl_xor_sync(0xFFFFFFFFu, cap, o));
      const unsigned long long k = __shfl_xor_sync(0xFFFFFFFFu, key, o);
      const uint32_t ks = __shfl_xor_sync(0xFFFFFFFFu, r, o);
      if (k > key) { key = k; r = ks; }
    }
  };
  combine(16);
  if (lane == 0) { w_served[warp] = served; w_cap[warp] = cap; w_key[warp] = key; w_slot[warp] = r; }
  __syncthreads();
  static_assert((WARPS & (WARPS - 1u)) == 0u && WARPS <= 32u, "lanes w, w + WARPS, ... hold warp w's sums");
  served = w_served[lane % WARPS]; cap = w_cap[lane % WARPS]; key = w_key[lane % WARPS]; r = w_slot[lane % WARPS];
  combine(WARPS / 2);
  if (served > 0xFFFFFFFFull) served = 0xFFFFFFFFull;
  const unsigned long long need = scale_pct_ceil(served * 1000000000ull / window_us, slack_pct);
  if (cap >= need) {                              // headroom suffices
    if (tid == 0) { out_variant[t] = INFAAS_AUTOSCALE_NONE; out_delta[t] = 0u; }
    return;
  }
  const unsigned long long deficit = need - cap;
  unsigned long long q_r = 0;
  uint32_t arch_r = 0;
  if (r != 0xFFFFFFFFu) { q_r = s_qps[r]; arch_r = s_arch[r]; }

  Action best;
  best.any = false;
  best.delta = 0;
  for (int k = 0; k < 5; ++k) best.w[k] = 0xFFFFFFFFu;
  v = v0;
#pragma unroll 1
  for (uint32_t s = lo + tid; s < hi; s += AUTOSCALE_THREADS) {
    if (s != lo + tid) { load_fixed(s, v); load_rest(s, v); }
    if (v.q == 0ull || v.lat > slo) continue;     // constraint (2): new instances meet the SLO
    uint32_t kind = 1;                             // 0 replicate, 1 upgrade
    if (s == r) kind = 0;
    else if (r != 0xFFFFFFFFu && (v.arch != arch_r || v.q <= q_r)) continue;
    const unsigned long long whole = deficit / v.q, delta = whole + (whole * v.q != deficit);
    if (delta > 0xFFFFFFFFull) continue;
    const unsigned long long a = (unsigned long long)v.cost * delta;                      // < 2^64
    const unsigned long long f = 1000000000ull + (unsigned long long)lambda_milli * v.load_lat;
    const unsigned long long cost_hi = __umul64hi(a, f), cost_lo = a * f;
    const uint32_t w[5] = {(uint32_t)(cost_hi >> 32), (uint32_t)cost_hi, (uint32_t)(cost_lo >> 32), (uint32_t)cost_lo,
                           kind << 31 | v.id};
    bool less = !best.any, same = best.any;
#pragma unroll
    for (int k = 0; k < 5; ++k) {
      less = less || (same && w[k] < best.w[k]);
      same = same && w[k] == best.w[k];
    }
    if (less) {
#pragma unroll
      for (int k = 0; k < 5; ++k) best.w[k] = w[k];
      best.delta = (uint32_t)delta;
      best.any = true;
    }
  }
  best = smallest(best);
  if (lane == 0) w_best[warp] = best;
  __syncthreads();
  if (warp == 0) {
    best = w_best[lane % WARPS];
    best.any = best.any && lane < WARPS;
    best = smallest(best);
    if (lane == 0) {
      out_variant[t] = best.any ? best.w[4] & 0x7FFFFFFFu : INFAAS_AUTOSCALE_ESCALATE;
      out_delta[t] = best.any ? best.delta : 0u;
    }
  }
}

}  // namespace

cudaError_t launch_autoscale(const DeviceCatalog &c, const uint32_t *s_inst, const uint16_t *s_arch,
                             const unsigned long long *s_qps, const uint32_t *task_slo, uint32_t window_us, uint32_t slack_pct,
                             uint32_t lambda_milli, uint32_t *d_variant, uint32_t *d_delta,
                             cudaStream_t stream) {
  return launch_chained(autoscale_kernel, c.n_tasks, AUTOSCALE_THREADS, 0, split_for(c), stream, c, s_inst, s_arch, s_qps, task_slo,
                        window_us, slack_pct, lambda_milli, d_variant, d_delta);
}

}  // namespace infaas
