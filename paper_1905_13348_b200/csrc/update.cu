// Load tallies: how many of a window's decisions each variant got (Section 4.2.2 of the paper
// tracks the load a variant serves from the queries it is given).  The queue recursion and the
// scan lists that follow from the counts are in rebuild.cu.
#include "common.cuh"

namespace infaas {

namespace {

// ------------------------------------------------------------------------------------
// Tally: count[v] += #decisions equal to v.  Lanes of a warp that hold the same variant
// are merged into one atomic (hot variants take most of a hot task's queries).
// ------------------------------------------------------------------------------------
__device__ __forceinline__ void tally_one(uint32_t d, bool live, uint32_t n_variants,
                                          uint32_t *count_by_id, uint32_t &n_feas,
                                          uint32_t &n_nofeas, uint32_t &n_inval) {
  bool feas = live && d < n_variants && !(d & INFAAS_NO_FEASIBLE);
  bool inval = live && !feas && (d == INFAAS_INVALID || !(d & INFAAS_NO_FEASIBLE));
  bool nofeas = live && !feas && !inval;
  n_feas += feas;
  n_nofeas += nofeas;
  n_inval += inval;
  unsigned fm = __ballot_sync(0xFFFFFFFFu, feas);
  if (feas) {
    unsigned peers = __match_any_sync(fm, d);
    int leader = __ffs(peers) - 1;
    if ((threadIdx.x & 31) == leader) atomicAdd(&count_by_id[d], (uint32_t)__popc(peers));
  }
}

__global__ void __launch_bounds__(256)
tally_kernel(const uint32_t *decision, uint64_t n, uint32_t n_variants,
             uint32_t *count_by_id, unsigned long long *counters) {
  __shared__ uint32_t blk[3];
  if (threadIdx.x < 3) blk[threadIdx.x] = 0;
  __syncthreads();
  chain_wait();
  chain_next();
  uint32_t n_feas = 0, n_nofeas = 0, n_inval = 0;
  const uint64_t n4 = n >> 2;
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  const uint4 *dec4 = reinterpret_cast<const uint4 *>(decision);
  // whole warps iterate together so that the warp-wide intrinsics see all 32 lanes
  const uint64_t n4_warp = (n4 + 31) & ~(uint64_t)31;
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n4_warp; i += stride) {
    bool live = i < n4;
    uint4 d = live ? dec4[i] : make_uint4(0, 0, 0, 0);
    tally_one(d.x, live, n_variants, count_by_id, n_feas, n_nofeas, n_inval);
    tally_one(d.y, live, n_variants, count_by_id, n_feas, n_nofeas, n_inval);
    tally_one(d.z, live, n_variants, count_by_id, n_feas, n_nofeas, n_inval);
    tally_one(d.w, live, n_variants, count_by_id, n_feas, n_nofeas, n_inval);
  }
  if (blockIdx.x == 0 && threadIdx.x < 32) {  // ragged tail, at most 3 elements
    uint64_t i = (n4 << 2) + threadIdx.x;
    bool live = i < n;
    uint32_t d = live ? decision[i] : 0;
    tally_one(d, live, n_variants, count_by_id, n_feas, n_nofeas, n_inval);
  }
  n_feas = __reduce_add_sync(0xFFFFFFFFu, n_feas);
  n_nofeas = __reduce_add_sync(0xFFFFFFFFu, n_nofeas);
  n_inval = __reduce_add_sync(0xFFFFFFFFu, n_inval);
  if ((threadIdx.x & 31) == 0) {
    atomicAdd(&blk[0], n_feas);
    atomicAdd(&blk[1], n_nofeas);
    atomicAdd(&blk[2], n_inval);
  }
  __syncthreads();
  if (threadIdx.x < 3 && blk[threadIdx.x]) atomicAdd(&counters[threadIdx.x], (unsigned long long)blk[threadIdx.x]);
}

// Same tallies with a private histogram per CTA in shared memory (one u32 bin per variant):
// shared-memory atomics absorb the hot variants, and each CTA adds only its non-zero bins
// to the global counts at the end.  Used when the batch is large.  If the bins of all
// variants do not fit, the ids are split into `parts` ranges of `bins` ids: CTA b counts
// range b % parts over the share b / parts of the decisions (every range sees all
// decisions); the counters come from range 0 alone.
constexpr int TALLY_SMEM_THREADS = 1024;

__global__ void __launch_bounds__(TALLY_SMEM_THREADS)
tally_smem_kernel(const uint32_t *decision, uint64_t n, uint32_t n_variants, uint32_t bins,
                  uint32_t parts, uint32_t *count_by_id,
                  unsigned long long *counters) {
  extern __shared__ uint32_t hist[];
  __shared__ uint32_t blk[3];
  const uint32_t part = blockIdx.x % parts, lo = part * bins, share = blockIdx.x / parts;
  const uint32_t my_bins = min(bins, n_variants - lo);
  const uint32_t spare = my_bins + (threadIdx.x & 31u);
  for (uint32_t i = threadIdx.x; i < my_bins; i += blockDim.x) hist[i] = 0;
  if (threadIdx.x < 3) blk[threadIdx.x] = 0;
  __syncthreads();
  chain_wait();
  chain_next();
  // per decision: one shared-memory atomic and two counters; invalid
  // decisions are what remains of the total
  uint32_t n_feas = 0, n_nofeas = 0, n_seen = 0;
  auto one = [&](uint32_t d) {
    // no branch: what is not in this CTA's range (ids below lo wrap around) lands in one of 32
    // spare bins, one per lane, that nobody reads
    atomicAdd(&hist[min(d - lo, spare)], 1u);
    n_feas += d < n_variants;                                    // d < n_variants < 2^31: bit 31 clear
    n_nofeas += (d - INFAAS_NO_FEASIBLE) < 0x7FFFFFFFu;          // bit 31 set and not INFAAS_INVALID
  };
  const uint32_t n4 = (uint32_t)(n >> 2);                        // n <= 2^32 - 1 (checked by the caller)
  const uint32_t stride = (gridDim.x / parts) * blockDim.x;
  const uint4 *dec4 = reinterpret_cast<const uint4 *>(decision);
  // four 128-bit loads in flight per thread
  uint32_t i = share * blockDim.x + threadIdx.x;
  for (; n4 >= 3 * stride && i < n4 - 3 * stride; i += 4 * stride) {
    const uint4 d0 = load_once(dec4 + i), d1 = load_once(dec4 + i + stride);
    const uint4 d2 = load_once(dec4 + i + 2 * stride), d3 = load_once(dec4 + i + 3 * stride);
    one(d0.x); one(d0.y); one(d0.z); one(d0.w);
    one(d1.x); one(d1.y); one(d1.z); one(d1.w);
    one(d2.x); one(d2.y); one(d2.z); one(d2.w);
    one(d3.x); one(d3.y); one(d3.z); one(d3.w);
    n_seen += 16;
  }
  for (; i < n4; i += stride) {
    const uint4 d = load_once(dec4 + i);
    one(d.x); one(d.y); one(d.z); one(d.w);
    n_seen += 4;
  }
  if (share == 0 && threadIdx.x < (n & 3)) { one(decision[((uint64_t)n4 << 2) + threadIdx.x]); ++n_seen; }
  uint32_t n_inval = n_seen - n_feas - n_nofeas;
  n_feas = __reduce_add_sync(0xFFFFFFFFu, n_feas);
  n_nofeas = __reduce_add_sync(0xFFFFFFFFu, n_nofeas);
  n_inval = __reduce_add_sync(0xFFFFFFFFu, n_inval);
  if ((threadIdx.x & 31) == 0 && part == 0) {
    atomicAdd(&blk[0], n_feas);
    atomicAdd(&blk[1], n_nofeas);
    atomicAdd(&blk[2], n_inval);
  }
  __syncthreads();
  for (uint32_t i = threadIdx.x; i < my_bins; i += blockDim.x) {
    const uint32_t h = hist[i];
    if (h) atomicAdd(&count_by_id[lo + i], h);
  }
  if (threadIdx.x < 3 && blk[threadIdx.x]) atomicAdd(&counters[threadIdx.x], (unsigned long long)blk[threadIdx.x]);
}

}  // namespace

constexpr uint32_t TALLY_SMEM_MAX_VARIANTS = 49152;   // 192 KB of bins
constexpr uint32_t TALLY_SMEM_MAX_PARTS = 8;           // beyond this many id ranges: global atomics
constexpr size_t TALLY_SMEM_ALONE = 116 * 1024;
// Below this size the clear and flush passes over the bins cost more than the shared-memory atomics
// save.  Selection and load update with the shared-memory / the global tally, us: 528 variants, 65,536 queries
// 13.9 / 17.6, 98,000: 13.9 / 20.2; 6,000 variants, 65,536: 16.2 / 15.3, 131,072: 17.2 / 21.2; 16,384 variants,
// 98,000: 16.5 / 15.1, 160,000: 18.7 / 23.6; 65,536 variants, 131,072: 19.0 / 17.5, 200,000: 19.8 / 24.1.
inline uint64_t tally_smem_min_n(uint32_t n_variants) {
  const uint64_t n = 65536 + 10ull * n_variants;
  return n < 163840 ? n : 163840;
}

cudaError_t launch_tally(const DeviceCatalog &c, const uint32_t *d_decision, uint64_t n,
                         int sm_count, cudaStream_t stream) {
  if (n == 0) return cudaSuccess;
  const uint32_t parts = (c.n_variants + TALLY_SMEM_MAX_VARIANTS - 1) / TALLY_SMEM_MAX_VARIANTS;
  if (n >= tally_smem_min_n(c.n_variants) && parts <= TALLY_SMEM_MAX_PARTS) {
    const uint32_t bins = ((c.n_variants + parts - 1) / parts + 3u) & ~3u;
    size_t smem = (size_t)(bins + 32) * 4;                       // 32 spare bins
    // more than half of an SM's shared memory: launched while the selection kernel drains, two CTAs
    // on the SMs that finish first would leave others idle (+5 us on 2^24 decisions)
    if (smem < TALLY_SMEM_ALONE) smem = TALLY_SMEM_ALONE;
    // one CTA of 1024 threads per SM: half as many histograms to clear and flush as two of 512
    uint64_t want = ((n >> 2) + TALLY_SMEM_THREADS * 8 - 1) / (TALLY_SMEM_THREADS * 8);
    uint64_t shares = (uint64_t)sm_count / parts;              // CTAs per id range
    if (shares > want) shares = want;
    if (shares < 1) shares = 1;
    return launch_chained(tally_smem_kernel, (uint32_t)(shares * parts), TALLY_SMEM_THREADS, smem, SPLIT_DRIVER, stream, d_decision, n,
                          c.n_variants, bins, parts, c.count_by_id, c.counters);
  }
  uint64_t want = ((n >> 2) + 255) / 256;
  const uint64_t most = (uint64_t)sm_count * 8;
  uint32_t grid = (uint32_t)(want < 1 ? 1 : (want > most ? most : want));
  return launch_chained(tally_kernel, grid, 256, 0, split_for(c), stream, d_decision, n, c.n_variants, c.count_by_id, c.counters);
}

cudaError_t prepare_tally_kernel() {
  return cudaFuncSetAttribute(tally_smem_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)((TALLY_SMEM_MAX_VARIANTS + 32) * 4));
}

}  // namespace infaas
