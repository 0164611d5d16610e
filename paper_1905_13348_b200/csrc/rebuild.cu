// Queue recursion, predicted latency and the per-task scan lists with their rank index.
//
// Section 4 of the paper says a loaded variant's latency is not its profiled one.  Here each
// variant's queue is advanced by one window of tallied decisions, its load-adjusted latency is
// recomputed, and every task's list of non-dominated variants is rebuilt in (cost, pred_lat,
// -acc, id) order (rebuild kernel).  On a state-aware catalog the same step moves the variants'
// life-cycle states with the load (Section 4, state machine) and builds the Active and the
// Inactive list of every task.
#include "common.cuh"

namespace infaas {

namespace {

constexpr uint32_t NONE = 0xFFFFFFFFu;
constexpr uint32_t REBUILD_THREADS = 1024;
constexpr uint32_t REBUILD_WARPS = REBUILD_THREADS / 32;

// The code of a latency or SLO: the IEEE-754 pattern of x converted to float toward zero, monotone and
// roughly logarithmic; the selection kernel derives the same bucket from it.
__device__ __forceinline__ uint32_t float_bits(uint32_t x) { return __float_as_uint(__uint2float_rz(x)); }
// Smallest u32 whose code is >= pattern (2^32 - 1 for patterns of 2^32 and above).
__device__ __forceinline__ uint32_t float_bits_floor(uint32_t pattern) {
  return __float2uint_ru(__uint_as_float(pattern));
}
constexpr uint32_t BITS_OF_2_POW_32 = 0x4F800000u;

constexpr uint32_t GRID_PITCH = GRID + 1;   // one word of padding per row of the prune's grid

// Shared memory of a CTA of B threads while it builds the index of one list segment; NB: SLO buckets.
template <uint32_t B, uint32_t NB>
struct IndexScratch {
  uint32_t pred[256], ids[256];     // the segment in scan order; latencies behind its end are NONE
  uint32_t sorted[256];             // its latencies ascending (equal ones in scan order)
  uint32_t ent[256];                // same order: accuracy rank << 24 | latency rank << 16 | last of its latency << 8 | position
  uint32_t Pd[256];                 // distinct latencies
  uint32_t bcnt[NB];                // how many of them per SLO bucket
  uint32_t wbits[MAX_ACC_WORDS];    // per bitmap word: the accuracies present
  // per latency rank: the most accurate entry (acc << 16 | 0xFFFF - position, 0 = none); per
  // accuracy rank: the fastest entry (its index in latency order, NONE = none)
  uint32_t rankA[256], rankB[256];
  uint16_t acc[256];
  unsigned char wpre[MAX_ACC_WORDS];         // accuracies present in the words before
  unsigned char at[256];                     // sorted order: position
  unsigned char stair[256];                  // latency rank holds a stair entry
  unsigned char part[B];                     // rank table: first position per column of a run of entries
  uint32_t warp_bcnt[B / 32u];               // latencies in the SLO buckets of a warp
  uint32_t ks, ka, base;

  // Entry `pos` of the segment (its accuracy's bit too).
  __device__ __forceinline__ void put(uint32_t pos, uint32_t latency, uint32_t accuracy, uint32_t id, uint32_t acc_lo) {
    ids[pos] = id; pred[pos] = latency; acc[pos] = (uint16_t)accuracy;
    const uint32_t x = accuracy - acc_lo, xw = x / ACC_WORD_BITS;
    atomicOr(&wbits[xw], 1u << (x - xw * ACC_WORD_BITS));
  }
  // Clears what is accumulated into (all threads; a barrier must follow).
  __device__ __forceinline__ void clear(uint32_t n_buckets, uint32_t nbw) {
#pragma unroll 1
    for (uint32_t i = threadIdx.x; i < 256u; i += B) { pred[i] = NONE; rankA[i] = 0u; rankB[i] = NONE; }
#pragma unroll 1
    for (uint32_t i = threadIdx.x; i < n_buckets; i += B) bcnt[i] = 0u;
#pragma unroll 1
    for (uint32_t i = threadIdx.x; i < nbw; i += B) wbits[i] = 0u;
  }
};

// Fixed part of the image for a task without index (also entry n_tasks): a header word,
// records and a bitmap that make every query of the task read "none".  All threads.
__device__ __forceinline__ void write_dummy_task(const DeviceCatalog &c, uint32_t t) {
  const uint32_t T = c.n_tasks;
  if (threadIdx.x == 0) reinterpret_cast<uint32_t *>(c.image + IMAGE_HDR_OFFSET)[t] = DUMMY_HEADER;
  uint32_t *rec = reinterpret_cast<uint32_t *>(c.image + image_rec_offset(T) + t * rec_stride(c.n_buckets));
#pragma unroll 1
  for (uint32_t j = threadIdx.x; j <= c.n_buckets; j += blockDim.x) rec[j] = 0u;
  uint32_t *bm = reinterpret_cast<uint32_t *>(c.image + image_bitmap_offset(T, c.n_buckets) + t * bitmap_stride(c.nbw));
#pragma unroll 1
  for (uint32_t j = threadIdx.x; j < c.nbw; j += blockDim.x) bm[j] = 0u;
}

// Bucket scale of the SLO records: S (16..23) and bmin such that n_buckets - 1 buckets of
// 2^S float patterns cover everything from the catalog's smallest profiled latency up to the
// largest SLO asked for so far (as a bit mask: every SLO seen is <= cap).
__device__ __forceinline__ void bucket_scale(const DeviceCatalog &c, uint32_t slo_seen, uint32_t &Sh, uint32_t &bmin) {
  uint32_t cap = slo_seen | SLO_CAP_FLOOR_US;
  cap |= cap >> 1; cap |= cap >> 2; cap |= cap >> 4; cap |= cap >> 8; cap |= cap >> 16;
  const uint32_t clo = c.lat_code_lo;
  const uint32_t chi = max(clo, __float_as_uint(__uint2float_rz(cap)) >> 16);
  // (a distance of 2^k spans at least 2^(k - sh) buckets: more than n_buckets below this start)
  const int start = 31 - (int)__clz((chi - clo) | 1u) - (31 - (int)__clz(c.n_buckets));
  uint32_t sh = (uint32_t)max(start, 0);
#pragma unroll 1
  while ((chi >> sh) - (clo >> sh) > c.n_buckets - 2u) ++sh;
  bmin = clo >> sh;
  Sh = 16u + sh;
}

// Inclusive scans over the lanes of a warp.
__device__ __forceinline__ uint32_t warp_scan_add(uint32_t x) {
  const uint32_t lane = threadIdx.x & 31u;
#pragma unroll
  for (uint32_t o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, x, o);
    if (lane >= o) x += y;
  }
  return x;
}
// (shfl_up leaves the lanes without a source unchanged: minimum and maximum need no guard)
template <class T>
__device__ __forceinline__ T warp_scan_min(T x) {
#pragma unroll
  for (uint32_t o = 1; o < 32; o <<= 1) x = min(x, __shfl_up_sync(0xFFFFFFFFu, x, o));
  return x;
}
__device__ __forceinline__ uint32_t warp_scan_max(uint32_t x) {
#pragma unroll
  for (uint32_t o = 1; o < 32; o <<= 1) x = max(x, __shfl_up_sync(0xFFFFFFFFu, x, o));
  return x;
}
// Exclusive: the lanes before this one (`none` in lane 0).
__device__ __forceinline__ uint32_t lanes_before(uint32_t incl, uint32_t none) {
  const uint32_t up = __shfl_up_sync(0xFFFFFFFFu, incl, 1);
  return threadIdx.x & 31u ? up : none;
}

// One atomic per allocation places a block in the image and, on a CTA's last allocation
// (`done`), counts the CTA as finished with the cursor.  The CTA that is counted last knows the
// final image size: it publishes it for the kernels that follow and clears the counter for the
// next rebuild.  One thread only, in two halves so that the atomic's round trip can overlap other
// work: place_block_issue returns the counter's old value, place_block_finish (same arguments)
// the block's offset behind the fixed part of the image.
__device__ __forceinline__ unsigned long long place_block_issue(const DeviceCatalog &c, uint32_t bytes, bool done) {
  return atomicAdd(c.alloc_ctr, ((unsigned long long)(done ? 1u : 0u) << 32) | bytes);
}
__device__ __forceinline__ uint32_t place_block_finish(const DeviceCatalog &c, unsigned long long old,
                                                       uint32_t bytes, bool done) {
  if (done && (uint32_t)(old >> 32) == gridDim.x - 1u) {
    c.image_hdr[0] = image_var_offset(c.n_tasks, c.n_buckets, c.nbw) + (uint32_t)old + bytes;
    *c.alloc_ctr = 0ull;
  }
  return (uint32_t)old;
}

// Builds the exact index of a list segment of F <= INDEX_MAX_F entries (layout in common.cuh) into
// a block of the image obtained from the block cursor.  S holds the segment in scan order (S.put), the
// other accumulators are clear.  Returns false (all threads) if it cannot be indexed: its block lies
// beyond the image's capacity or beyond what the header's offset field addresses.
// `xi`: NONE for the task's first segment (header word, SLO records and bitmap go into the
// fixed part of the image), else the index of this further segment (header to xhdr[xi], bitmap
// into the block, no records: only the slow path comes here).  `next`: 1 + index of the task's
// next segment, 0 if this is the last.  `done`: the CTA's last allocation.
//
// The chain is bound by latency (barriers and shared-memory round trips) and by the instructions of
// the warps that have nothing to do in a step, so it has few steps (three barriers inside), no
// division, and the block's place is asked for as early as its size is known (one atomic that all
// CTAs send to the same word: 0.4 us): one pair loop (latency order), accuracy ranks straight from the
// bitmap, and the rank table as a running minimum down its columns -- F steps per column, cut into
// runs of entries so that all warps work, instead of F bits per cell.
template <uint32_t B, uint32_t NB>
__device__ __forceinline__ bool build_index(const DeviceCatalog &c, uint32_t t, uint32_t F, IndexScratch<B, NB> &S,
                                            uint32_t xi, uint32_t next, bool done, uint32_t Sh, uint32_t bmin) {
  constexpr uint32_t WARPS = B / 32u;
  static_assert(B >= 256u && INDEX_MAX_F < 254u, "one thread per entry");
  const uint32_t tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5;
  const bool first = xi == NONE;
  const uint32_t acc_lo = c.acc_lo, nbw = c.nbw;      // the catalog's accuracy window

  // 1. latency order: entry p comes behind the entries before it in the list that are not slower and
  // those after it that are faster (latencies are at least 1).  1 << ls lanes per entry, 4 entries per load
  uint32_t ls = 3;
  while (ls && (F << ls) > B) --ls;
  if ((32u * warp) >> ls < F) {
    const uint32_t p = tid >> ls, sub = tid & ((1u << ls) - 1u), mine = min(p, F - 1u), own = mine & ~3u;
    const uint32_t pp = S.pred[mine];
    uint32_t cnt = 0;
#pragma unroll 4
    for (uint32_t q = 4u * sub; q < F; q += 4u << ls) {
      const uint4 v = *reinterpret_cast<const uint4 *>(&S.pred[q]);
      const uint32_t lim = pp - (uint32_t)(q >= own);
      cnt += (uint32_t)(v.x <= lim) + (uint32_t)(v.y <= lim) + (uint32_t)(v.z <= lim) + (uint32_t)(v.w <= lim);
    }
    if (sub == 0u) {                                   // equal latencies in front of p inside its own four
      const uint4 v = *reinterpret_cast<const uint4 *>(&S.pred[own]);
      const uint32_t e = mine & 3u;
      cnt += (uint32_t)(e > 0u && v.x == pp) + (uint32_t)(e > 1u && v.y == pp) + (uint32_t)(e > 2u && v.z == pp);
    }
    __syncwarp();
#pragma unroll 1
    for (uint32_t o = 1u; o < (1u << ls); o <<= 1) cnt += __shfl_xor_sync(0xFFFFFFFFu, cnt, o);
    if (p < F && sub == 0u) {
      S.sorted[cnt] = pp;
      S.at[cnt] = (unsigned char)p;
    }
  }
  // running popcounts of the accuracy bitmap, one word per thread (the last warps first: they have no
  // entries); the bitmap itself, where its place is fixed
  uint32_t *bitmap = reinterpret_cast<uint32_t *>(c.image + image_bitmap_offset(c.n_tasks, c.n_buckets) + t * bitmap_stride(nbw));
#pragma unroll 1
  for (uint32_t w0 = 32u * (WARPS - 1u - warp); w0 < nbw; w0 += B) {           // uniform per warp
    uint32_t below = 0;
#pragma unroll 4
    for (uint32_t x = lane; x < w0; x += 32u) below += __popc(S.wbits[x]);
    below = __reduce_add_sync(0xFFFFFFFFu, below);
    const uint32_t w = w0 + lane, bits = w < nbw ? S.wbits[w] : 0u, pc = __popc(bits);
    const uint32_t incl = below + warp_scan_add(pc);
    if (w < nbw) {
      S.wpre[w] = (unsigned char)(incl - pc);
      if (first) bitmap[w] = ((incl - pc) << 24) | bits;
    }
    if (w == nbw - 1u) S.ka = incl;
  }
  __syncthreads();

  // 2. the block's place in the image (the atomic is in flight until step 3 ends): its size needs the number of
  // distinct latencies, which the last warp counts for itself, a barrier before the others know; dense
  // latency ranks, accuracy ranks and the best entry per rank, one sorted entry per thread
  const uint32_t Ka = S.ka, width = Ka + 1u;
  unsigned long long placed = 0;
  uint32_t bytes = 0;
  if (warp == WARPS - 1u) {
    uint32_t distinct = 0;
#pragma unroll 4
    for (uint32_t x = lane; x < F; x += 32u) distinct += (uint32_t)(x == 0u || S.sorted[x] != S.sorted[x - 1u]);
    distinct = __reduce_add_sync(0xFFFFFFFFu, distinct);
    bytes = block_layout(F, distinct, Ka, first ? 0u : nbw).bytes;
    if (lane == 31u) {
      placed = place_block_issue(c, bytes, done);
      S.ks = distinct;
    }
  }
  if (32u * warp < F) {
    const uint32_t i = tid;
    uint32_t before = 0;
#pragma unroll 1
    for (uint32_t x = lane; x < 32u * warp; x += 32u)
      before += __popc(__ballot_sync(0xFFFFFFFFu, x == 0u || S.sorted[x] != S.sorted[x - 1u]));
    const uint32_t v = S.sorted[i];                                                 // (behind F: not used)
    const bool fresh = i < F && (i == 0u || v != S.sorted[i - 1u]);
    const unsigned m = __ballot_sync(0xFFFFFFFFu, fresh);
    if (i < F) {
      const uint32_t r = before + __popc(m & ((2u << lane) - 1u)) - 1u;
      const uint32_t last = i == F - 1u || v != S.sorted[i + 1u];
      if (fresh) {
        S.Pd[r] = v;
        // larger latencies than the largest SLO asked for so far share the last bucket
        atomicAdd(&S.bcnt[min(max(float_bits(v) >> Sh, bmin) - bmin, c.n_buckets - 1u)], 1u);
      }
      const uint32_t p = S.at[i], acc = S.acc[p], x = acc - acc_lo, xw = x / ACC_WORD_BITS;
      const uint32_t ra = S.wpre[xw] + __popc(S.wbits[xw] & ((1u << (x - xw * ACC_WORD_BITS)) - 1u));
      S.ent[i] = (ra << 24) | (r << 16) | (last << 8) | p;
      atomicMax(&S.rankA[r], (acc << 16) | (0xFFFFu - p));                          // most accurate, first position
      atomicMin(&S.rankB[ra], i);                                                   // fastest, first position
    }
  }
  __syncthreads();
  const uint32_t Ks = S.ks;
  const BlockLayout BL = block_layout(F, Ks, Ka, first ? 0u : nbw);
  const SlowLayout SL = slow_layout(F, Ks, Ka);

  // 3. rank table, first half.  T2[r][k] = smallest position among the entries whose latency rank
  // is < r and whose accuracy rank is >= k: a running minimum over the entries in latency order.
  // A thread takes one column and one run of entries: here the run's minimum.
  const uint32_t cols = (width + 31u) >> 5, lc = cols > 1u ? 32u - __clz(cols - 1u) : 0u;   // warps side by side: 1 << lc
  constexpr uint32_t LOG_WARPS = B == 256u ? 3u : B == 512u ? 4u : 5u;
  static_assert(WARPS == 1u << LOG_WARPS, "log2 of the warps");
  const uint32_t runs = WARPS >> lc, run_len = max(8u, (((F + runs - 1u) >> (LOG_WARPS - lc)) + 3u) & ~3u);
  const uint32_t run = warp >> lc, colw = warp & ((1u << lc) - 1u), col = colw * 32u + lane;
  const uint32_t i0 = min(F, run * run_len), i1 = colw < cols ? min(F, i0 + run_len) : i0;
  const uint32_t col_key = col << 24;
  if (i0 < i1 && i1 < F) {
    uint32_t v = 0xFFu;
#pragma unroll 4
    for (uint32_t i = i0; i < i1; ++i) {
      const uint32_t e = S.ent[i];
      if (e >= col_key) v = min(v, e & 0xFFu);
    }
    S.part[tid] = (unsigned char)v;
  }
  // stair entries: those more accurate than everything faster (one per latency at most); 32 latency
  // ranks per warp
  const uint32_t ws = (warp + WARPS / 2u) & (WARPS - 1u);         // (not the warps with a run)
  uint32_t best_a = 0;                                            // latency ranks < this thread's
  if (32u * ws <= Ks) {
    const uint32_t r = 32u * ws + lane;
    uint32_t below = 0;
#pragma unroll 1
    for (uint32_t i = lane; i < 32u * ws; i += 32u) below = max(below, S.rankA[i]);
    below = __reduce_max_sync(0xFFFFFFFFu, below);
    const uint32_t x = r < Ks ? S.rankA[r] : 0u;
    best_a = max(below, lanes_before(warp_scan_max(x), 0u));
    if (r < Ks) S.stair[r] = best_a == 0u || (x >> 16) > (best_a >> 16);
  }
  // SLO records, first half: latencies in the buckets before this thread's (`per` consecutive ones) in its warp;
  // the warps' sums are added behind the barrier (each warp adding up all buckets before its own took 10 us of
  // the 16 windows of 128 x 512, more with 2048 buckets)
  constexpr uint32_t PER = NB > B ? NB / B : 1u;
  const uint32_t nb = c.n_buckets, per = nb > B ? PER : 1u, j0 = tid * per;
  uint32_t below = 0;
  if (first && 32u * warp * per < nb) {
    uint32_t n = S.bcnt[j0];
    if (PER > 1u && per > 1u)
#pragma unroll
      for (uint32_t k = 1; k < PER; ++k) n += S.bcnt[j0 + k];
    const uint32_t incl = warp_scan_add(n);
    below = incl - n;
    if (lane == 31u) S.warp_bcnt[warp] = incl;
  }
  if (tid == B - 1u) {
    uint32_t base = image_var_offset(c.n_tasks, c.n_buckets, nbw) + place_block_finish(c, placed, bytes, done);
    if (base + bytes > c.image_capacity || base + BL.t2 >= IMAGE_T2_LIMIT) base = NONE;
    S.base = base;
  }
  __syncthreads();
  const uint32_t base = S.base;
  if (base == NONE) return false;
  unsigned char *blk = c.image + base;
  unsigned char *slow = blk + BL.slow;

  // 4. SLO records, second half
  if (first && 32u * warp * per < nb) {
    below += __reduce_add_sync(0xFFFFFFFFu, lane < warp ? S.warp_bcnt[lane] : 0u);
    uint32_t *rec = reinterpret_cast<uint32_t *>(c.image + image_rec_offset(c.n_tasks) + t * rec_stride(nb));
#pragma unroll 1
    for (uint32_t j = j0; j < j0 + per; ++j) {
      const uint32_t cnt = S.bcnt[j];
      uint32_t r = ((Ks + 1u) << 24) | (cnt << 8) | below;          // exact slow path
      if (cnt == 0u) {
        r = below << 24;
      } else if (cnt == 1u) {
        const uint32_t lo = j ? float_bits_floor((bmin + j) << Sh) : 0u;
        const uint32_t nxt = (bmin + j + 1u) << Sh;
        const uint32_t hi = (j == nb - 1u || nxt >= BITS_OF_2_POW_32) ? NONE : float_bits_floor(nxt) - 1u;
        const uint32_t thr = S.Pd[below];
        if ((lo >> 24) == (hi >> 24))
          r = thr <= lo ? (below + 1u) << 24 : (below << 24) | (0x00FFFFFFu - ((thr - 1u) & 0x00FFFFFFu));
      }
      rec[j] = r;
      if (j == nb - 1u) rec[nb] = r;                               // what an SLO beyond the last bucket reads
      below += cnt;
    }
  }
  // rank table, second half: each run starts from the minimum of the runs before it and writes a
  // row after the last entry of every latency
  unsigned char *T2 = blk + BL.t2;
  if (i0 < i1 && col < width) {
    uint32_t v = F;
#pragma unroll 4
    for (uint32_t w = 0; w < run; ++w) v = min(v, (uint32_t)S.part[(((w << lc) + colw) << 5) + lane]);
    if (run == 0u) T2[col] = (unsigned char)F;                   // nothing is fast enough
    unsigned char *row = T2 + (((S.ent[i0] >> 16) & 0xFFu) + 1u) * width + col;
#pragma unroll 4
    for (uint32_t i = i0; i < i1; ++i) {
      const uint32_t e = S.ent[i];
      if (e >= col_key) v = min(v, e & 0xFFu);
      if (e & 0x100u) { *row = (unsigned char)v; row += width; }
    }
    if (i1 == F) { row[0] = (unsigned char)F; row[width] = (unsigned char)F; }   // rows Ks + 1, Ks + 2: the slow path's
  }

  // the small tables.  What the nearest-miss search reads: bestA[r] over latency ranks < r, the stair
  // entries in ascending latency, ordStart[r] = stair entries with latency rank < r (the warps of step
  // 3); position 0xFF stands for "none"
  if (32u * ws <= Ks) {
    const uint32_t r = 32u * ws + lane;
    uint32_t before = 0;
#pragma unroll 1
    for (uint32_t i = lane; i < 32u * ws; i += 32u) before += __popc(__ballot_sync(0xFFFFFFFFu, S.stair[i]));
    const bool st = r < Ks && S.stair[r];
    const uint32_t o = before + __popc(__ballot_sync(0xFFFFFFFFu, st) & ((1u << lane) - 1u));
    if (r <= Ks) {
      reinterpret_cast<uint32_t *>(slow + SL.bestA)[r] =
          best_a ? (best_a >> 16) | ((0xFFFFu - (best_a & 0xFFFFu)) << 16) : 0xFFu << 16;
      slow[SL.ordStart + r] = (unsigned char)o;
    }
    if (st) {
      const uint32_t a = S.rankA[r];
      reinterpret_cast<uint2 *>(slow + SL.walk)[o] = make_uint2(S.Pd[r], (a >> 16) | ((0xFFFFu - (a & 0xFFFFu)) << 16));
    }
    if (r == Ks)
      c.slow[first ? t : c.n_tasks + xi] = make_uint4(base + BL.slow, F | (Ks << 8) | (Ka << 16), 0u, o | (next << 8));
  }
  // bestB[k] over accuracy ranks >= k, 32 ranks from the top down per warp
  const uint32_t wb = (warp + WARPS / 2u) & (WARPS - 1u);
  if (32u * wb <= Ka) {
    const uint32_t q0 = 32u * wb, q = q0 + lane;                  // q-th value of bestB from the top; bestB[Ka] is none
    uint32_t above = NONE;
#pragma unroll 1
    for (uint32_t i = lane; i < q0; i += 32u) above = min(above, S.rankB[Ka - 1u - i]);
    above = __reduce_min_sync(0xFFFFFFFFu, above);
    const uint32_t i = min(above, lanes_before(warp_scan_min(q < Ka ? S.rankB[Ka - 1u - q] : NONE), NONE));
    if (q <= Ka)
      reinterpret_cast<uint2 *>(slow + SL.bestB)[Ka - q] = i == NONE ? make_uint2(0u, 0xFFu) : make_uint2(S.sorted[i], S.at[i]);
  }
  uint32_t *ids_end = reinterpret_cast<uint32_t *>(blk + BL.t2);   // ids, reversed; slot F holds PENDING
  const uint32_t p = (tid + 256u) & (B - 1u);                      // (the last 256 threads)
  if (p <= F) ids_end[-1 - (int)p] = p < F ? S.ids[p] : PENDING;
  if (p < Ks) reinterpret_cast<uint32_t *>(slow + SL.Pd)[p] = S.Pd[p];
  if (!first)
#pragma unroll 1
    for (uint32_t w = tid; w < nbw; w += B) reinterpret_cast<uint32_t *>(blk + BL.bitmap)[w] = ((uint32_t)S.wpre[w] << 24) | S.wbits[w];
  if (tid == 0u) {
    if (first) reinterpret_cast<uint32_t *>(c.image + IMAGE_HDR_OFFSET)[t] = (base + BL.t2) | (width << 24);
    else c.xhdr[xi] = make_uint4(base + BL.t2, width, base + BL.bitmap, 0u);
  }
  return true;
}

// What the queue recursion reads of one variant.
struct Row {
  uint32_t lat, batch, queued, id, order, count, state, load_lat, drain;
  unsigned long long served;
};
// ... what no kernel writes
__device__ __forceinline__ Row load_fixed(const DeviceCatalog &c, uint32_t slot, uint32_t window_us) {
  Row r;
  r.lat = c.s_lat[slot];
  r.batch = c.s_batch[slot];
  r.order = c.s_order[slot];
  r.id = c.s_id[slot];
  const unsigned long long drain = (unsigned long long)window_us * r.batch / r.lat;   // queries served per window
  r.drain = drain > NONE ? NONE : (uint32_t)drain;
  return r;
}
// ... and the rest
__device__ __forceinline__ void load_load(const DeviceCatalog &c, uint32_t slot, bool advance, Row &r) {
  r.queued = c.s_queued[slot];
  r.count = 0; r.served = 0; r.state = INFAAS_STATE_ACTIVE; r.load_lat = 0;
  if (c.stateful) { r.state = c.s_state[slot]; r.load_lat = c.s_load_lat[slot]; }
  if (advance) {
    r.count = c.count_by_id[r.id];
    r.served = c.s_served[slot];
  }
}
// Queue recursion and states; returns the predicted latency and leaves the new state in r.state.
__device__ __forceinline__ uint32_t advance_row(const DeviceCatalog &c, uint32_t slot, Row &r, bool advance) {
  uint32_t queued = r.queued;
  if (advance) {
    unsigned long long arrived = (unsigned long long)queued + r.count;
    if (arrived > NONE) arrived = NONE;
    queued = arrived > r.drain ? (uint32_t)arrived - r.drain : 0u;
    c.s_served[slot] = r.served + r.count;
    c.s_queued[slot] = queued;
    if (c.stateful) {
      // loaded by its first queries; at peak throughput while a backlog remains
      if (r.state == INFAAS_STATE_INACTIVE && r.count > 0) r.state = INFAAS_STATE_ACTIVE;
      if (r.state == INFAAS_STATE_ACTIVE || r.state == INFAAS_STATE_OVERLOADED)
        r.state = queued > 0 ? INFAAS_STATE_OVERLOADED : INFAAS_STATE_ACTIVE;
      c.s_state[slot] = (unsigned char)r.state;
    }
  }
  unsigned long long p = r.lat;
  if (queued) {                     // batch sizes are mostly powers of two
    const unsigned long long w = (unsigned long long)queued * r.lat;
    p += r.batch & (r.batch - 1u) ? w / r.batch : w >> (31 - __clz((int)r.batch));
  }
  const uint32_t pred = p > NONE ? NONE : (uint32_t)p;
  c.s_pred[slot] = pred;
  return pred;
}

// The same variable of CTA `rank` of this CTA's cluster.
template <class T>
__device__ __forceinline__ T *peer(T *p, uint32_t rank) {
  unsigned long long a;
  asm("mapa.u64 %0, %1, %2;" : "=l"(a) : "l"(p), "r"(rank));
  return reinterpret_cast<T *>(a);
}
// Barrier over the K CTAs of a task's cluster (all their threads), for shared and global memory.
__device__ __forceinline__ void task_sync(uint32_t K) {
  if (K > 1u) {
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  } else {
    __syncthreads();
  }
}

// Queue recursion, prune and list of one task, by the K CTAs of its cluster: the list goes into the
// task's region, segment s < K of it also into CTA s's S, which is cleared here.  Contains chain_wait.
// Returns the list's length.
//
// List of the Active variants (all variants of a catalog without states).  Slots are in (cost,
// 10000-acc, id) order, so with `order` = position in (10000-acc, local) order a variant q before
// p in both orders with pred_q <= pred_p dominates p, and the only other way to be dominated is a
// faster variant of the same cost and accuracy.  The two orders never change, only pred does, so
// nothing is sorted: pred is reduced into a grid of at most 64 x 64 cells (runs of local indices
// x runs of positions in accuracy order); after a running minimum along rows and columns, the cell
// diagonally before p's tells whether something in a strictly earlier row and column dominates it.
// What passes (a few more than survive) is compared with the entries of its own row and column
// only.  Survivors of equal cost are a staircase (later in accuracy order = faster), so list
// positions follow from counting survivors: those before the run of equal cost, then the run
// backwards.
//
// Each CTA has a share of the grid's rows, with their variants: the running minimum down the columns
// goes on from the last rows of the CTAs before it, what passes is made known to the CTAs behind it (by
// accuracy position), survivors to all.  4 x 4096 variants on a trade-off surface, lists of up to 505 entries: a window of
// 20,011 queries took 8 us longer with the list made by the first CTA alone.
//
// List of the Inactive variants: ordered by (eff, 10000-acc, id) with eff in place of cost and
// pred; at most the fastest variant (lowest id) of every distinct accuracy is on it, if it is
// faster than everything more accurate, and the list runs from the lowest accuracy up.  CTA 0 makes it.
__device__ __forceinline__ uint32_t build_list(const DeviceCatalog &c, uint32_t t, uint32_t share, uint32_t K, bool advance,
                                               uint32_t window_us, unsigned char *dyn,
                                               IndexScratch<REBUILD_THREADS, MAX_BUCKETS> &S, uint32_t &slo_seen) {
  constexpr uint32_t KEEP_WORDS = INFAAS_MAX_TASK_VARIANTS / 32;
  __shared__ uint32_t grid[GRID * GRID_PITCH];                    // this CTA's rows
  __shared__ uint32_t carry[GRID];                                // per column: smallest of the rows of the CTAs before
  __shared__ uint32_t keep[KEEP_WORDS + 1], keep_pre[KEEP_WORDS + 1];   // bit sets: survivors, by local index ...
  __shared__ uint32_t passed_local[KEEP_WORDS], passed_acc[KEEP_WORDS];   // ... what the grid lets through, both orders
  __shared__ unsigned long long warp_min[REBUILD_WARPS];
  __shared__ uint32_t warp_cnt[REBUILD_WARPS];
  __shared__ uint32_t n_cand, n_inactive;
  constexpr uint32_t B = REBUILD_THREADS;

  const uint32_t tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5;
  const uint32_t base = c.task_off[t], V = c.task_off[t + 1] - base;
  const TaskShare sh = task_share(V, K, share);
  const uint32_t cs = sh.cs, ng = sh.ng, rows = sh.rows, y0 = sh.y0, lo = sh.lo, hi = sh.hi;
  const uint32_t own = hi - lo, own_rows = (own + (1u << cs) - 1u) >> cs;
  // shared memory per variant (REBUILD_ROW_SMEM bytes); those by local index: of this CTA's, from lo
  uint2 *by_acc = reinterpret_cast<uint2 *>(dyn);                 // accuracy order: (pred, local), of what passed
  uint2 *by_local = by_acc + V;                                    // (pred, accuracy position); position 0xFFFF: not listed
  uint32_t *run_min = reinterpret_cast<uint32_t *>(by_local + V); // at the first of each (cost, accuracy): smallest pred
  uint16_t *cand = reinterpret_cast<uint16_t *>(run_min + V);     // entries the grid lets through
  auto run_min_of = [&](uint32_t order) {                         // (a run can begin in an earlier CTA's share)
    const uint32_t f = (order >> 13) & 0x1FFFu;
    if (f >= lo) return run_min + (f - lo);
    const uint32_t o = (f >> cs) / rows;
    return peer(run_min + (f - ((o * rows) << cs)), o);
  };

  unsigned char *region = c.regions + c.reg_off[t];
  unsigned long long *keys_g = reinterpret_cast<unsigned long long *>(region);
  uint32_t *ids_g = reinterpret_cast<uint32_t *>(region + 8u * V);

  // 1. queue recursion, states, predicted latencies; coarse grid.  Each thread's first variant
  // stays in registers.  Before chain_wait: only what no kernel writes, and clearing.
  const uint32_t own0 = lo + tid;
  Row r0;
  r0.drain = 0;
  uint32_t acc0 = 0, run0 = 0, class0 = 0, pred0 = 0;
  if (own0 < hi) {
    r0 = load_fixed(c, base + own0, window_us);
    acc0 = c.s_acc[base + own0];
    run0 = c.s_cost_run[base + own0];
    if (c.stateful) class0 = c.s_class[base + own0];
  }
#pragma unroll 1
  for (uint32_t i = tid; i < rows * GRID_PITCH; i += B) grid[i] = NONE;
#pragma unroll 1
  for (uint32_t i = tid; i < own; i += B) run_min[i] = NONE;
#pragma unroll 1
  for (uint32_t i = tid; i <= KEEP_WORDS; i += B) { keep[i] = 0u; if (i < KEEP_WORDS) passed_acc[i] = 0u; }
  S.clear(c.n_buckets, c.nbw);
  if (tid < GRID) carry[tid] = NONE;
  if (tid == 0u) { n_cand = 0u; n_inactive = 0u; }
  task_sync(K);
  asm volatile("" : "+r"(r0.drain));                               // (else the compiler moves the division behind the wait)
  chain_wait();
  chain_next();
  slo_seen = *c.slo_seen;                                          // wanted by the index, requested early
  Row r = r0;
#pragma unroll 1
  for (uint32_t i = own0; i < hi;) {
    load_load(c, base + i, advance, r);
    const uint32_t pred = advance_row(c, base + i, r, advance);
    const uint32_t pos = r.order & 0x1FFFu;
    const bool listed = r.state == INFAAS_STATE_ACTIVE;
    by_local[i - lo] = listed ? make_uint2(pred, pos) : make_uint2(NONE, 0xFFFFu);
    if (listed) {
      // NONE stands for "no entry" in the grid: a saturated latency counts as one less there
      atomicMin(&grid[((i >> cs) - y0) * GRID_PITCH + (pos >> cs)], min(pred, NONE - 1u));
      if (r.order >> 31) atomicMin(run_min_of(r.order), pred);
    }
    if (i == own0) { pred0 = pred; r0.state = r.state; r0.load_lat = r.load_lat; }
    i += B;
    if (i < hi) r = load_fixed(c, base + i, window_us);
  }
  __syncthreads();
  // 2. running minimum along the rows, then down the columns (GRID = two values per lane)
#pragma unroll 1
  for (uint32_t y = warp; y < own_rows; y += REBUILD_WARPS) {
    uint32_t *row = grid + y * GRID_PITCH;
    const uint32_t x0 = warp_scan_min(lane < ng ? row[lane] : NONE);
    if (lane < ng) row[lane] = x0;
    if (ng > 32u) {
      const uint32_t before = __shfl_sync(0xFFFFFFFFu, x0, 31);
      const uint32_t x1 = min(warp_scan_min(lane + 32u < ng ? row[lane + 32u] : NONE), before);
      if (lane + 32u < ng) row[lane + 32u] = x1;
    }
  }
  __syncthreads();
#pragma unroll 1
  for (uint32_t x = warp; x < ng; x += REBUILD_WARPS) {
    uint32_t *col = grid + x;
    const uint32_t x0 = warp_scan_min(lane < own_rows ? col[lane * GRID_PITCH] : NONE);
    if (lane < own_rows) col[lane * GRID_PITCH] = x0;
    if (own_rows > 32u) {
      const uint32_t before = __shfl_sync(0xFFFFFFFFu, x0, 31);
      const uint32_t x1 = min(warp_scan_min(lane + 32u < own_rows ? col[(lane + 32u) * GRID_PITCH] : NONE), before);
      if (lane + 32u < own_rows) col[(lane + 32u) * GRID_PITCH] = x1;
    }
  }
  task_sync(K);
  // (a CTA with variants comes behind full ones only)
  if (share && own && tid < ng) {
    uint32_t v = NONE;
#pragma unroll 1
    for (uint32_t o = 0; o < share; ++o) v = min(v, *peer(&grid[(rows - 1u) * GRID_PITCH + tid], o));
    carry[tid] = v;
  }
  __syncthreads();
  // 3. what the grid lets through ...
#pragma unroll 1
  for (uint32_t b = lo; b < hi; b += B) {
    const uint32_t i = b + tid;
    bool pass = false;
    uint2 a = make_uint2(0u, 0u);
    if (i < hi) {
      a = by_local[i - lo];
      if (a.y != 0xFFFFu) {
        const uint32_t y = (i >> cs) - y0, x = a.y >> cs;
        const uint32_t g = x ? min(carry[x - 1u], y ? grid[(y - 1u) * GRID_PITCH + x - 1u] : NONE) : NONE;
        const uint32_t order = i == own0 ? r0.order : c.s_order[base + i];
        // (a latency of NONE - 1 cannot be told from a saturated one in the grid: step 4 looks at all)
        pass = g > min(a.x, NONE - 1u) || (a.x == NONE - 1u && g == NONE - 1u);
        if (order >> 31) pass = pass && a.x <= *run_min_of(order);
      }
    }
    const unsigned m = __ballot_sync(0xFFFFFFFFu, pass);
    uint32_t at = 0;
    if (m && lane == 0u) at = atomicAdd(&n_cand, (uint32_t)__popc(m));
    at = __shfl_sync(0xFFFFFFFFu, at, 0);
    if (lane == 0u && i < hi) passed_local[(i - lo) >> 5] = m;
    if (pass) {
      cand[at + __popc(m & ((1u << lane) - 1u))] = (uint16_t)(i - lo);
#pragma unroll 1
      for (uint32_t o = share; o < K; ++o) {
        *peer(&by_acc[a.y], o) = make_uint2(a.x, i);
        atomicOr(peer(&passed_acc[a.y >> 5], o), 1u << (a.y & 31u));
      }
    }
  }
  task_sync(K);
  // 4. ... against the entries before it in its own row and column of the grid that were let through
  // too (dominance is transitive and what is dominated by nothing is let through): four lanes for
  // the row, four for the column
  const uint32_t nc = n_cand;
#pragma unroll 1
  for (uint32_t x0 = 0; x0 < nc; x0 += B / 8u) {
    const uint32_t x = x0 + (tid >> 3);
    uint32_t dom = 0, p = 0;
    if (x < nc) {
      p = cand[x];
      const uint2 a = by_local[p];
      const bool row = !(tid & 4u);
      const uint2 *v = row ? by_local : by_acc;
      const uint32_t *bits = row ? passed_local : passed_acc;
      const uint32_t end = row ? p : a.y, limit = row ? a.y : lo + p;
      const uint32_t from = !row && a.x == NONE - 1u ? 0u : (end >> cs) << cs;
#pragma unroll 1
      for (uint32_t w = from >> 5; w <= end >> 5 && !dom; ++w) {
        uint32_t m = bits[w] & (0x11111111u << (tid & 3u));
        if (w == from >> 5) m &= ~0u << (from & 31u);
        if (w == end >> 5) m &= (1u << (end & 31u)) - 1u;
#pragma unroll 1
        while (m && !dom) {
          const uint2 e = v[32u * w + (uint32_t)__ffs(m) - 1u];
          m &= m - 1u;
          dom = (uint32_t)(e.x <= a.x) & (uint32_t)(e.y < limit);
        }
      }
    }
    dom = __ballot_sync(0xFFFFFFFFu, dom != 0u) >> (lane & 24u) & 0xFFu;
    if (x < nc && !(tid & 7u) && !dom) atomicOr(&keep[(lo + p) >> 5], 1u << (p & 31u));
  }
  if (K > 1u) {                                                    // survivors to all, each word by the CTA that has it
    __syncthreads();
    const uint32_t w = sh.w0 + tid;
    if (w < sh.w1) {
      const uint32_t bits = keep[w];
#pragma unroll 1
      for (uint32_t o = 0; o < K; ++o)
        if (o != share) *peer(&keep[w], o) = bits;
    }
  }
  task_sync(K);
  // 5. survivors before each word of the bit set
  const uint32_t n_words = (V + 31u) >> 5;
  if (32u * warp <= n_words) {
    uint32_t below = 0;
#pragma unroll 4
    for (uint32_t x = lane; x < 32u * warp; x += 32u) below += __popc(keep[x]);
    below = __reduce_add_sync(0xFFFFFFFFu, below);
    const uint32_t pc = tid < n_words ? __popc(keep[tid]) : 0u;
    const uint32_t incl = below + warp_scan_add(pc);
    if (tid <= n_words) keep_pre[tid] = incl - pc;
  }
  const uint32_t n_class = c.stateful && share == 0u ? c.n_class[t] : 0u;
  uint32_t *class_eff = reinterpret_cast<uint32_t *>(by_acc), *class_id = class_eff + n_class;   // by_acc is not needed any more
#pragma unroll 1
  for (uint32_t k = tid; k < n_class; k += B) { class_eff[k] = NONE; class_id[k] = NONE; }
  __syncthreads();
  // 6. the list into the task's region, its first segment also into the index scratch
  auto emit = [&](uint32_t pos, uint32_t pred, uint32_t acc, uint32_t id) {
    keys_g[pos] = ((unsigned long long)acc << 32) | pred;
    ids_g[pos] = id;
    const uint32_t seg = pos / INDEX_MAX_F;
    if (seg < K) peer(&S, seg)->put(pos - seg * INDEX_MAX_F, pred, acc, id, c.acc_lo);
  };
  auto before = [&](uint32_t i) { return keep_pre[i >> 5] + __popc(keep[i >> 5] & ((1u << (i & 31u)) - 1u)); };
#pragma unroll 1
  for (uint32_t i = own0; i < hi; i += B) {
    if (!((keep[i >> 5] >> (i & 31u)) & 1u)) continue;
    const bool reg = i == own0;
    const uint32_t run = reg ? run0 : c.s_cost_run[base + i];
    const uint32_t pos = before(run & 0xFFFFu) + before(run >> 16) - 1u - before(i);
    emit(pos, reg ? pred0 : by_local[i - lo].x, reg ? acc0 : c.s_acc[base + i], reg ? r0.id : c.s_id[base + i]);
  }
  // the counts are cleared here, far behind their loads: a store to a line whose load is still in flight
  // holds up everything behind it (4 us a launch when the store came right behind)
  if (advance)
#pragma unroll 1
    for (uint32_t i = own0; i < hi; i += B) c.count_by_id[i == own0 ? r0.id : c.s_id[base + i]] = 0u;
  uint32_t F = keep_pre[n_words];
  if (c.stateful && share == 0u) {                                 // (lo = 0)
    // the fastest Inactive variant of every accuracy class: its latency, then the lowest id with it
    auto eff_of = [&](uint32_t i) {
      const unsigned long long e = (unsigned long long)(i == own0 && i < hi ? pred0 : c.s_pred[base + i]) +
                                   (i == own0 && i < hi ? r0.load_lat : c.s_load_lat[base + i]);
      return e > NONE ? NONE : (uint32_t)e;
    };
    auto inactive = [&](uint32_t i) { return (i == own0 && i < hi ? r0.state : c.s_state[base + i]) == INFAAS_STATE_INACTIVE; };
    auto class_of = [&](uint32_t i) { return i == own0 && i < hi ? class0 : c.s_class[base + i]; };
#pragma unroll 1
    for (uint32_t i = tid; i < V; i += B)
      if (inactive(i)) atomicMin(&class_eff[class_of(i)], eff_of(i));
    __syncthreads();
#pragma unroll 1
    for (uint32_t i = tid; i < V; i += B)
      if (inactive(i) && class_eff[class_of(i)] == eff_of(i)) atomicMin(&class_id[class_of(i)], i == own0 && i < hi ? r0.id : c.s_id[base + i]);
    __syncthreads();
    // each thread takes consecutive classes (one, up to 1024 of them): running minimum from the
    // highest accuracy down, survivors, their number.  A class without entry counts as 2^32.
    const uint32_t per = max(1u, (n_class + B - 1u) / B), k0 = min(n_class, tid * per), k1 = min(n_class, k0 + per);
    const uint32_t used = (n_class + 32u * per - 1u) / (32u * per);        // warps that have classes
    auto eff_at = [&](uint32_t k) { return class_id[k] == NONE ? 1ull << 32 : (unsigned long long)class_eff[k]; };
    unsigned long long mine = 1ull << 32;
#pragma unroll 1
    for (uint32_t k = k0; k < k1; ++k) mine = min(mine, eff_at(k));
    unsigned long long best = 1ull << 32;
    if (warp < used) {
      const unsigned long long incl = warp_scan_min(mine);
      if (lane == 31u) warp_min[warp] = incl;
      best = __shfl_up_sync(0xFFFFFFFFu, incl, 1);
      if (lane == 0u) best = 1ull << 32;
    }
    if (used > 1u) {
      __syncthreads();
#pragma unroll 1
      for (uint32_t w = 0; w < min(warp, used); ++w) best = min(best, warp_min[w]);
    }
    // on the list: faster than every more accurate variant (equally fast ones are dominated)
    uint32_t n = 0;
    unsigned long long ahead = best;
#pragma unroll 1
    for (uint32_t k = k0; k < k1; ++k) {
      const unsigned long long x = eff_at(k);
      n += x < ahead;
      ahead = min(ahead, x);
    }
    const uint32_t n_incl = warp_scan_add(n);
    if (lane == 31u) warp_cnt[warp] = n_incl;
    if (used > 1u) __syncthreads();
    if (warp < used) {
      uint32_t before_n = n_incl - n, total = 0;
      if (used > 1u) {
#pragma unroll 1
        for (uint32_t w = 0; w < used; ++w) {
          before_n += w < warp ? warp_cnt[w] : 0u;
          total += warp_cnt[w];
        }
      } else {
        total = __shfl_sync(0xFFFFFFFFu, n_incl, 31);
      }
      if (tid == 0u) n_inactive = total;
      ahead = best;
#pragma unroll 1
      for (uint32_t k = k0; k < k1; ++k) {
        const unsigned long long x = eff_at(k);
        if (x < ahead) { emit(F + total - 1u - before_n, (uint32_t)x, c.class_acc[base + k], class_id[k]); ++before_n; }
        ahead = min(ahead, x);
      }
    }
    __syncthreads();
    F += n_inactive;
  }
  if (share == 0u && tid == 0u) c.f_len[t] = F;
  task_sync(K);
  if (K > 1u) F = *reinterpret_cast<volatile uint32_t *>(c.f_len + t);   // (with the Inactive list's, which CTA 0 made)
  return F;
}

// Index of a task's list, segment by segment (INDEX_MAX_F positions each; almost always one); of K CTAs
// the one numbered `share` takes every K-th.  The two lists of a state-aware catalog count as one, the
// Inactive entries behind the Active ones: "first position that meets both requirements, else the
// smallest distance at the lowest position" is all the index knows about order.  Returns false if
// there is no index (empty list, or no room).
template <uint32_t B, uint32_t NB>
__device__ __forceinline__ bool index_list(const DeviceCatalog &c, uint32_t t, uint32_t F, IndexScratch<B, NB> &S, uint32_t share,
                                           uint32_t K, uint32_t Sh, uint32_t bmin) {
  bool indexed = F > 0;
  bool counted = false;                       // has this CTA made its last allocation?
  if (indexed) {
    const uint32_t nseg = (F + INDEX_MAX_F - 1u) / INDEX_MAX_F;
#pragma unroll 1
    for (uint32_t sg = share; sg < nseg && indexed; sg += K) {
      const uint32_t off = sg * INDEX_MAX_F, Fseg = min(INDEX_MAX_F, F - off), x0 = nseg > 1u ? c.seg_base[t] : 0u;
      if (sg >= K) {                              // not there yet: back from the task's region
        const unsigned char *region = c.regions + c.reg_off[t];
        const unsigned long long *keys_g = reinterpret_cast<const unsigned long long *>(region);
        const uint32_t *ids_g = reinterpret_cast<const uint32_t *>(region + 8u * (c.task_off[t + 1] - c.task_off[t]));
        __syncthreads();
        S.clear(c.n_buckets, c.nbw);
        __syncthreads();
        if (threadIdx.x < Fseg) {
          const unsigned long long e = keys_g[off + threadIdx.x];
          S.put(threadIdx.x, (uint32_t)e, (uint32_t)(e >> 32), ids_g[off + threadIdx.x], c.acc_lo);
        }
        __syncthreads();
      }
      indexed = build_index(c, t, Fseg, S, sg ? x0 + sg - 1u : NONE, sg + 1u < nseg ? x0 + sg + 1u : 0u, sg + K >= nseg, Sh, bmin);
      counted = sg + K >= nseg;
    }
  }
  if (!counted && threadIdx.x == 0u) place_block_finish(c, place_block_issue(c, 0u, true), 0u, true);   // nothing (more) to place
  return indexed;
}

// What is left to write once a task's list is indexed, or is not (one CTA per task).
__device__ __forceinline__ void finish_task(const DeviceCatalog &c, uint32_t t, uint32_t F, bool indexed, bool advance, uint32_t Sh,
                                            uint32_t bmin) {
  const uint32_t tid = threadIdx.x;
  if (!indexed) {
    // no index: every query of this task reads "none"
    write_dummy_task(c, t);
    if (tid == 0u) c.slow[t] = make_uint4(0u, 0u, F == 0 ? TASK_FLAG_INVALID : TASK_FLAG_NOT_INDEXED, 0u);
  }
  if (t == 0u) {
    // the bucket scale every CTA has used, for the selection kernel; at load time also entry n_tasks
    // (queries whose task is out of range) and the dummy block, which never change
    if (tid == 0u) {
      c.image_hdr[1] = (127u - Sh) << 23;
      c.image_hdr[2] = __float_as_uint(-(float)bmin);
    }
    if (!advance) {
      write_dummy_task(c, c.n_tasks);
      if (tid < IMAGE_DUMMY_BYTES / 4u) reinterpret_cast<uint32_t *>(c.image)[tid] = tid == 3u ? PENDING : 0u;
    }
  }
}

// Tasks of more than 512 variants: c.rebuild_ctas CTAs per task, a cluster, which share the list's variants and
// then its segments.
//
// Bound by the latency of its chain of barriers and shared-memory round trips, and by fetching its
// code: every line of it runs about once per launch, and with the compiler's unrolling (116 KB of
// code) 40 % of the stalls were for instructions.  So the loops are not unrolled (50 KB) except the
// few that run long.  4 CTAs for tasks of more than 1024 variants (rule and figures in infaas_catalog_load).  With
// them a twentieth of the stalls are for instructions, 27 % at barriers, 14 % for the cluster barriers' fences.
__global__ void __launch_bounds__(REBUILD_THREADS)
rebuild_kernel(DeviceCatalog c, int advance, uint32_t window_us) {
  extern __shared__ __align__(16) unsigned char dyn[];
  __shared__ __align__(16) IndexScratch<REBUILD_THREADS, MAX_BUCKETS> S;
  const uint32_t K = c.rebuild_ctas, t = blockIdx.x >> (K >> 1), share = blockIdx.x & (K - 1u);   // K = 1 or 4
  uint32_t slo_seen, bmin, Sh;                                     // SLO buckets
  const uint32_t F = build_list(c, t, share, K, advance, window_us, dyn, S, slo_seen);
  bucket_scale(c, slo_seen, Sh, bmin);
  const bool indexed = index_list(c, t, F, S, share, K, Sh, bmin);
  if (share == 0u) finish_task(c, t, F, indexed, advance, Sh, bmin);
}

// Queue recursion, prune and list of one task of at most B variants, one per thread; otherwise as
// build_list.  Contains chain_wait.  Returns the list's length.
//
// List of the Active variants: p is dominated by a faster variant of the same cost and accuracy, or by
// a variant q before it in both orders (local, accuracy) with pred_q <= pred_p.  Both orders are fixed, so
// everything about them is known before the wait.  Warp g owns the 32 variants at accuracy positions
// 32 g .. 32 g + 31.  Those q in lower groups come before all of its own in accuracy order: a running
// minimum over their latencies in local order (B / 32 consecutive variants per lane, then one warp
// scan) answers for them.  Those inside the group are compared directly, against a bit mask of which
// of them come before in both orders (laid down with the catalog).  No list of candidates, one barrier.
//
// List of the Inactive variants: the fastest (lowest id) of every accuracy class, if it is faster than
// everything more accurate, from the lowest accuracy up.
template <uint32_t B>
__device__ __forceinline__ uint32_t build_list_small(const DeviceCatalog &c, uint32_t t, bool advance, uint32_t window_us,
                                                     IndexScratch<B, B> &S, uint32_t &Sh, uint32_t &bmin) {
  constexpr uint32_t GROUPS = B / 32u, E = B / 32u;                // E: consecutive variants (or classes) per lane
  static_assert(GROUPS < 32u, "a lane per word of a bit set, and one behind them");
  // Where element i is in an array of which each lane reads E consecutive elements: lane l's j-th at j * PITCH + l,
  // without bank conflicts for readers (j fixed) and for writers (32 consecutive i).
  constexpr uint32_t PITCH = 32u + 32u / E;
  auto at = [](uint32_t i) { return (i % E) * PITCH + i / E; };
  // latencies as the prune compares them: NONE = not listed, so a saturated one counts as one less
  __shared__ uint32_t by_lane[E * PITCH];                          // by local index (laid out by `at`)
  __shared__ __align__(16) uint32_t by_pos[B];                  // ... by accuracy position
  __shared__ uint32_t run_min[B];                               // at the first of each (cost, accuracy): smallest pred
  __shared__ uint16_t pos_of[B];                                // accuracy position of each local index
  __shared__ uint32_t listed[GROUPS], dominated[GROUPS], spared[GROUPS];   // bit sets by local index
  __shared__ uint32_t class_eff[E * PITCH], class_id[E * PITCH];   // per accuracy class: smallest latency, lowest id with it
  __shared__ uint16_t class_acc[E * PITCH];
  const uint32_t tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5;
  const uint32_t base = c.task_off[t], V = c.task_off[t + 1] - base;
  const bool live = tid < V;
  unsigned char *region = c.regions + c.reg_off[t];
  unsigned long long *keys_g = reinterpret_cast<unsigned long long *>(region);
  uint32_t *ids_g = reinterpret_cast<uint32_t *>(region + 8u * V);

  // 1. before the wait: what no kernel writes, and clearing
  Row r;
  r.drain = 0;
  uint32_t acc = 0, run = 0, cls = 0, pos = 0xFFFFu;
  uint2 own = make_uint2(0u, 0u);                                  // local index at accuracy position tid, mask of its group
  if (live) {
    r = load_fixed(c, base + tid, window_us);
    acc = c.s_acc[base + tid];
    run = c.s_cost_run[base + tid];
    own = c.by_acc[base + tid];
    pos = r.order & 0x1FFFu;
    if (c.stateful) cls = c.s_class[base + tid];
  }
  pos_of[tid] = (uint16_t)pos;
  by_lane[at(tid)] = NONE;
  by_pos[tid] = NONE;
  run_min[tid] = NONE;
  if (tid < GROUPS) { dominated[tid] = 0u; spared[tid] = 0u; }
  if (c.stateful) {
    class_eff[at(tid)] = NONE; class_id[at(tid)] = NONE;
    if (live) class_acc[at(cls)] = (uint16_t)acc;
  }
  S.clear(c.n_buckets, c.nbw);
  __syncthreads();
  // this lane's E variants: which belong to lower groups, which to this warp's
  uint32_t lower = 0, same = 0;
#pragma unroll
  for (uint32_t j = 0; j < E; ++j) {
    const uint32_t g = pos_of[lane * E + j] >> 5;
    lower |= (uint32_t)(g < warp) << j;
    same |= (uint32_t)(g == warp) << j;
  }
  // (the compiler would move the division and the masks behind the wait, to their use: 1000 cycles)
  asm volatile("" : "+r"(r.drain), "+r"(lower), "+r"(same));
  chain_wait();
  chain_next();
  const uint32_t slo_seen = *c.slo_seen;
  // 2. queue recursion, states, predicted latencies
  uint32_t pred = NONE, eff = NONE;
  bool active = false, inactive = false;
  if (live) {
    load_load(c, base + tid, advance, r);
    pred = advance_row(c, base + tid, r, advance);
    active = r.state == INFAAS_STATE_ACTIVE;
    inactive = r.state == INFAAS_STATE_INACTIVE;
    if (active) {
      by_lane[at(tid)] = by_pos[pos] = min(pred, NONE - 1u);
      if (r.order >> 31) atomicMin(&run_min[(r.order >> 13) & 0x1FFFu], pred);
    }
    if (inactive) {
      const unsigned long long e = (unsigned long long)pred + r.load_lat;
      eff = e > NONE ? NONE : (uint32_t)e;
      atomicMin(&class_eff[at(cls)], eff);
    }
  }
  const unsigned m = __ballot_sync(0xFFFFFFFFu, active);
  if (lane == 0u) listed[warp] = m;
  bucket_scale(c, slo_seen, Sh, bmin);
  __syncthreads();
  // 3. prune
  if (32u * warp < V) {
    uint32_t x[E], least = NONE;
#pragma unroll
    for (uint32_t j = 0; j < E; ++j) {
      x[j] = by_lane[j * PITCH + lane];
      least = min(least, (lower >> j) & 1u ? x[j] : NONE);
    }
    least = lanes_before(warp_scan_min(least), NONE);
    uint32_t dom = 0;
#pragma unroll
    for (uint32_t j = 0; j < E; ++j) {
      dom |= (uint32_t)(((same >> j) & 1u) && least <= x[j]) << j;
      least = min(least, (lower >> j) & 1u ? x[j] : NONE);
    }
    if (dom) atomicOr(&dominated[(lane * E) >> 5], dom << ((lane * E) & 31u));
  }
  if (live) {                                                      // the variant at accuracy position tid
    const uint32_t p = by_pos[tid], o = own.x;
    uint32_t le = 0;
#pragma unroll
    for (uint32_t j = 0; j < 8u; ++j) {
      const uint4 v = *reinterpret_cast<const uint4 *>(&by_pos[32u * warp + 4u * j]);
      le |= (uint32_t)(v.x <= p) << (4u * j) | (uint32_t)(v.y <= p) << (4u * j + 1u) | (uint32_t)(v.z <= p) << (4u * j + 2u) |
            (uint32_t)(v.w <= p) << (4u * j + 3u);
    }
    if (le & own.y) atomicOr(&dominated[o >> 5], 1u << (o & 31u));   // (one that is not listed: no harm)
  }
  const bool slower_twin = active && (r.order >> 31) && pred > run_min[(r.order >> 13) & 0x1FFFu];
  if (slower_twin) atomicOr(&dominated[warp], 1u << lane);
  if (active && pred == NONE - 1u && !slower_twin) {               // saturated ones looked as fast: look again
    bool dom = false;
#pragma unroll 1
    for (uint32_t q = 0; q < tid && !dom; ++q)
      dom = ((listed[q >> 5] >> (q & 31u)) & 1u) && pos_of[q] < pos && c.s_pred[base + q] <= pred;
    if (!dom) atomicOr(&spared[warp], 1u << lane);
  }
  if (inactive && class_eff[at(cls)] == eff) atomicMin(&class_id[at(cls)], r.id);
  __syncthreads();
  // 4. the list into the task's region, its first segment also into the index scratch.  Positions:
  // survivors before the run of equal cost, then the run backwards
  const uint32_t kept = lane < GROUPS ? listed[lane] & (~dominated[lane] | spared[lane]) : 0u, n_kept = __popc(kept);
  const uint32_t before_word = warp_scan_add(n_kept) - n_kept;
  const uint32_t n_active = __shfl_sync(0xFFFFFFFFu, before_word + n_kept, 31);
  auto before = [&](uint32_t i) {                                  // survivors before local index i <= B (all lanes)
    const int w = (int)(i >> 5);                                   // (word GROUPS is empty)
    return __shfl_sync(0xFFFFFFFFu, before_word, w) + __popc(__shfl_sync(0xFFFFFFFFu, kept, w) & ((1u << (i & 31u)) - 1u));
  };
  auto emit = [&](uint32_t at_pos, uint32_t latency, uint32_t accuracy, uint32_t id) {
    keys_g[at_pos] = ((unsigned long long)accuracy << 32) | latency;
    ids_g[at_pos] = id;
    if (at_pos < INDEX_MAX_F) S.put(at_pos, latency, accuracy, id, c.acc_lo);
  };
  const uint32_t list_pos = before(run & 0xFFFFu) + before(run >> 16) - 1u - before(tid);
  const uint32_t own_word = __shfl_sync(0xFFFFFFFFu, kept, (int)warp);
  if ((own_word >> lane) & 1u) emit(list_pos, pred, acc, r.id);
  // the counts are cleared here, far behind their loads: a store to a line whose load is still in flight
  // holds up everything behind it
  if (advance && live) c.count_by_id[r.id] = 0u;
  uint32_t n_inactive = 0;
  if (c.stateful) {
    // (every warp goes through all classes.)  E classes per lane, from the highest accuracy down: those with an entry, their running minimum,
    // survivors, their number
    uint32_t x[E], some = 0, least = NONE;
#pragma unroll
    for (uint32_t j = 0; j < E; ++j) {
      x[j] = class_eff[j * PITCH + lane];
      some |= (uint32_t)(class_id[j * PITCH + lane] != NONE) << j;
      least = min(least, x[j]);                                    // (NONE in a class without entry)
    }
    least = lanes_before(warp_scan_min(least), NONE);
    bool first = !(__ballot_sync(0xFFFFFFFFu, some != 0u) & ((1u << lane) - 1u));   // none before this lane's
    // on the list: faster than every more accurate variant (equally fast ones are dominated)
    uint32_t on = 0;
#pragma unroll
    for (uint32_t j = 0; j < E; ++j) {
      const bool here = (some >> j) & 1u;
      on |= (uint32_t)(here && (first || x[j] < least)) << j;
      least = min(least, x[j]);
      first = first && !here;
    }
    const uint32_t n = __popc(on), incl = warp_scan_add(n);
    n_inactive = __shfl_sync(0xFFFFFFFFu, incl, 31);
    // one class per thread: the list runs from the lowest accuracy up
    const uint32_t top = n_active + n_inactive - 1u - (incl - n), its_top = __shfl_sync(0xFFFFFFFFu, top, (int)(tid / E)),
                   its_on = __shfl_sync(0xFFFFFFFFu, on, (int)(tid / E)), j = tid % E, k = at(tid);
    if ((its_on >> j) & 1u) emit(its_top - __popc(its_on & ((1u << j) - 1u)), class_eff[k], class_acc[k], class_id[k]);
  }
  __syncthreads();
  return n_active + n_inactive;
}

// Tasks of at most B variants: one CTA of B threads per task, a thread per variant (B = 256 or 512).
//
// Bound by the latency of its chain: the loads after the wait (1.7 K cycles, of which the gather of
// counts that other SMs' atomics have just written is half), seven barriers with a few shared-memory round trips each,
// and the instructions of every warp.  Cycles after the wait, 64 tasks x 256 variants with lists of up to 100
// entries, this kernel / rebuild_kernel with its 1024 threads: 11.2 K / 16.6 K; lists of up to 50: 9.7 K /
// 16.4 K; 128 x 512, up to 134: 14.3 K / 19.6 K; two lists per task: 10.5 K / 16.7 K.  A window of 65,536
// queries: 15.3 -> 13.4 us (64 x 256), 16.2 -> 15.2 (128 x 512); 12.6 and 13.9 since the selection keeps off its SMs.  512 threads for tasks of up to 256: the
// steps with work for few warps 30 % faster, the rank table slower, the sum the same.
template <uint32_t B>
__global__ void __launch_bounds__(B)
rebuild_small_kernel(DeviceCatalog c, int advance, uint32_t window_us) {
  __shared__ __align__(16) IndexScratch<B, B> S;
  const uint32_t t = blockIdx.x;
  uint32_t Sh, bmin;
  const uint32_t F = build_list_small<B>(c, t, advance, window_us, S, Sh, bmin);
  if (threadIdx.x == 0u) c.f_len[t] = F;
  const bool indexed = index_list(c, t, F, S, 0u, 1u, Sh, bmin);
  finish_task(c, t, F, indexed, advance, Sh, bmin);
}

static_assert(REBUILD_CLUSTER == 4, "task and share from the CTA's index in rebuild_kernel");

}  // namespace

cudaError_t prepare_rebuild_kernel() {
  return cudaFuncSetAttribute(rebuild_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)(INFAAS_MAX_TASK_VARIANTS * REBUILD_ROW_SMEM));
}

cudaError_t rebuild_clusters_at_once(uint32_t max_task_variants, uint32_t *n) {
  cudaLaunchAttribute attr = {};
  attr.id = cudaLaunchAttributeClusterDimension;
  attr.val.clusterDim.x = REBUILD_CLUSTER;
  attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(REBUILD_CLUSTER);
  cfg.blockDim = dim3(REBUILD_THREADS);
  cfg.dynamicSmemBytes = (size_t)max_task_variants * REBUILD_ROW_SMEM;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  int clusters = 0;
  const cudaError_t e = cudaOccupancyMaxActiveClusters(&clusters, rebuild_kernel, &cfg);
  *n = clusters > 0 ? (uint32_t)clusters : 0u;
  return e;
}

cudaError_t launch_rebuild(const DeviceCatalog &c, bool advance_queues, uint32_t window_us,
                           cudaStream_t stream) {
  // a thread per variant up to 512 (as fast as it gets with registers and bit masks), beyond that in rounds
  if (c.max_task_variants <= REBUILD_THREAD_MAX)
    return launch_chained(c.max_task_variants <= 256u ? rebuild_small_kernel<256> : rebuild_small_kernel<512>, c.n_tasks,
                          c.max_task_variants <= 256u ? 256u : 512u, 0, split_for(c), stream, c, advance_queues ? 1 : 0, window_us);
  const size_t smem = (size_t)c.max_task_variants * REBUILD_ROW_SMEM;
  return launch_chained_cluster(rebuild_kernel, c.n_tasks * c.rebuild_ctas, c.rebuild_ctas, REBUILD_THREADS, smem, split_for(c), stream, c,
                                advance_queues ? 1 : 0, window_us);
}

}  // namespace infaas
