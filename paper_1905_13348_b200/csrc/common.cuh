// Shared declarations of the CUDA path: the device-side catalog layout, the packed image
// the selection kernel reads, and the launch functions the C ABI calls.  Nothing in this
// directory is used by, or uses, the CPU oracle.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "infaas.h"

namespace infaas {

// ---------------------------------------------------------------------------------------
// Scan list of a task: its non-dominated variants sorted by (cost, pred_lat, 10000-acc, id).
// Position p in that order is what selection returns the smallest feasible of.
//
// A state-aware catalog has two lists per task, one after the other: the Active variants in
// the order above, then the Inactive ones with pred_lat + loading latency (saturating) in
// place of both cost and pred_lat; each list is pruned on its own, variants in other states
// are in neither.  "First feasible position, else the smallest distance at the lowest
// position" over the two lists in this order is the state-aware answer, and that is all the
// index below knows about order, so the two lists are indexed as one.
//
// A list is cut into segments of at most INDEX_MAX_F consecutive positions (almost always
// one).  The selection kernel's fast path looks at the first segment only; if that holds
// nothing feasible the slow path goes through the others in order.  For a segment of F
// entries the rebuild kernel derives an exact index:
//   Pd[0..Ks)  distinct pred_lat values ascending,  Ad[0..Ka)  distinct acc_bp ascending,
//   r(slo) = #{Pd <= slo},  k(min_acc) = #{Ad < min_acc},
//   T2[r][k] = first position whose pred_lat is among the r smallest values and whose
//              acc_bp is not among the k smallest values, or F if there is none.
//
// r comes from one record of a table of n_buckets records per task.  The bucket of an
// SLO is  j = clamp((bits(slo) >> S) - bmin, 0, n_buckets - 1)  with bits(x) = the IEEE-754 pattern
// of x converted to float toward zero (a monotone, roughly logarithmic code) and one S = 16..23
// and bmin for the whole catalog.  A record is  R << 24 | C  and
// r = (record + (slo & 0xFFFFFF)) >> 24:
//   - no distinct latency inside the bucket: R = the rank there, C = 0 (never carries);
//   - one latency `thr` inside it, and all SLOs of the bucket agree in their top byte:
//     R = rank below, C = 0xFFFFFF - ((thr - 1) & 0xFFFFFF), so the add carries into R
//     exactly when slo >= thr;
//   - otherwise R = Ks + 1, C = rank below | latencies inside << 8: rows Ks + 1 and Ks + 2 (the add
//     may carry) of T2 hold only F, which sends the query to the exact slow path; that finds the
//     rank among the latencies the record names.
// The buckets run from the smallest profiled latency of the catalog (a predicted latency is
// never below it) up to the largest SLO any batch has asked for so far (kept as a bit mask,
// at least SLO_CAP_FLOOR_US); larger latencies share the last bucket.  The rebuild kernel derives
// S and bmin from these two and publishes them beside the image size.
// k comes from a bitmap over accuracy values with running popcounts (24 bitmap bits and an
// 8-bit prefix count per word), exact at one basis point.  Every bitmap covers the same
// window of accuracies, that of the whole catalog (fixed at load: acc_lo, a multiple of 24,
// and nbw words), so the word an accuracy falls into does not depend on the task.
//
// Image (what the selection kernel stages in shared memory):
//   dummy  64 bytes (what tasks without an index point at: every query of theirs reads
//          "none" and goes to the slow path)
//   hdr    (n_tasks + 1) u32, one per task: t2_off | (Ka + 1) << 24; entry n_tasks serves
//          queries whose task is out of range; padded to 128 bytes
//   rec    (n_tasks + 1) x (n_buckets + 1) u32 records (the last one twice), rec_stride(n_buckets) bytes apart
//   bitmap (n_tasks + 1) x nbw u32: the accuracy bitmaps of the tasks' first segments,
//          bitmap_stride(nbw) bytes apart
//   var    per-segment blocks, each 16-byte aligned:
//          ids   u32[F + 1] in REVERSE order: ids[p] sits at t2_off - 4 - 4p, and the slot
//                of p = F holds PENDING -- the fast path needs no compare for "none"
//          T2    u8[(Ks + 3) * (Ka + 1)]  at t2_off (a multiple of 4)
//          bitmap u32[nbw]  (further segments only)
//          slow-path tables (SlowLayout below)
//
// Per task in global memory (`regions`): keys u64[V] (pred_lat | acc_bp << 32, scan order,
// F used; for Inactive entries the latency includes the loading latency) and ids u32[V], for
// lists without an index and for inspection.
// ---------------------------------------------------------------------------------------
constexpr uint32_t INDEX_MAX_F = 248;
constexpr uint32_t MIN_BUCKETS = 256, MAX_BUCKETS = 2048;
constexpr uint32_t ACC_WORD_BITS = 24;
constexpr uint32_t MAX_ACC_WORDS = 420;          // accuracies 0 .. 10000 need at most 417 + 1 words
constexpr uint32_t IMAGE_T2_LIMIT = 1u << 24;    // t2_off is a 24-bit field
constexpr uint32_t SLO_CAP_FLOOR_US = (1u << 20) - 1u;  // the buckets cover latencies at least up to here
constexpr uint32_t PENDING = 0xFFFFFFFEu;        // never a valid decision (ids stop at 2^31-2)

constexpr uint32_t TASK_FLAG_INVALID = 1u;       // no variant: answer INFAAS_INVALID
constexpr uint32_t TASK_FLAG_NOT_INDEXED = 2u;   // list without index: the slow path walks it

inline __host__ __device__ uint32_t round_up_u32(uint32_t x, uint32_t a) { return (x + a - 1) / a * a; }

// A task's records and its bitmap start an odd number of words after the previous task's, so
// that the tasks' hot entries (the same buckets, the lowest bitmap word) fall into different
// shared-memory banks.
inline __host__ __device__ uint32_t rec_stride(uint32_t nb) { return 4u * (nb + 1u); }   // bytes from one task's records to the next's
// SLO buckets per task: 256, more for tasks of more than 256 variants while all records together stay
// within 48 KB (up to 22 tasks).  Long lists have several latencies per bucket, and every query of
// such a bucket takes the slow path: 2^22 queries on trade-off catalogs with 256 buckets / with more,
// us: 4 x 4096 variants (lists of up to 315 entries) 96.2 / 74.6, 8 x 1000 60.0 / 55.4, 2 x 1000 45.4 /
// 39.8; the rebuild takes up to 1.7 us longer.  The records can push an image out of shared memory that
// would fit with 256 buckets; both ways are as fast then: 4 x 1100 48.9 / 48.0, 5 x 1100 46.7 / 48.6.
inline __host__ __device__ uint32_t buckets_for(uint32_t n_tasks, uint32_t max_task_variants) {
  uint32_t nb = MIN_BUCKETS;
  while (nb < MAX_BUCKETS && nb < max_task_variants && rec_stride(2u * nb) * (n_tasks + 1u) <= 48u * 1024u) nb *= 2u;
  return nb;
}
inline __host__ __device__ uint32_t bitmap_stride(uint32_t nbw) { return 4u * (nbw | 1u); }   // same, bitmaps
constexpr uint32_t IMAGE_DUMMY_BYTES = 64u;               // the dummy block opens the image
constexpr uint32_t IMAGE_HDR_OFFSET = IMAGE_DUMMY_BYTES;  // the task words follow it
inline __host__ __device__ uint32_t image_rec_offset(uint32_t n_tasks) {
  return round_up_u32(IMAGE_HDR_OFFSET + 4u * (n_tasks + 1u), 128u);
}
inline __host__ __device__ uint32_t image_bitmap_offset(uint32_t n_tasks, uint32_t nb) {
  return image_rec_offset(n_tasks) + rec_stride(nb) * (n_tasks + 1u);
}
inline __host__ __device__ uint32_t image_var_offset(uint32_t n_tasks, uint32_t nb, uint32_t nbw) {
  return round_up_u32(image_bitmap_offset(n_tasks, nb) + bitmap_stride(nbw) * (n_tasks + 1u), 64u);
}
// The task word of a task without index (and of entry n_tasks): T2 is the one zero byte at
// offset 16 of the dummy block with row width 0, the id slot of position 0 below it holds
// PENDING.  The dummy block sits at the very start of the image, where the task word's 24-bit
// offset reaches it however large the fixed tables are.
constexpr uint32_t DUMMY_HEADER = 16u;

// Byte offsets of the slow-path tables inside a segment's block, relative to their start
// (8-byte aligned), for a list of F entries with Ks / Ka distinct latencies / accuracies.
//   walk[o]   uint2 (pred_lat, acc | position << 16): the "stair" entries -- those no other
//             entry beats in both latency and accuracy -- in ascending latency (Fs <= F of
//             them, all with different latencies; space for F)
//   bestB[k]  uint2 (pred_lat, position) of the lowest-latency entry among those whose
//             accuracy rank is >= k (first position among equals); position 0xFF if none
//   Pd[i]     u32 distinct latencies
//   bestA[r]  u32 acc | position << 16 of the highest-accuracy entry among those whose
//             latency rank is < r (first position among equals); position 0xFF if none
//   ordStart[r] u8 first walk index whose latency rank is >= r
struct SlowLayout {
  uint32_t walk, bestB, Pd, bestA, ordStart, bytes;
};
inline __host__ __device__ SlowLayout slow_layout(uint32_t F, uint32_t Ks, uint32_t Ka) {
  SlowLayout L;
  L.walk = 0;
  L.bestB = L.walk + 8u * F;
  L.Pd = L.bestB + 8u * (Ka + 1u);
  L.bestA = L.Pd + 4u * Ks;
  L.ordStart = L.bestA + 4u * (Ks + 1u);
  L.bytes = round_up_u32(L.ordStart + Ks + 1u, 8u);
  return L;
}

// Offsets inside a segment's block and its size; `nbw` = 0 for a task's first segment (its
// bitmap lives in the fixed part of the image).
struct BlockLayout {
  uint32_t t2, bitmap, slow, bytes;   // ids start at 0; t2 = 4 (F + 1)
};
inline __host__ __device__ BlockLayout block_layout(uint32_t F, uint32_t Ks, uint32_t Ka, uint32_t nbw) {
  BlockLayout B;
  B.t2 = 4u * (F + 1u);
  B.bitmap = round_up_u32(B.t2 + (Ks + 3u) * (Ka + 1u), 4u);
  B.slow = round_up_u32(B.bitmap + 4u * nbw, 8u);
  B.bytes = round_up_u32(B.slow + slow_layout(F, Ks, Ka).bytes, 16u);
  return B;
}
// Worst-case bytes of one segment's block.
inline __host__ __device__ uint32_t block_capacity(uint32_t V, uint32_t nbw) {
  const uint32_t F = V < INDEX_MAX_F ? V : INDEX_MAX_F;
  return block_layout(F, F, F, nbw).bytes;
}
inline __host__ __device__ uint32_t region_capacity(uint32_t V) { return round_up_u32(12u * V, 64u); }

// Slow-path parameters of a list segment (one uint4 each, global memory; a task's first
// segment at index task, further segments at n_tasks + their index).
//   x = image offset of the slow tables   y = F | Ks << 8 | Ka << 16   z = flags
//   w = Fs | (1 + index of the task's next segment, 0 if none) << 8
// Header of a further segment (xhdr, global memory):
//   x = t2_off   y = Ka + 1   z = image offset of its bitmap   w = 0
// ---------------------------------------------------------------------------------------
// Device catalog.  "Slot" order: variants bucketed by task, inside a task by (cost, 10000-acc,
// id); task t owns slots task_off[t] .. task_off[t+1]-1 and all s_* arrays are indexed by slot.
// A variant's local index is its slot less the task's first.  Cost and accuracy never change, so
// everything about the list order that does not hang on the predicted latency is laid down here
// once: s_order, s_cost_run, s_class, class_acc and by_acc below.
// ---------------------------------------------------------------------------------------
struct DeviceCatalog {
  uint32_t n_variants;
  uint32_t n_tasks;
  uint32_t max_task_variants;

  const uint32_t *task_off;  // [n_tasks + 1]
  const uint32_t *reg_off;   // [n_tasks + 1] byte offset of each task's region
  const uint32_t *s_lat;
  const uint16_t *s_batch;
  const uint16_t *s_acc;
  const uint32_t *s_cost;
  const uint32_t *s_id;
  const uint32_t *s_order;     // position in (10000-acc, local) order (13 bits) | first local index of the
                               // same (cost, acc) << 13 (13 bits) | bit 31: others share (cost, acc)
  const uint32_t *s_cost_run;  // local indices of equal cost: first | (last + 1) << 16
  const uint16_t *s_class;     // rank of the accuracy among the task's distinct ones, 0 = highest
  const uint16_t *class_acc;   // accuracy of class k of task t at [task_off[t] + k]
  const uint32_t *n_class;     // [n_tasks] distinct accuracies
  const uint2 *by_acc;         // task t's variant at accuracy position p, at [task_off[t] + p]: x = its local index, y = bit
                               // m (m < p % 32): the variant m places into p's 32 comes before it in local order too
  uint32_t *s_queued;
  uint32_t *s_pred;
  unsigned long long *s_served;
  uint32_t *count_by_id;     // [n_variants], zero between windows
  uint32_t stateful;         // 1: states and loading latencies below take part (else all Active)
  unsigned char *s_state;    // INFAAS_STATE_* per slot
  const uint32_t *s_load_lat;  // loading latency per slot, microseconds

  unsigned char *regions;    // per task: keys u64[V], ids u32[V] (scan order)
  uint32_t *f_len;           // [n_tasks] list length F
  uint4 *slow;               // [n_tasks + n_extra] slow-path parameters of the segments
  const uint32_t *seg_base;  // [n_tasks + 1] index of each task's first further segment
  uint4 *xhdr;               // [n_extra] headers of the further segments (first segments: in the image)

  unsigned char *image;      // packed image, image_capacity bytes, 256-byte aligned
  uint32_t image_capacity;
  uint32_t *image_hdr;       // published by the rebuild kernel: [0] bytes of the image, [1] the bucket
                             // scale 2^-S and [2] -bmin, both as float patterns
  uint32_t n_buckets;        // SLO buckets per task
  uint32_t rebuild_ctas;     // CTAs per task of the rebuild kernel (1 or REBUILD_CLUSTER)
  uint32_t acc_lo, nbw;      // accuracy window of every bitmap: acc_lo (multiple of 24) .. acc_lo + 24 nbw - 1
  uint32_t lat_code_lo;      // bits(smallest profiled latency) >> 16: where the SLO buckets start

  unsigned long long *counters;  // [3] feasible, no-feasible, invalid
  unsigned long long *alloc_ctr; // rebuild kernel: block cursor (low 32 bits) | CTAs done allocating << 32;
                                 // zero between kernels
  uint32_t *err;                 // sticky device error word (0 = fine)
  uint32_t *slo_seen;            // OR of all SLOs the selection kernel has read
};

// What the layout kernel reads (rows by id; members = each task's ids in ascending order) and the
// arrays it fills (see DeviceCatalog; s_arch, s_qps = floor(10^9 * batch / lat_us) are the
// autoscaler's, hw_by_id the worker choice's, slot_of_id the host's).
struct CatalogLayout {
  const infaas_variant *rows;
  const uint32_t *members, *task_off;
  uint32_t *s_lat, *s_cost, *s_id, *s_queued, *s_order, *s_cost_run, *n_class, *slot_of_id;
  uint16_t *s_batch, *s_acc, *s_arch, *s_class, *class_acc;
  uint2 *by_acc;
  unsigned long long *s_qps;
  unsigned char *hw_by_id;
};

// Device error codes stored in DeviceCatalog::err.
enum : uint32_t {
  DEV_ERR_NONE = 0,
  DEV_ERR_STAGE_TIMEOUT = 1,   // the bulk copy into shared memory did not complete in time
};

// Largest dynamic shared memory the selection kernel may be given (227 KB per CTA on
// sm_100, minus its static shared memory).
constexpr uint32_t SELECT_MAX_SMEM = 227u * 1024u - 256u;
// Shared memory of the rebuild kernel per variant of the largest task.
constexpr uint32_t REBUILD_ROW_SMEM = 22u;
constexpr uint32_t REBUILD_CLUSTER = 4u;   // CTAs per large task

// The rebuild kernel's coarse grid over a task of V variants (at most GRID x GRID cells; row = run of 2^cs
// local indices, column = run of as many positions in accuracy order) and what CTA `share` of the task's K has
// of it: rows from y0, local indices lo .. hi - 1, and words w0 .. w1 - 1 of the bit sets by local index.  The
// rows of a CTA are an even number, so its variants are whole words; behind the last variant a CTA has nothing
// at all, no part of the last word either: every word has one CTA that writes it.
constexpr uint32_t GRID = 64;
struct TaskShare {
  uint32_t cs, ng, rows, y0, lo, hi, w0, w1;
};
inline __host__ __device__ TaskShare task_share(uint32_t V, uint32_t K, uint32_t share) {
  TaskShare s;
  s.cs = 4;
#pragma unroll 1
  while (V > (GRID << s.cs)) ++s.cs;
  s.ng = (V + (1u << s.cs) - 1u) >> s.cs;
  s.rows = K > 1u ? ((s.ng + K - 1u) / K + 1u) & ~1u : s.ng;
  s.y0 = share * s.rows;
  const uint32_t lo = s.y0 << s.cs, hi = (s.y0 + s.rows) << s.cs;
  s.lo = lo < V ? lo : V;
  s.hi = hi < V ? hi : V;
  s.w0 = s.lo >> 5;
  s.w1 = s.lo < s.hi ? (s.hi + 31u) >> 5 : s.w0;
  return s;
}

// Once per device, with that device current: raise the kernels' shared-memory limits.
cudaError_t prepare_select_kernel();
cudaError_t prepare_tally_kernel();
cudaError_t prepare_rebuild_kernel();
// How many clusters of REBUILD_CLUSTER CTAs of the rebuild kernel the current device runs at once.
cudaError_t rebuild_clusters_at_once(uint32_t max_task_variants, uint32_t *n);

// Kernels of one stream overlap at their seams (programmatic dependent launch): a kernel launched
// with launch_chained may start while its predecessor still runs.  Before chain_wait() it touches
// only what no kernel writes once the catalog is loaded (the layout: infaas_catalog_load waits for
// the layout kernel before it launches the first chained one); chain_wait() returns when everything
// before the kernel in the stream is complete and visible.  A kernel lets its successor start
// (chain_next) only after its own chain_wait, so at most two overlap.  Measured: a window of 65,536
// queries (two kernels) 24.1 -> 19.6 us, a step of 2^24 queries (three) 77 -> 70 us.
__device__ __forceinline__ void chain_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void chain_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
// What an earlier kernel of the stream may have written changes while an overlapped kernel is already
// running, so it is read with ordinary loads, which stay behind chain_wait() -- not with __ldg or
// through const __restrict__, which promise that it does not change and may be moved over the wait.
// (The layout's arrays are fixed.)  Measured with __ldg: the words the rebuild publishes came 0.2 us
// early, before the wait.  load_once: an ordinary load of what is read once, evicted first.
__device__ __forceinline__ uint2 load_once(const uint2 *p) {
  uint2 v;
  asm volatile("ld.global.cs.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "l"(p));
  return v;
}
__device__ __forceinline__ uint4 load_once(const uint4 *p) {
  uint4 v;
  asm volatile("ld.global.cs.v4.u32 {%0, %1, %2, %3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
  return v;
}
// How an SM's 228 KB are split between L1 and shared memory: a CTA only starts beside those of the previous
// kernel where the split suits both.  Catalogs whose rebuild has a thread per variant (19 or 27 KB a CTA) ask for 32 KB
// with every kernel around it, else the driver's choice.  Of 64 x 256 variants the rebuild's CTAs shared the few
// SMs that the selection's did not occupy with the driver's choice, 64 KB or 100 KB (64 CTAs on 14 SMs, a window of
// 65,536 queries 17.6 us), and have an SM each with 32 KB (13.4 us).  The rebuild of larger tasks (41 KB and 22 bytes
// per variant) does not fit into 32 KB: it would wait until the selection's SMs are empty and split anew, a window
// of 20,000 queries, 32 KB / driver's choice, us: 64 x 600 variants 19.0 / 18.3, 64 x 1000 on a trade-off surface 26.6 /
// 25.7, 33 x 1100 32.3 / 27.6 and 36.3 / 30.7.
// 32 KB also hold one CTA of the rebuild at a time, so more than 148 tasks run in waves of one CTA per SM.
constexpr uint32_t REBUILD_THREAD_MAX = 512u;   // largest task whose rebuild has a thread per variant
constexpr int SPLIT_32K = 14;                   // per cent
constexpr int SPLIT_DRIVER = cudaSharedmemCarveoutDefault;
inline int split_for(const DeviceCatalog &c) { return c.max_task_variants <= REBUILD_THREAD_MAX ? SPLIT_32K : SPLIT_DRIVER; }
template <class... P, class... A>
inline cudaError_t launch_chained_cluster(void (*kernel)(P...), uint32_t grid, uint32_t cluster, uint32_t block, size_t smem,
                                          int split, cudaStream_t stream, A... args) {
  cudaLaunchAttribute attr[3] = {};
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  uint32_t n = 1;
  if (split != SPLIT_DRIVER) {
    attr[n].id = cudaLaunchAttributePreferredSharedMemoryCarveout;
    attr[n++].val.sharedMemCarveout = (unsigned)split;
  }
  if (cluster > 1) {
    attr[n].id = cudaLaunchAttributeClusterDimension;
    attr[n].val.clusterDim.x = cluster;
    attr[n].val.clusterDim.y = attr[n].val.clusterDim.z = 1;
    ++n;
  }
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cfg.attrs = attr;
  cfg.numAttrs = n;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}
template <class... P, class... A>
inline cudaError_t launch_chained(void (*kernel)(P...), uint32_t grid, uint32_t block, size_t smem, int split,
                                  cudaStream_t stream, A... args) {
  return launch_chained_cluster(kernel, grid, 1, block, smem, split, stream, args...);
}

// Launchers (host).  All are asynchronous on `stream` and allocate nothing.
cudaError_t launch_layout(const CatalogLayout &o, uint32_t n_tasks, uint32_t max_task_variants, cudaStream_t stream);
cudaError_t launch_rebuild(const DeviceCatalog &c, bool advance_queues, uint32_t window_us,
                           cudaStream_t stream);
cudaError_t launch_tally(const DeviceCatalog &c, const uint32_t *d_decision, uint64_t n,
                         int sm_count, cudaStream_t stream);
// Shared memory the launcher actually reserves for the image when asked for `image_smem`.
uint32_t select_image_smem(uint32_t image_smem);
// `image_smem`: bytes of dynamic shared memory reserved for the staged image (multiple of
// 16).  If the image is larger at run time the kernel reads it from global memory instead.
// `image_seen`: bytes of the image when the host last looked.
// `tally`: the kernel also adds the decisions to the pending per-variant counts and the
// catalog's counters (what launch_tally would do with them).
// Returns cudaErrorInvalidValue if n is too large for the launch geometry.
cudaError_t launch_select(const DeviceCatalog &c, const uint16_t *d_task, const uint32_t *d_slo,
                          const uint16_t *d_min_acc, uint64_t n, uint32_t *d_decision,
                          int sm_count, uint32_t image_smem, uint32_t image_seen, bool tally, cudaStream_t stream);
// Batches below this size are tallied by the selection kernel itself in infaas_select_update.  A window
// (select, tally, rebuild) with the fused / the separate tally, us: 64 tasks x 256 variants, 131,072
// queries 16.0 / 23.8, 196,000: 15.6 / 17.1, 262,143: 16.7 / 16.7; 128 x 512, 160,000: 14.4 / 19.6, 262,143:
// 18.7 / 21.3.  Few, hot variants would be better off without below it too (4 x 132, 131,072: 20.4 / 13.6,
// 262,143: 31.0 / 13.7): their counts are a few words that all atomics go to.
constexpr uint64_t FUSED_TALLY_MAX_N = 192 * 1024;

// Scaling-up step of the Model-Autoscaler for every task, from the pending per-variant
// counts; s_inst / s_arch / s_qps (floor(10^9 * batch / lat_us)) are per slot, task_slo per
// task; outputs have n_tasks entries.
cudaError_t launch_autoscale(const DeviceCatalog &c, const uint32_t *s_inst, const uint16_t *s_arch,
                             const unsigned long long *s_qps, const uint32_t *task_slo, uint32_t window_us, uint32_t slack_pct,
                             uint32_t lambda_milli, uint32_t *d_variant, uint32_t *d_delta,
                             cudaStream_t stream);

// Tables ordered by variant id, from and to the per-slot arrays.
struct LoadStateTail {
  unsigned long long counters[3];
  uint32_t err, image_bytes;
};
cudaError_t launch_load_state(const DeviceCatalog &c, const uint32_t *slot_of_id, LoadStateTail *tail,
                              unsigned long long *served, uint32_t *queued, uint32_t *pred, cudaStream_t stream);
cudaError_t launch_states(const DeviceCatalog &c, const uint32_t *slot_of_id, unsigned char *state, cudaStream_t stream);
// s_value[slot] = value_by_id[id] (0 without a table); with state_by_id also the states; with by_task
// also task_value[t] = by_task[t].
cudaError_t launch_scatter(const DeviceCatalog &c, const uint32_t *value_by_id, uint32_t *s_value,
                           const unsigned char *state_by_id, const uint32_t *by_task, uint32_t *task_value,
                           cudaStream_t stream);

// Worker choice.  Build: one worker per variant from the instance table {variant, worker, load}
// and the worker table {hardware code, utilisation} (device arrays); best_inst [n_variants] and
// best_hw [256] are scratch.  Assign: worker[q] = worker_of[decision[q]] for decisions below
// n_variants, INFAAS_INVALID otherwise.
cudaError_t launch_workers_build(uint32_t n_variants, const unsigned char *hw_by_id,
                                 const uint32_t *inst_variant, const uint32_t *inst_worker,
                                 const uint32_t *inst_load, uint32_t n_inst, const unsigned char *worker_hw,
                                 const uint32_t *worker_util, uint32_t n_workers,
                                 unsigned long long *best_inst, unsigned long long *best_hw,
                                 uint32_t *worker_of, cudaStream_t stream);
cudaError_t launch_assign_workers(const uint32_t *d_decision, uint64_t n, uint32_t n_variants,
                                  const uint32_t *worker_of, uint32_t *d_worker, int sm_count, int split,
                                  cudaStream_t stream);

// Integer-pipe probe: two CTAs per SM run `iters` steps of independent add / xor / compare /
// conditional-add chains; *lane_ops receives the number of lane-operations the launch executes.
cudaError_t launch_intpipe_probe(uint32_t iters, uint32_t seed, uint32_t *d_sink, int sm_count,
                                 unsigned long long *lane_ops, cudaStream_t stream);

// Remembers a CUDA error's text for infaas_last_cuda_error() (calling thread) and clears the
// runtime's error state; returns INFAAS_E_CUDA.
int record_cuda_error(cudaError_t e);

}  // namespace infaas
