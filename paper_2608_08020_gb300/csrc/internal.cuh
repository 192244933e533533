// Internal definitions shared by the library's translation units.
#pragma once

#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <stdint.h>
#include <string>
#include <utility>

#include "gambit.h"

namespace gb {

constexpr int kMaxBeams = 1024;    // slots per pool (one thread per slot in the planners)
constexpr int kChunk = 16;         // tokens per split-KV work unit (a page is 1..4 chunks)
constexpr int kDecodeWarps = 8;    // warps per CTA of the split-KV decode kernel (one CTA per SM)
constexpr int kDecodeStages = 3;   // TMA ring depth per warp
constexpr int kDecodeCtasPerSm = 1;
constexpr int kMaxDecodeWarps = 4096;
#ifndef GB_MMA_WARPS
#define GB_MMA_WARPS 12  // warps per CTA of the warp-MMA per-beam kernel (one CTA per SM)
#endif
constexpr int kMmaWarps = GB_MMA_WARPS;
constexpr int kMaxCowJobs = 1024;
constexpr int kMaxSegDepth = 16;
constexpr int kMaxSegRecords = 48;  // grouped partial records per beam (segments x token splits)
constexpr int kStatsRing = 4096;   // steps kept in the step-stats ring
constexpr int kStatsWords = 10;  // words per step record of the step-stats ring
constexpr int kMlpScratchFloats = 320 * 128 * 128;  // K-split partials of the MLP scorer's first layer (20 MiB)

// Control words at the start of the metadata buffer.
enum Ctl : int {
  kCtlStatus = 0,      // first device-side error (GB_OK when none)
  kCtlStepOk = 1,      // 1 while the current decode step has its pages
  kCtlDone = 2,        // last-CTA-done ticket counter (reset by the last CTA)
  kCtlCursor = 3,      // lowest free-bitmap word that may hold a free page
  kCtlNextLineage = 4, // next lineage id to hand out
  kCtlFree = 5,        // number of free pages
  kCtlCowJobs = 6,     // copy-on-write jobs of the open step (rows copied by each layer's append)
  kCtlSegCount = 7,    // shared-prefix segments found by the last rebuild
  kCtlSegMembers = 8,  // (beam, depth) memberships handed out by the last rebuild
  kCtlSegTiles = 9,    // 128-row query tiles over all segments
  kCtlSegRowTok = 10,  // sum over segments of (query rows of one KV head) x tokens
  kCtlSegTileTok = 11, // sum over segments of (128-row tiles) x tokens
  kCtlSteps = 12,      // steps opened so far (index into the step-stats ring)
  kCtlSegSplit = 13,   // tokens per grouped work unit (segments are split along tokens)
  kCtlTeam = 14,       // warps per team of the local form this step takes on the default path, 0: the roles
                       // (an fp32 pool: of the last layer-step's team form, 0: the even split)
  kCtlTeamPerBeam = 15,  // the same on the per-beam path
  kCtlSegTok = 16,     // sum over segments of their tokens (the shared tokens the grouped path reads once)
  kCtlBarCount = 17,   // grid-barrier arrivals of the tournament kernel (only grows)
  kCtlActive = 18,     // active slots of the open step
  kCtlSegGen = 19,     // segment rebuilds so far (stamps the per-page claim words)
  kCtlSegAlloc = 20,   // words 20-21: (segments << 32 | member slots) handed out by the running rebuild
  kCtlTailShared = 22, // 1 when a partial tail page may be shared (set by seed and forks, cleared by the planner)
  kCtlCounters = 24,   // words 24-26 and 28-30: the two counter sets of the attention launches (Counters)
  kCtlWords = 32
};

// Control words of a call on caller-owned rows: its kernels record errors in kCtlStatus, the last one
// publishes that in kRowsStatus and clears it, so that no launch has to clear it first.
constexpr int kRowsStatus = 2;
constexpr int kRowsShare = 3;  // chunks per warp of the call

// Words of a counter set.
enum CounterWord : int {
  kCntGrpNext = 0,   // next grouped work unit to hand out
  kCntGrpDone = 1,   // grouped-role CTAs finished
  kCntPairNext = 2,  // next (beam, KV head) pair to merge
  kCntWords = 4
};

// Byte offsets of the metadata regions.
struct MetaLayout {
  size_t ctl, tables, seq_len, active, gen, nsteps, mean, lineage, refcnt, free_bits;
  size_t plan, cow, cow_old, partials, total, stats;
  // shared-prefix segments
  size_t seg_cover, seg_nseg, seg_owner, seg_i0, seg_len, seg_rep, seg_g, seg_mem_off, seg_fill, seg_members,
      seg_tile_seg, seg_tile_t, grec, seg_bid, seg_rec_off, seg_nrec, seg_splits, seg_tile_split, seg_hist, pair_cnt;
  int words;            // free-bitmap words
  size_t mlp_scratch;   // MLP scorer partial sums
  int partial_records;  // split-KV partial records
  int record_floats;    // floats per partial record: G*(D+2)
};

MetaLayout meta_layout(const gb_pool_config& c);

// Plain-old-data view of a pool passed by value to kernels.
struct PoolView {
  int layers, Hq, Hkv, D, P, G, dtype, esize, max_beams, max_pages, words;
  long long num_pages;
  char* kv;             // KV pool base
  long long page_elems; // elements of one (layer, page): 2*Hkv*P*D
  int* ctl;
  int* tables;          // [max_beams][max_pages]
  int* seq_len;
  int* active;
  int* gen;
  int* nsteps;
  float* mean;
  unsigned* lineage;
  int* refcnt;
  unsigned* free_bits;
  int* plan;            // [2 modes][3][max_beams + 1]: offsets, chunk counts, start tokens
  int* cow;             // [kMaxCowJobs][3] (old page, new page, rows) of the open step's copy-on-writes
  int* cow_old;         // [max_beams] the page a beam's tail page was copied from by the open step, or -1
  // Shared-prefix segments (rebuilt after seed, prune/branch and release):
  int grouped;          // 1 when the grouped tensor-core path exists for this pool's dtype/shape
  int group_min;        // segments need at least this many sharing beams
  int* seg_cover;       // [max_beams] leading full pages of the beam covered by segments
  int* seg_nseg;        // [max_beams] segments the beam belongs to (by depth)
  unsigned long long* seg_owner;  // [num_pages] claim word of a segment-start page: (rebuild gen << 32) | (segment id + 1)
  int* seg_i0;          // [segments] first table index
  int* seg_len;         // [segments] pages
  int* seg_rep;         // [segments] a member beam whose table lists the pages
  int* seg_g;           // [segments] member beams
  int* seg_mem_off;     // [segments] offset of its members
  int* seg_fill;        // [segments] members written so far
  int* seg_members;     // [memberships] beam * kMaxSegDepth + depth
  int* seg_tile_seg;    // [tiles] segment of each 128-row query tile
  int* seg_tile_t;      // [tiles] tile index within the segment
  int* seg_tile_split;  // [tiles] token split of the unit
  int* seg_splits;      // [segments] token splits of the segment
  int* seg_bid;         // [max_beams][kMaxSegDepth] segment id of the beam's k-th segment
  int* seg_rec_off;     // [max_beams][kMaxSegDepth] first grouped record of that segment
  int* seg_nrec;        // [max_beams] grouped records of the beam
  int* seg_hist;        // [2][256] work units per length bucket, and units placed per bucket (rebuild scratch)
  int num_sms;          // multiprocessors (sizes the grouped work split)
  float* grec;          // [max_beams][kMaxSegDepth][Hkv] grouped partial records
  int* stats;           // [kStatsRing][kStatsWords] work of recent steps (see gb_pool_read_step_stats)
  float* partials;
  int* pair_cnt;        // [2][max_beams * Hkv] per-beam records written for each (beam, KV head) by the
                        // running attention launch, one array per counter set (Counters)
  int record_floats;
  float* mlp_scratch;   // [kMlpScratchFloats] K-split partials of the MLP scorer
};

// Plan arrays: mode 0 = per-beam only, mode 1 = with grouped coverage.
__host__ __device__ inline int* plan_off(const PoolView& v, int mode) {
  return v.plan + (size_t)mode * 3 * (v.max_beams + 1);
}
__host__ __device__ inline int* plan_n(const PoolView& v, int mode) {
  return plan_off(v, mode) + (v.max_beams + 1);
}
__host__ __device__ inline int* plan_start(const PoolView& v, int mode) {
  return plan_off(v, mode) + 2 * (v.max_beams + 1);
}

// The counters of one attention launch (work queue, finished CTAs, records per pair).  There are
// two sets: launch n of a pool uses set n & 1 and zeroes the other one, which launch n - 1 used
// and launch n + 1 will, so no launch has to come between two attention launches to reset them.
// n counts layers: steps opened so far x layers + layer, so consecutive launches alternate; a
// layer appended without attention (k_append) zeroes both sets, and so does k_init.
struct Counters {
  int* c;     // words kCntGrpNext, kCntGrpDone, kCntPairNext
  int* pair;  // [max_beams * Hkv]
};
__device__ __forceinline__ Counters counters(const PoolView& v, int set) {
  return {v.ctl + kCtlCounters + kCntWords * set, v.pair_cnt + (size_t)set * v.max_beams * v.Hkv};
}
__device__ __forceinline__ int counter_set(const PoolView& v, int layer, int steps) {  // steps: v.ctl[kCtlSteps]
  return (steps * v.layers + layer) & 1;
}
// Zero set `set`, spread over the grid (`cta` of CTAs of this size).
__device__ __forceinline__ void zero_counters(const PoolView& v, int set, int cta, int nctas) {
  const Counters k = counters(v, set);
  for (int i = cta * (int)blockDim.x + (int)threadIdx.x; i < v.max_beams * v.Hkv; i += nctas * (int)blockDim.x)
    k.pair[i] = 0;
  if (cta == 0 && threadIdx.x < kCntWords) k.c[threadIdx.x] = 0;
}

#ifndef GB_DECODE_WEIGHT
#define GB_DECODE_WEIGHT 56  // relative cost of a per-beam token against a grouped tile token (percent)
#endif

#ifndef GB_SPLIT_BYTES_PER_SM
#define GB_SPLIT_BYTES_PER_SM (8ll << 20)
#endif

// A mode-1 step launches one attention kernel with a grouped and a per-beam role.  When the
// step's attention reads little per SM (below GB_SPLIT_BYTES_PER_SM), both roles are
// latency-bound and run side by side, each on its own share of the CTAs (one per SM): the
// per-beam role takes decode_ctas(v, grid) of them, in proportion to its (16-token chunk x
// KV head) tokens against the grouped role's (128-row tile x token) work per KV head, and
// the grouped role the rest.  Otherwise the per-beam CTAs follow the grouped ones onto the SMs
// they leave.  The roles and the merge compute the same split from the step's plan.
// A grouped unit costs about 256 tokens beside its own (its queries, its record).  Two CTAs more than
// the share, rounded up: where the tails are short the share is 7-15 CTAs and one too few costs 5% of
// the step.  Per layer-step (us), with weight 45, no unit term and the share rounded / now, for trees
// named by beams x tokens, prompt, tokens between rounds (and the per-beam tokens over the grouped
// ones): 98.5 / 61.2 (64 x 4090, 1000, 512; 0.04), 282 / 193 (198 x 8190, 1000, 512; 0.04), 229 / 182
// (198 x 7800, 512, 512; 0.11), 188 / 178 (90 x 9000, 2000, 1200, G = 8; 0.51), 215 / 206 (128 x 6100, 200,
// 1000; 0.63), 104 / 101 (300 x 3000, 50, 200, G = 2; 0.78).  No difference where the tails are a fair
// share: 69.3 / 68.9 (64 x 3900, 512, 512; 0.34), 114.5 / 114.4 (250 x 7000, 100, 700; 0.92), 117.5 / 117.4
// (120 x 12000, 1000, 2000, G = 8; 0.68).
__device__ __forceinline__ int decode_ctas(const PoolView& v, int grid);

// Element offset of row `row` of the K (kv=0) or V (kv=1) slab of (layer, page, head).
__device__ __forceinline__ long long kv_elem_offset(const PoolView& v, int layer, long long page,
                                                    int kv, int head, int row) {
  return ((((long long)layer * v.num_pages + page) * 2 + kv) * v.Hkv + head) * (long long)v.P * v.D +
         (long long)row * v.D;
}

// Programmatic dependent launch.  Every kernel of the library calls pdl_wait() before any global
// memory access but those named here: launched normally it returns at once; launched with
// programmatic stream serialization (launch_pdl) the kernel may be scheduled while the
// previous kernel in the stream is still running, and pdl_wait() blocks until that
// kernel has completed and its writes are visible - the same ordering as a plain launch,
// without the gap between the two kernels.  pdl_launch_dependents() lets the next
// kernel be scheduled as soon as every CTA of this one has called it or left; each kernel calls it
// only after its own pdl_wait, so all but the directly preceding kernel have completed when one starts.
// Before the wait, three kernels read what the directly preceding kernel cannot have written:
//   - k_attention and k_decode_mma of layers above 0: the step's control words, and in the small-step
//     form its plan, tables and first K/V chunks (enter, below);
//   - k_fused_gemm: its rows of the weights;
//   - k_gemm_partials with early_w: its first weight tiles (the scorer's, whose preceding kernel is one
//     of the scorer's).
// What a preceding kernel of the library writes (q, partial sums, activity) is read through pointers
// without __restrict__: const __restrict__ data may be read as constant for the kernel's whole life,
// which here begins before those writes.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Small attention steps (local.cuh) of layers above 0 begin before the previous kernel has
// completed: the step's plan, tables and every K/V row but the step's own were final when layer 0's
// launch began (each kernel of the library lets its dependents go only after its own pdl_wait, so
// all but the directly preceding kernel have completed by then, and no call between the layers of
// a step changes them), so page ids and the first K/V loads go out while the kernel that makes q
// and the new rows drains.  `early` threads wait here, before they read q, the new rows or the
// counters, and before any global write.  (The same in the roles of large steps gained nothing:
// the next launch's loads then compete with the tail of this one.)  How early depends on the kernel:
// k_decode_mma is one CTA per SM; of k_attention's 2 x SM CTAs the second half has nothing to do in the
// small-step form but must get an SM to say so, so the next launch begins as the first half leaves.
__device__ __forceinline__ void enter(bool early) {
  if (early) {
    pdl_wait();
    pdl_launch_dependents();
  }
}

__device__ __forceinline__ bool split_sms(const PoolView& v, long long td, long long tg) {
  const long long bytes = (td + tg) * 2 * v.D * v.esize;
  return td > 0 && tg > 0 && bytes < GB_SPLIT_BYTES_PER_SM * v.num_sms;
}
__device__ __forceinline__ int decode_ctas(const PoolView& v, int grid) {
  const long long td = (long long)plan_off(v, 1)[v.max_beams] * kChunk;  // tokens x KV heads
  const long long tg = (long long)v.ctl[kCtlSegTileTok] * v.Hkv;
  if (!split_sms(v, td, tg)) return grid;
  const long long wd = td * GB_DECODE_WEIGHT, wg = (tg + 256ll * v.ctl[kCtlSegTiles] * v.Hkv) * 100;
  long long n = (wd * grid + wd + wg - 1) / (wd + wg);
  if (2 * n < grid) n += 2;
  return (int)(n > grid - 1 ? grid - 1 : n);
}

__device__ __forceinline__ void set_status(int* ctl, int code) {
  atomicCAS(&ctl[kCtlStatus], GB_OK, code);
}

// Mark page p free (bitmap, allocation cursor, free count).
__device__ __forceinline__ void mark_free(const PoolView& v, int p) {
  atomicOr(&v.free_bits[p >> 5], 1u << (p & 31));
  atomicMin(&v.ctl[kCtlCursor], p >> 5);
  atomicAdd(&v.ctl[kCtlFree], 1);
}

// Drop one reference to page p; frees it when the count reaches zero.
__device__ __forceinline__ void unref_page(const PoolView& v, int p) {
  if (atomicSub(&v.refcnt[p], 1) == 1) mark_free(v, p);
}

// Block-wide exclusive scan of one int per thread (blockDim.x <= 1024, multiple of 32).
// `tmp` must hold 33 ints of shared memory.  Returns the exclusive prefix; *total gets the sum.
__device__ __forceinline__ int block_exclusive_scan(int x, int* tmp, int* total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
  int inc = x;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    int y = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += y;
  }
  if (lane == 31) tmp[warp] = inc;
  __syncthreads();
  if (warp == 0) {
    int w = lane < nwarps ? tmp[lane] : 0;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      int y = __shfl_up_sync(0xffffffffu, w, o);
      if (lane >= o) w += y;
    }
    if (lane < nwarps) tmp[lane] = w;  // inclusive warp totals
    if (lane == nwarps - 1) tmp[32] = w;
  }
  __syncthreads();
  int r = inc - x + (warp > 0 ? tmp[warp - 1] : 0);
  *total = tmp[32];
  __syncthreads();
  return r;
}

// Host side --------------------------------------------------------------------

// Launch with programmatic stream serialization (see pdl_wait).  Built with -DGB_NO_PDL
// it is a plain launch.
template <typename... KArgs, typename... Args>
inline cudaError_t launch_pdl(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                              Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
#ifndef GB_NO_PDL
  cfg.attrs = attr;
  cfg.numAttrs = 1;
#endif
  return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}

struct DecodeShape {
  int dtype, D, G;
};
bool decode_supported(int dtype, int D, int G);

}  // namespace gb

// The opaque host handle.
struct gb_pool {
  gb_pool_config cfg;
  gb::MetaLayout layout;
  gb::PoolView view;
  int device;
  int num_sms;
  int decode_warps;   // warps launched by the split-KV decode kernel
  int next_layer;     // layer expected by the next decode/append call (0 opens a step)
  int step_tokens;    // tokens reserved by the open step
  bool seeded;
  int group_min;
  int capacity = 0;   // the tree's capacity C for the tournament (0: max_beams)
  alignas(64) unsigned char tmap[128];      // CUtensorMap over the KV pool (grouped path)
  bool have_tmap = false;
  alignas(64) unsigned char dtmap[128];     // CUtensorMap over the KV pool (per-beam bf16 path)
  alignas(64) unsigned char dtmap_half[128];  // the same with an 8-token box (short tail chunks)
  bool have_dtmap = false;
  int tmap_oob = 0;                          // first row group past the tensor map (loads zeros)
  std::string last_error;
  unsigned long long launches = 0;          // kernels launched by this pool
  cudaEvent_t prof_start[GB_PROF_SLOTS] = {};  // caller-owned instrumentation events
  cudaEvent_t prof_stop[GB_PROF_SLOTS] = {};
};

namespace gb {
gb_status fail(gb_pool* pool, gb_status code, const char* what);

// Instrumentation: record the caller's event pair around one kernel, if set.  Under
// stream capture the records become external event nodes, so the events are recorded
// (and can be timed) each time the graph runs.
inline void prof_record(cudaEvent_t e, cudaStream_t s) {
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  cudaStreamIsCapturing(s, &cs);
  cudaEventRecordWithFlags(e, s, cs == cudaStreamCaptureStatusActive ? cudaEventRecordExternal : cudaEventRecordDefault);
}
inline void prof_begin(gb_pool* p, int which, cudaStream_t s) {
  if (p->prof_start[which]) prof_record(p->prof_start[which], s);
}
inline void prof_end(gb_pool* p, int which, cudaStream_t s) {
  if (p->prof_stop[which]) prof_record(p->prof_stop[which], s);
}
gb_status check_launch(gb_pool* pool, const char* what);
// Raise a kernel's dynamic shared memory limit to `bytes` on the current device.  The
// attribute belongs to the device, so it is set once per (kernel, device), under a lock.
cudaError_t set_max_dynamic_smem(const void* kernel, int bytes);


// Kernel launchers implemented in the other translation units.
// The attention of one layer-step on s, written to out: mode 0, the per-beam kernel; mode 1,
// the attention kernel with the grouped and per-beam roles (launch_attention).  Every kernel
// merges its records itself.
// The launch also writes the step's new rows into the pool.
cudaError_t launch_decode(gb_pool* pool, int layer, const void* q, const void* k_new, const void* v_new, float scale,
                          float* out, int mode, bool allow_local, cudaStream_t s);
cudaError_t launch_decode_view(const PoolView& v, int W, const void* q, float scale, float* out, cudaStream_t s);
cudaError_t rebuild_segments(gb_pool* pool, cudaStream_t s);
cudaError_t launch_forks(gb_pool* pool, const int32_t* parent_of, cudaStream_t s);
cudaError_t launch_attention(gb_pool* pool, int layer, const void* q, const void* k_new, const void* v_new, float scale,
                             float* out, bool allow_local, cudaStream_t s);
cudaError_t launch_wait_selftest(gb_pool* pool, cudaStream_t s);
void make_kv_tensor_maps(gb_pool* pool);
cudaError_t launch_probe(gb_pool* pool, const void* hidden, int hidden_dtype, int H, const float* w,
                         float bias, const uint8_t* mask, float* score_out, const float* scores_in,
                         cudaStream_t s);
// Split-K bf16 GEMM on the tensor cores (gemm.cu): P[s][m][n] over k-range s of A[m][k] B[n][k].
// early_w: B was not written by the kernel before this one in the stream, so its first loads need
// not wait for that kernel.
int gemm_splits(int M, int N, int K, int num_sms, size_t max_floats);
cudaError_t gemm_partials(const void* A, int M, const void* B, int N, int K, int splits, float* P, int* ctl,
                          bool early_w, cudaStream_t s);
cudaError_t launch_mlp(gb_pool* pool, const void* hidden, int H, const void* w1, const float* b1, const float* w2,
                       float b2, int dh, const uint8_t* mask, float* score_out, cudaStream_t s);
cudaError_t launch_prune_branch(gb_pool* pool, int K, int fanout, int warmup, const uint8_t* elig,
                                int32_t* parent_out, uint8_t* pruned_out, uint32_t* lineage_out,
                                cudaStream_t s);
}  // namespace gb
