// Paged KV pool: creation, seeding, per-step page reservation, KV append and
// release.  Pages are refcounted; a branched child shares its parent's pages
// (Section 3.1, after Eq. 3: the child inherits the parent's KV through prefix
// caching) and pruning frees only pages nobody else references.
//
// Allocation rule: the lowest free page id, slots served in ascending order,
// token by token.  Planners run as a single CTA with one thread per slot so
// the order is exactly that sequential rule.
#include <algorithm>
#include <cstring>
#include <mutex>
#include <set>
#include <tuple>
#include <vector>

#include "internal.cuh"
#include "step_form.cuh"

namespace gb {

static size_t align256(size_t x) { return (x + 255) & ~size_t(255); }

// One layer-step's new K (or V) rows.
static size_t new_rows_bytes(const gb_pool_config& c) {
  return (size_t)c.max_beams * c.num_kv_heads * c.head_dim * (c.kv_dtype == GB_BF16 ? 2 : 4);
}

MetaLayout meta_layout(const gb_pool_config& c) {
  MetaLayout m{};
  const size_t B = (size_t)c.max_beams;
  const int G = c.num_q_heads / c.num_kv_heads;
  size_t o = 0;
  auto take = [&](size_t bytes) { size_t at = o; o = align256(o + bytes); return at; };
  m.ctl = take(kCtlWords * sizeof(int));
  m.tables = take(B * c.max_pages_per_beam * sizeof(int));
  m.seq_len = take(B * sizeof(int));
  m.active = take(B * sizeof(int));
  m.gen = take(B * sizeof(int));
  m.nsteps = take(B * sizeof(int));
  m.mean = take(B * sizeof(float));
  m.lineage = take(B * sizeof(unsigned));
  m.refcnt = take((size_t)c.num_pages * sizeof(int));
  m.words = (int)((c.num_pages + 31) / 32);
  m.free_bits = take((size_t)m.words * sizeof(unsigned));
  m.plan = take(2 * 3 * (B + 1) * sizeof(int));
  m.cow = take(kMaxCowJobs * 3 * sizeof(int));
  m.cow_old = take(B * sizeof(int));
  m.record_floats = G * (c.head_dim + 2);
  m.partial_records = kMaxDecodeWarps + (int)B * c.num_kv_heads;  // record index: warp + b * Hkv + h
  m.partials = take((size_t)m.partial_records * m.record_floats * sizeof(float));
  const size_t BD = B * kMaxSegDepth;
  m.seg_cover = take(B * sizeof(int));
  m.seg_nseg = take(B * sizeof(int));
  m.seg_owner = take((size_t)c.num_pages * sizeof(unsigned long long));
  m.seg_i0 = take(BD * sizeof(int));
  m.seg_len = take(BD * sizeof(int));
  m.seg_rep = take(BD * sizeof(int));
  m.seg_g = take(BD * sizeof(int));
  m.seg_mem_off = take(BD * sizeof(int));
  m.seg_fill = take(BD * sizeof(int));
  m.seg_members = take(BD * sizeof(int));
  m.seg_tile_seg = take(B * kMaxSegRecords * sizeof(int));  // work entries <= records
  m.seg_tile_t = take(B * kMaxSegRecords * sizeof(int));
  m.grec = take(B * kMaxSegRecords * c.num_kv_heads * m.record_floats * sizeof(float));
  m.seg_bid = take(BD * sizeof(int));
  m.seg_rec_off = take(BD * sizeof(int));
  m.seg_nrec = take(B * sizeof(int));
  m.seg_splits = take(BD * sizeof(int));
  m.seg_tile_split = take(B * kMaxSegRecords * sizeof(int));
  m.seg_hist = take(2 * 256 * sizeof(int));
  m.pair_cnt = take(2 * B * c.num_kv_heads * sizeof(int));
  m.stats = take((size_t)kStatsRing * kStatsWords * sizeof(int));
  // Also holds a step's new K and V rows where the caller's output overlaps them.
  m.mlp_scratch = take(std::max((size_t)kMlpScratchFloats * sizeof(float), 2 * new_rows_bytes(c)));
  m.total = o;
  return m;
}

bool decode_supported(int dtype, int D, int G) {
  if (!(G == 2 || G == 4 || G == 8)) return false;
  if (dtype == GB_BF16) return D == 128;
  if (dtype == GB_F32) return D == 64;
  return false;
}

gb_status fail(gb_pool* pool, gb_status code, const char* what) {
  if (pool) pool->last_error = what;
  return code;
}

cudaError_t set_max_dynamic_smem(const void* kernel, int bytes) {
  static std::mutex mu;
  static std::set<std::tuple<const void*, int, int>> done;  // (kernel, device, bytes) already set
  int device = 0;
  cudaError_t e = cudaGetDevice(&device);
  if (e != cudaSuccess) return e;
  std::lock_guard<std::mutex> lock(mu);
  if (done.count(std::make_tuple(kernel, device, bytes))) return cudaSuccess;
  e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e == cudaSuccess) done.insert(std::make_tuple(kernel, device, bytes));
  return e;
}

gb_status check_launch(gb_pool* pool, const char* what) {
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) {
    if (pool) pool->last_error = std::string(what) + ": " + cudaGetErrorString(e);
    return GB_ERR_CUDA;
  }
  return GB_OK;
}

// ---------------------------------------------------------------------------
// Device helpers
// ---------------------------------------------------------------------------

// Block-wide search for the `need` lowest free pages, starting at the cursor
// word.  Writes them ascending into out[0..need).  Returns the number found
// (uniform).  Does not modify the bitmap.
__device__ int find_lowest_free(const PoolView& v, int need, int* out, int* tmp) {
  int found = 0;
  int w0 = v.ctl[kCtlCursor];
  if (w0 < 0) w0 = 0;
  while (found < need && w0 < v.words) {
    const int w = w0 + threadIdx.x;
    unsigned bits = w < v.words ? v.free_bits[w] : 0u;
    if (w == v.words - 1 && (v.num_pages & 31)) bits &= (1u << (v.num_pages & 31)) - 1u;
    int total;
    int r = found + block_exclusive_scan(__popc(bits), tmp, &total);
    while (bits && r < need) {
      const int bit = __ffs(bits) - 1;
      bits &= bits - 1u;
      out[r++] = w * 32 + bit;
    }
    found += total;
    w0 += blockDim.x;
  }
  __syncthreads();
  return found < need ? found : need;
}

// Take pages out[0..n) from the free set (bitmap, count, cursor).
__device__ void take_pages(const PoolView& v, const int* pages, int n) {
  for (int r = threadIdx.x; r < n; r += blockDim.x) {
    const int p = pages[r];
    atomicAnd(&v.free_bits[p >> 5], ~(1u << (p & 31)));
  }
  if (threadIdx.x == 0 && n > 0) {
    v.ctl[kCtlFree] -= n;
    v.ctl[kCtlCursor] = pages[n - 1] >> 5;
  }
  __syncthreads();
}

// ---------------------------------------------------------------------------
// Kernels
// ---------------------------------------------------------------------------

__global__ void k_init(PoolView v) {
  pdl_wait();
  pdl_launch_dependents();
  const long long tid = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  const long long stride = (long long)gridDim.x * blockDim.x;
  for (long long w = tid; w < v.words; w += stride) {
    unsigned bits = 0xffffffffu;
    if (w == v.words - 1 && (v.num_pages & 31)) bits = (1u << (v.num_pages & 31)) - 1u;
    v.free_bits[w] = bits;
  }
  for (long long i = tid; i < (long long)v.max_beams * v.max_pages; i += stride) v.tables[i] = -1;
  for (long long i = tid; i < 2LL * v.max_beams * v.Hkv; i += stride) v.pair_cnt[i] = 0;
  if (tid == 0) {
    for (int i = 0; i < kCtlWords; ++i) v.ctl[i] = 0;
    v.ctl[kCtlNextLineage] = 1;
    v.ctl[kCtlFree] = (int)v.num_pages;
  }
}

// Reserve the prompt's pages for n root beams (one CTA).
__global__ void __launch_bounds__(1024) k_seed_alloc(PoolView v, int n_beams, int prompt_len) {
  pdl_wait();
  pdl_launch_dependents();
  __shared__ int tmp[33];
  __shared__ int s_pages[2048];
  const int npg = (prompt_len + v.P - 1) / v.P;
  if (npg > v.max_pages || npg > 2048 || npg > v.ctl[kCtlFree]) {
    if (threadIdx.x == 0) { set_status(v.ctl, GB_ERR_OOM); v.ctl[kCtlStepOk] = 0; }
    return;
  }
  const int got = find_lowest_free(v, npg, s_pages, tmp);
  if (got < npg) {
    if (threadIdx.x == 0) set_status(v.ctl, GB_ERR_OOM);
    return;
  }
  take_pages(v, s_pages, npg);
  for (int i = threadIdx.x; i < npg; i += blockDim.x) v.refcnt[s_pages[i]] = n_beams;
  for (int i = threadIdx.x; i < n_beams * npg; i += blockDim.x)
    v.tables[(size_t)(i / npg) * v.max_pages + (i % npg)] = s_pages[i % npg];
  const int lin0 = v.ctl[kCtlNextLineage];
  __syncthreads();
  for (int b = threadIdx.x; b < n_beams; b += blockDim.x) {
    v.seq_len[b] = prompt_len;
    v.active[b] = 1;
    v.gen[b] = 0;
    v.nsteps[b] = 0;
    v.mean[b] = 0.f;
    v.lineage[b] = (unsigned)(lin0 + b);
  }
  if (threadIdx.x == 0) {
    v.ctl[kCtlNextLineage] = lin0 + n_beams;
    v.ctl[kCtlTailShared] = 1;  // the prompt's last page may be partial
  }
}

// Copy the prompt's K/V ([layer][T][Hkv][D]) into the pages listed in slot 0's table.
__global__ void k_seed_write(PoolView v, int prompt_len, const char* kp, const char* vp) {
  pdl_wait();
  pdl_launch_dependents();
  const int vec_per_row = v.D * v.esize / 16;
  const long long rows = (long long)v.layers * prompt_len * v.Hkv;
  const long long total = rows * vec_per_row * 2;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total;
       i += (long long)gridDim.x * blockDim.x) {
    const int kv = (int)(i / (rows * vec_per_row));
    long long r = i % (rows * vec_per_row);
    const int vec = (int)(r % vec_per_row);
    r /= vec_per_row;
    const int head = (int)(r % v.Hkv);
    r /= v.Hkv;
    const int t = (int)(r % prompt_len);
    const int layer = (int)(r / prompt_len);
    const int page = v.tables[t / v.P];
    if (page < 0 || page >= v.num_pages) continue;
    const char* src = (kv ? vp : kp) + ((((long long)layer * prompt_len + t) * v.Hkv + head) * v.D) * v.esize;
    char* dst = v.kv + kv_elem_offset(v, layer, page, kv, head, t % v.P) * v.esize;
    reinterpret_cast<uint4*>(dst)[vec] = reinterpret_cast<const uint4*>(src)[vec];
  }
}

// Open a step of n_tokens tokens for every active slot (one CTA, thread = slot):
// reserve pages in the sequential order (token by token, slots ascending),
// copy still-shared partial tail pages, advance lengths, build decode plans.
// All or nothing: if the pool cannot supply every page the step is a no-op.
__global__ void __launch_bounds__(1024) k_step_begin(PoolView v, int n_tokens, const int* seg_cover) {
  pdl_wait();
  pdl_launch_dependents();
  __shared__ int tmp[33];
  __shared__ int s_alloc[kMaxBeams];
  __shared__ int s_tail[kMaxBeams];
  __shared__ int s_act[kMaxBeams], s_cow[kMaxBeams];  // active slots, slots that copy their tail page
  constexpr int kTailHashBits = 11, kTailHash = 1 << kTailHashBits;
  static_assert(kTailHash >= 2 * kMaxBeams, "a probe always finds its page or a free entry");
  __shared__ int s_hkey[kTailHash], s_hmax[kTailHash];
  __shared__ int s_ncow, s_len;
  __shared__ int s_tok[2];
  __shared__ int s_ctl[8];  // free pages, steps, and the segment totals of the step record
  const int b = threadIdx.x;
  // Every load that depends on nothing else goes out first, together.
  const bool act = b < v.max_beams && v.active[b] != 0;
  const int L = act ? v.seq_len[b] : 0;
  const int cover = (seg_cover != nullptr && b < v.max_beams) ? seg_cover[b] : 0;
  if (b == 0) {
    s_ncow = 0;
    s_len = 0;
    s_tok[0] = s_tok[1] = 0;
    s_ctl[0] = v.ctl[kCtlFree];
    s_ctl[1] = v.ctl[kCtlSteps];
    s_ctl[2] = v.ctl[kCtlSegRowTok];
    s_ctl[3] = v.ctl[kCtlSegTileTok];
    s_ctl[4] = v.ctl[kCtlSegCount];
    s_ctl[5] = v.ctl[kCtlSegTiles];
    s_ctl[6] = v.ctl[kCtlSegTok];
    s_ctl[7] = v.ctl[kCtlTailShared];
  }

  // Copy-on-write decision for a still-shared partial tail page: holders decide in slot order
  // against the current refcount, so every holder but the highest slot copies.  Only after a seed
  // or a fork can a partial tail page be shared; the first step after one resolves them all.  The
  // highest holder of each page comes from a hash table in shared memory (a scan over the other
  // slots' pages took up to 10 us for 256 slots).
  __syncthreads();
  const bool tails_shared = s_ctl[7] != 0;
  int tail = -1;
  bool cow = false;
  if (tails_shared) {
    if (act && (L % v.P) != 0) tail = v.tables[(size_t)b * v.max_pages + L / v.P];
    const int R = tail >= 0 ? v.refcnt[tail] : 0;
    for (int i = b; i < kTailHash; i += blockDim.x) {
      s_hkey[i] = -1;
      s_hmax[i] = -1;
    }
    s_tail[b] = tail;
    __syncthreads();
    int at = 0;
    if (R > 1) {
      at = (int)(((unsigned)tail * 2654435761u) >> (32 - kTailHashBits));
      for (;;) {  // fewer pages than entries, so a probe ends
        const int k = atomicCAS(&s_hkey[at], -1, tail);
        if (k == -1 || k == tail) break;
        at = (at + 1) & (kTailHash - 1);
      }
      atomicMax(&s_hmax[at], b);
    }
    __syncthreads();
    cow = R > 1 && s_hmax[at] > b;
  }
  // Pages this slot needs over the whole step, and the table capacity check.
  int need_total = 0;
  bool too_long = false;
  if (act) {
    const int first_new = (L + v.P - 1) / v.P;        // first page index that needs a fresh page
    const int last_idx = (L + n_tokens - 1) / v.P;    // page index of the last new token
    need_total = (last_idx >= first_new ? last_idx - first_new + 1 : 0) + (cow ? 1 : 0);
    too_long = last_idx >= v.max_pages;
  }
  int total_need, nact;
  if (act) s_len = L;  // any active slot's length
  block_exclusive_scan(need_total, tmp, &total_need);
  const int arank = block_exclusive_scan(act ? 1 : 0, tmp, &nact);
  const bool any_too_long = __syncthreads_or(too_long);
  if (any_too_long || total_need > s_ctl[0]) {
    if (b == 0) v.ctl[kCtlCowJobs] = 0;
    if (b == 0) { set_status(v.ctl, GB_ERR_OOM); v.ctl[kCtlStepOk] = 0; }
    return;
  }

  // The sequential rule takes the lowest free page at every need, token by token and slots
  // ascending; nothing is freed in between, so the r-th need of the step gets the r-th lowest free
  // page.  Beams of one length (all advance together and a child takes its parent's length; only a
  // child of a released slot starts at 0) need their pages at the same tokens, so need r is copy r of the first
  // ncow, then page j = (r - ncow) / nact of active slot (r - ncow) % nact, and one pass over the
  // bitmap places them all.  (A pass per token with its block barriers took 88 us for 256 beams x
  // 199 tokens.)  Other states take the sequential form below.
  const bool uniform = !__syncthreads_or(act && L != s_len);
  if (uniform) {
    int ncow;
    const int cr = block_exclusive_scan(cow ? 1 : 0, tmp, &ncow);
    if (cow) s_cow[cr] = b;
    if (act) s_act[arank] = b;
    if (cow) atomicSub(&v.refcnt[tail], 1);
    __syncthreads();
    const int len = s_len, first_new = (len + v.P - 1) / v.P;
    int found = 0, w0 = max(v.ctl[kCtlCursor], 0);
    while (found < total_need && w0 < v.words) {
      const int w = w0 + b;
      unsigned bits = w < v.words ? v.free_bits[w] : 0u;
      if (w == v.words - 1 && (v.num_pages & 31)) bits &= (1u << (v.num_pages & 31)) - 1u;
      int total;
      int r = found + block_exclusive_scan(__popc(bits), tmp, &total);
      const unsigned before = bits;
      while (bits && r < total_need) {
        const int page = w * 32 + __ffs(bits) - 1;
        bits &= bits - 1u;
        int slot, idx;
        if (r < ncow) {  // copy-on-write of a shared tail page
          slot = s_cow[r];
          idx = len / v.P;
          v.cow[3 * r] = s_tail[slot];
          v.cow[3 * r + 1] = page;
          v.cow[3 * r + 2] = len % v.P;
        } else {
          const int j = (r - ncow) / nact;
          slot = s_act[r - ncow - j * nact];
          idx = first_new + j;
        }
        v.refcnt[page] = 1;
        v.tables[(size_t)slot * v.max_pages + idx] = page;
        if (++r == total_need) v.ctl[kCtlCursor] = w;
      }
      if (bits != before) v.free_bits[w] = (v.free_bits[w] & ~before) | bits;
      found += total;
      w0 += blockDim.x;
    }
    if (b == 0) {
      s_ncow = ncow;
      if (total_need > 0) v.ctl[kCtlFree] = s_ctl[0] - total_need;
    }
    if (found < total_need) {  // cannot happen after the count check
      if (b == 0) { set_status(v.ctl, GB_ERR_OOM); v.ctl[kCtlStepOk] = 0; }
      return;
    }
    __syncthreads();
  } else {
    for (int k = 0; k < n_tokens; ++k) {
      const int pos = L + k;
      const bool need_new = act && (pos % v.P) == 0;
      const bool need = need_new || (k == 0 && cow);
      if (!__syncthreads_or(need)) continue;
      int n_need;
      const int rank = block_exclusive_scan(need ? 1 : 0, tmp, &n_need);
      const int got = find_lowest_free(v, n_need, s_alloc, tmp);
      if (got < n_need) {  // cannot happen after the count check; keep the pool consistent
        if (b == 0) { set_status(v.ctl, GB_ERR_OOM); v.ctl[kCtlStepOk] = 0; }
        return;
      }
      take_pages(v, s_alloc, n_need);
      if (need) {
        const int page = s_alloc[rank];
        v.refcnt[page] = 1;
        v.tables[(size_t)b * v.max_pages + pos / v.P] = page;
        if (!need_new) {  // copy-on-write of the shared tail page
          atomicSub(&v.refcnt[tail], 1);
          const int j = atomicAdd(&s_ncow, 1);
          if (j < kMaxCowJobs) {
            v.cow[3 * j] = tail;
            v.cow[3 * j + 1] = page;
            v.cow[3 * j + 2] = L % v.P;
          }
        }
      }
      __syncthreads();
    }
  }
  // The rows [0, L % P) of each copied page are copied layer by layer by the kernel that writes
  // the layer's new rows: the append kernel from the job list, the attention launch from cow_old.
  if (b == 0) v.ctl[kCtlCowJobs] = min(s_ncow, kMaxCowJobs);
  if (b < v.max_beams) v.cow_old[b] = cow ? tail : -1;

  const int Lnew = act ? L + n_tokens : 0;
  if (act) {
    v.seq_len[b] = Lnew;
    v.gen[b] += n_tokens;
  }
  // Decode plans: mode 0 reads every token per beam; mode 1 skips the prefix
  // covered by grouped shared-prefix segments.
  int chunks[2];
#pragma unroll
  for (int mode = 0; mode < 2; ++mode) {
    int start = 0;
    if (mode == 1 && act) start = cover * v.P;
    if (start > Lnew) start = Lnew;
    const int n = act ? (Lnew - start + kChunk - 1) / kChunk : 0;
    const int toks = __reduce_add_sync(0xffffffffu, act ? Lnew - start : 0);
    if ((b & 31) == 0) atomicAdd(&s_tok[mode], toks);  // read after the scan's barriers
    int total;
    const int off = block_exclusive_scan(n * v.Hkv, tmp, &total);
    if (b < v.max_beams) {
      plan_off(v, mode)[b] = off;
      plan_n(v, mode)[b] = n;
      plan_start(v, mode)[b] = start;
    }
    if (b == 0) plan_off(v, mode)[v.max_beams] = total;
    chunks[mode] = total;
  }
  // The last warp, while the first writes the step's record.
  if (b >> 5 == (int)(blockDim.x >> 5) - 1 && v.dtype == GB_BF16 && v.D == 128)
    choose_forms(v, chunks[0], chunks[1], nact, s_ctl[3], s_ctl[5], s_ctl[4], s_ctl[6]);
  if (b == 0) {
    // Work of this step: tokens each path reads per KV head, and the segment work of the
    // grouped path (valid until the next rebuild).
    const int step = s_ctl[1];
    int* e = v.stats + (size_t)(step % kStatsRing) * kStatsWords;
    e[0] = s_tok[0];
    e[1] = s_tok[1];
    e[2] = v.grouped ? s_ctl[2] : 0;
    e[3] = v.grouped ? s_ctl[3] : 0;
    e[4] = v.grouped ? s_ctl[4] : 0;
    e[5] = v.grouped ? s_ctl[5] : 0;
    e[6] = n_tokens;
    e[7] = step;
    e[8] = v.grouped ? s_ctl[6] : 0;
    e[9] = nact;
    v.ctl[kCtlSteps] = step + 1;
    v.ctl[kCtlActive] = nact;
  }
  if (b == 0) {
    if (tails_shared) v.ctl[kCtlTailShared] = 0;
    v.ctl[kCtlStepOk] = 1;
  }
}

// Write n_tokens new K/V rows per active slot for one layer at positions
// [seq_len - n_tokens, seq_len).  kin/vin: [n_tokens][max_beams][Hkv][D].
__global__ void k_append(PoolView v, int layer, int n_tokens, const char* kin, const char* vin) {
  pdl_wait();
  pdl_launch_dependents();
  // Both counter sets of the attention launches (Counters): the previous attention launch has
  // completed (pdl_wait), and this layer's own, which would alternate them, does not come.
  if (blockIdx.x == 0 && blockIdx.y == 0) {
    zero_counters(v, 0, 0, 1);
    zero_counters(v, 1, 0, 1);
  }
  if (v.ctl[kCtlStepOk] == 0) return;
  const int vec_per_row = v.D * v.esize / 16;
  // Copy-on-write of still-shared partial tail pages, this layer's rows [0, rows).
  // Rows differ from every row written below, so both loops run concurrently.
  const int ncow = v.ctl[kCtlCowJobs];
  const long long per_job = 2LL * v.Hkv * v.P * vec_per_row;
  const long long nthreads = (long long)gridDim.x * gridDim.y * blockDim.x;
  for (long long i = ((long long)blockIdx.y * gridDim.x + blockIdx.x) * blockDim.x + threadIdx.x; i < per_job * ncow;
       i += nthreads) {
    const int j = (int)(i / per_job);
    long long r = i % per_job;
    const int vec = (int)(r % vec_per_row); r /= vec_per_row;
    const int row = (int)(r % v.P); r /= v.P;
    if (row >= v.cow[3 * j + 2]) continue;
    const int head = (int)(r % v.Hkv);
    const int kv = (int)(r / v.Hkv);
    const uint4* src = reinterpret_cast<const uint4*>(v.kv + kv_elem_offset(v, layer, v.cow[3 * j], kv, head, row) * v.esize);
    uint4* dst = reinterpret_cast<uint4*>(v.kv + kv_elem_offset(v, layer, v.cow[3 * j + 1], kv, head, row) * v.esize);
    dst[vec] = src[vec];
  }
  // New rows.  blockIdx.y walks (page of the new range, K|V), blockIdx.x the slots: one CTA writes
  // the new tokens of one page of one beam, all heads, so the slot's state and its page id are read
  // once for up to P tokens, the source is read in rows of Hkv * 256 contiguous bytes, and a
  // thread's loads (four at a time) are independent.  A thread per 16-byte piece that looked its
  // own page up ran at 3.8 TB/s of reads and writes (110 us for 256 beams x 199 tokens x 2 KiB).
  const int runs = (n_tokens + v.P - 1) / v.P + 1;
  for (int y = blockIdx.y; y < 2 * runs; y += gridDim.y) {
    const int kv = y & 1;
    for (int b = blockIdx.x; b < v.max_beams; b += gridDim.x) {
      if (!v.active[b]) continue;
      const int L = v.seq_len[b], pos0 = L - n_tokens;
      if (pos0 < 0) continue;
      const int pi = pos0 / v.P + (y >> 1);
      const int t0 = max(pos0, pi * v.P), t1 = min(L, (pi + 1) * v.P);
      if (t0 >= t1) continue;
      const int page = v.tables[(size_t)b * v.max_pages + pi];
      if (page < 0 || page >= v.num_pages) {
        if (threadIdx.x == 0) set_status(v.ctl, GB_ERR_INVALID);
        continue;
      }
      const int row16 = v.Hkv * 16;  // 16-byte pieces of one token (a head's row is 256 bytes)
      const uint4* src = reinterpret_cast<const uint4*>(kv ? vin : kin) + ((size_t)(t0 - pos0) * v.max_beams + b) * row16;
      uint4* dst = reinterpret_cast<uint4*>(v.kv + kv_elem_offset(v, layer, page, kv, 0, t0 - pi * v.P) * v.esize);
      const size_t tok_stride = (size_t)v.max_beams * row16;
      const int count = (t1 - t0) * row16;
      for (int i0 = threadIdx.x; i0 < count; i0 += 4 * blockDim.x) {
        uint4 x[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int i = i0 + u * blockDim.x;
          if (i < count) x[u] = __ldcs(src + (size_t)(i / row16) * tok_stride + i % row16);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int i = i0 + u * blockDim.x;
          const int t = i / row16, r = i - t * row16;
          if (i < count) dst[((r >> 4) * v.P + t) * 16 + (r & 15)] = x[u];
        }
      }
    }
  }
}

// Release listed slots (one CTA), 1024 entries of the list at a time.  An entry is taken when its
// slot is in range, active, and not named by an earlier entry; the first entry that is not decides
// the status, as if they were processed in order.  Each taken slot's references are dropped by a
// warp of its own (one slot after another took 2 us each, most of it two dependent loads).
__global__ void __launch_bounds__(1024) k_release(PoolView v, const int* slots, int n) {
  pdl_wait();
  pdl_launch_dependents();
  __shared__ int s_first[kMaxBeams];  // first entry of this part of the list that names the slot
  __shared__ int s_take[1024];
  __shared__ int s_bad;               // (entry << 3) | code of the first bad entry
  const int tid = threadIdx.x;
  for (int base = 0; base < n; base += 1024) {
    s_first[tid] = 0x7fffffff;
    if (tid == 0) s_bad = 0x7fffffff;
    __syncthreads();
    const int s = base + tid < n ? slots[base + tid] : -1;
    const bool in = base + tid < n && s >= 0 && s < v.max_beams;
    if (in) atomicMin(&s_first[s], tid);
    __syncthreads();
    const bool take = in && s_first[s] == tid && v.active[s];
    if (base + tid < n && !take) atomicMin(&s_bad, (tid << 3) | (in ? GB_ERR_STATE : GB_ERR_INVALID));
    s_take[tid] = take ? s : -1;
    __syncthreads();
    if (tid == 0 && s_bad != 0x7fffffff) set_status(v.ctl, s_bad & 7);
    for (int i = tid >> 5; i < min(1024, n - base); i += 32) {
      const int t = s_take[i];
      if (t < 0) continue;
      const int npg = (v.seq_len[t] + v.P - 1) / v.P;
      for (int j = tid & 31; j < npg; j += 32) {
        const int p = v.tables[(size_t)t * v.max_pages + j];
        if (p >= 0 && p < v.num_pages) unref_page(v, p);
      }
    }
    __syncthreads();
    if (take) {
      v.active[s] = 0;
      v.seq_len[s] = 0;
      v.gen[s] = 0;
    }
    __threadfence_block();
    __syncthreads();
  }
}

__global__ void k_clear_status(PoolView v) {
  pdl_wait();
  pdl_launch_dependents(); v.ctl[kCtlStatus] = GB_OK; }

}  // namespace gb

using namespace gb;

// ---------------------------------------------------------------------------
// C ABI
// ---------------------------------------------------------------------------

static gb_status validate(const gb_pool_config* c) {
  if (!c) return GB_ERR_INVALID;
  if (c->num_layers < 1 || c->num_q_heads < 1 || c->num_kv_heads < 1 ||
      c->num_q_heads % c->num_kv_heads != 0 || c->head_dim < 1 || c->num_pages < 1 ||
      c->num_pages > (int64_t)0x7fffffff || c->max_beams < 1 || c->max_beams > kMaxBeams ||
      c->max_pages_per_beam < 1 || c->group_min_beams < 0)
    return GB_ERR_INVALID;
  if (!(c->page_size == 16 || c->page_size == 32 || c->page_size == 64)) return GB_ERR_INVALID;
  if (c->kv_dtype != GB_F32 && c->kv_dtype != GB_BF16) return GB_ERR_INVALID;
  if (!decode_supported(c->kv_dtype, c->head_dim, c->num_q_heads / c->num_kv_heads))
    return GB_ERR_UNSUPPORTED;
  return GB_OK;
}

static size_t kv_bytes_of(const gb_pool_config* c) {
  const size_t es = c->kv_dtype == GB_BF16 ? 2 : 4;
  return (size_t)c->num_layers * (size_t)c->num_pages * 2 * c->num_kv_heads * c->page_size *
         c->head_dim * es;
}

extern "C" gb_status gb_pool_workspace_bytes(const gb_pool_config* cfg, size_t* kv_bytes,
                                             size_t* meta_bytes) {
  gb_status st = validate(cfg);
  if (st != GB_OK) return st;
  if (kv_bytes) *kv_bytes = kv_bytes_of(cfg);
  if (meta_bytes) *meta_bytes = meta_layout(*cfg).total;
  return GB_OK;
}

extern "C" gb_status gb_pool_init(const gb_pool_config* cfg, void* kv_dev, void* meta_dev,
                                  gb_stream_t stream, gb_pool** out) {
  if (!out) return GB_ERR_INVALID;
  *out = nullptr;
  gb_status st = validate(cfg);
  if (st != GB_OK) return st;
  if (!kv_dev || !meta_dev || ((uintptr_t)kv_dev & 255) || ((uintptr_t)meta_dev & 255))
    return GB_ERR_INVALID;
  gb_pool* p = new gb_pool();
  p->cfg = *cfg;
  p->layout = meta_layout(*cfg);
  if (cudaGetDevice(&p->device) != cudaSuccess ||
      cudaDeviceGetAttribute(&p->num_sms, cudaDevAttrMultiProcessorCount, p->device) != cudaSuccess) {
    delete p;
    return GB_ERR_CUDA;
  }
  p->decode_warps = std::min(kMaxDecodeWarps, p->num_sms * kDecodeCtasPerSm * kDecodeWarps);
  p->next_layer = 0;
  p->step_tokens = 0;
  p->seeded = false;
  p->group_min = cfg->group_min_beams > 0 ? cfg->group_min_beams : 2;
  PoolView& v = p->view;
  v.layers = cfg->num_layers;
  v.Hq = cfg->num_q_heads;
  v.Hkv = cfg->num_kv_heads;
  v.D = cfg->head_dim;
  v.P = cfg->page_size;
  v.G = v.Hq / v.Hkv;
  v.dtype = cfg->kv_dtype;
  v.esize = cfg->kv_dtype == GB_BF16 ? 2 : 4;
  v.max_beams = cfg->max_beams;
  v.max_pages = cfg->max_pages_per_beam;
  v.words = p->layout.words;
  v.num_pages = cfg->num_pages;
  v.kv = static_cast<char*>(kv_dev);
  v.page_elems = 2LL * v.Hkv * v.P * v.D;
  char* m = static_cast<char*>(meta_dev);
  const MetaLayout& L = p->layout;
  v.ctl = reinterpret_cast<int*>(m + L.ctl);
  v.tables = reinterpret_cast<int*>(m + L.tables);
  v.seq_len = reinterpret_cast<int*>(m + L.seq_len);
  v.active = reinterpret_cast<int*>(m + L.active);
  v.gen = reinterpret_cast<int*>(m + L.gen);
  v.nsteps = reinterpret_cast<int*>(m + L.nsteps);
  v.mean = reinterpret_cast<float*>(m + L.mean);
  v.lineage = reinterpret_cast<unsigned*>(m + L.lineage);
  v.refcnt = reinterpret_cast<int*>(m + L.refcnt);
  v.free_bits = reinterpret_cast<unsigned*>(m + L.free_bits);
  v.plan = reinterpret_cast<int*>(m + L.plan);
  v.cow = reinterpret_cast<int*>(m + L.cow);
  v.cow_old = reinterpret_cast<int*>(m + L.cow_old);
  v.partials = reinterpret_cast<float*>(m + L.partials);
  v.record_floats = L.record_floats;
  v.seg_cover = reinterpret_cast<int*>(m + L.seg_cover);
  v.seg_nseg = reinterpret_cast<int*>(m + L.seg_nseg);
  v.seg_owner = reinterpret_cast<unsigned long long*>(m + L.seg_owner);
  v.seg_i0 = reinterpret_cast<int*>(m + L.seg_i0);
  v.seg_len = reinterpret_cast<int*>(m + L.seg_len);
  v.seg_rep = reinterpret_cast<int*>(m + L.seg_rep);
  v.seg_g = reinterpret_cast<int*>(m + L.seg_g);
  v.seg_mem_off = reinterpret_cast<int*>(m + L.seg_mem_off);
  v.seg_fill = reinterpret_cast<int*>(m + L.seg_fill);
  v.seg_members = reinterpret_cast<int*>(m + L.seg_members);
  v.seg_tile_seg = reinterpret_cast<int*>(m + L.seg_tile_seg);
  v.seg_tile_t = reinterpret_cast<int*>(m + L.seg_tile_t);
  v.grec = reinterpret_cast<float*>(m + L.grec);
  v.seg_bid = reinterpret_cast<int*>(m + L.seg_bid);
  v.seg_rec_off = reinterpret_cast<int*>(m + L.seg_rec_off);
  v.seg_nrec = reinterpret_cast<int*>(m + L.seg_nrec);
  v.seg_splits = reinterpret_cast<int*>(m + L.seg_splits);
  v.seg_tile_split = reinterpret_cast<int*>(m + L.seg_tile_split);
  v.seg_hist = reinterpret_cast<int*>(m + L.seg_hist);
  v.pair_cnt = reinterpret_cast<int*>(m + L.pair_cnt);
  v.num_sms = p->num_sms;
  v.stats = reinterpret_cast<int*>(m + L.stats);
  v.mlp_scratch = reinterpret_cast<float*>(m + L.mlp_scratch);
  v.group_min = p->group_min;
  // The grouped tensor-core path needs bf16 K/V with D = 128 (kind::f16 MMAs, 128-byte rows)
  // and pages of 8 to 64 tokens that tile a 64-token K/V tile exactly.
  v.grouped = (cfg->kv_dtype == GB_BF16 && cfg->head_dim == 128 && cfg->page_size % 8 == 0 &&
               64 % cfg->page_size == 0)
                  ? 1
                  : 0;
  make_kv_tensor_maps(p);
  // The grouped path runs as a role of the attention kernel beside the per-beam role, so it
  // needs both tensor maps.
  if (v.grouped && !(p->have_tmap && p->have_dtmap && p->num_sms * kMmaWarps <= kMaxDecodeWarps)) v.grouped = 0;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  if (cudaMemsetAsync(m, 0, L.partials, s) != cudaSuccess ||
      cudaMemsetAsync(m + L.seg_cover, 0, L.seg_owner - L.seg_cover, s) != cudaSuccess ||
      cudaMemsetAsync(m + L.seg_owner, 0, (size_t)cfg->num_pages * sizeof(unsigned long long), s) != cudaSuccess) {
    delete p;
    return GB_ERR_CUDA;
  }
  p->launches += 1;
  k_init<<<std::max(1, std::min(p->num_sms * 4, (int)((v.max_beams * (long long)v.max_pages + 255) / 256))), 256, 0, s>>>(v);
  st = check_launch(p, "init");
  if (st != GB_OK) {
    delete p;
    return st;
  }
  *out = p;
  return GB_OK;
}

extern "C" gb_status gb_pool_destroy(gb_pool* pool) {
  delete pool;
  return GB_OK;
}

extern "C" const char* gb_last_error(gb_pool* pool) {
  return pool ? pool->last_error.c_str() : "";
}

extern "C" gb_status gb_pool_seed(gb_pool* pool, int n_beams, int prompt_len, const void* k_prompt_dev,
                                  const void* v_prompt_dev, gb_stream_t stream) {
  if (!pool) return GB_ERR_INVALID;
  if (pool->seeded) return fail(pool, GB_ERR_STATE, "seed: pool already seeded");
  if (n_beams < 1 || n_beams > pool->cfg.max_beams || prompt_len < 1 || !k_prompt_dev || !v_prompt_dev)
    return fail(pool, GB_ERR_INVALID, "seed: bad arguments");
  if ((prompt_len + pool->cfg.page_size - 1) / pool->cfg.page_size > 2048)
    return fail(pool, GB_ERR_UNSUPPORTED, "seed: prompt longer than 2048 pages");
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  k_seed_alloc<<<1, 1024, 0, s>>>(pool->view, n_beams, prompt_len);
  pool->launches += 2;
  gb_status st = check_launch(pool, "seed_alloc");
  if (st != GB_OK) return st;
  const long long vecs = 2LL * pool->cfg.num_layers * prompt_len * pool->cfg.num_kv_heads *
                         (pool->view.D * pool->view.esize / 16);
  const int grid = (int)std::min<long long>((vecs + 255) / 256, pool->num_sms * 8LL);
  k_seed_write<<<std::max(grid, 1), 256, 0, s>>>(pool->view, prompt_len,
                                                 static_cast<const char*>(k_prompt_dev),
                                                 static_cast<const char*>(v_prompt_dev));
  st = check_launch(pool, "seed_write");
  if (st != GB_OK) return st;
  pool->seeded = true;
  if (rebuild_segments(pool, s) != cudaSuccess) return check_launch(pool, "segments");
  return GB_OK;
}

// Shared by gb_decode_attention and gb_append_kv: open the step at layer 0 and write the new
// rows of `layer`, unless the attention launch that follows writes them itself (`fused`).
static gb_status append_layer(gb_pool* pool, int layer, int n_tokens, const void* k, const void* v, bool fused,
                              cudaStream_t s) {
  if (!pool->seeded) return fail(pool, GB_ERR_STATE, "pool not seeded");
  if (layer < 0 || layer >= pool->cfg.num_layers || n_tokens < 1 || !k || !v)
    return fail(pool, GB_ERR_INVALID, "append: bad arguments");
  if (layer != pool->next_layer) return fail(pool, GB_ERR_STATE, "layers of a step must be called in order");
  if (layer == 0) {
    prof_begin(pool, GB_PROF_PLAN, s);
    // One thread per slot (rounded up to a warp): the planner's block scans span only the pool's slots.
    launch_pdl(k_step_begin, 1, std::max(32, (pool->cfg.max_beams + 31) / 32 * 32), 0, s, pool->view, n_tokens,
               pool->view.grouped ? pool->view.seg_cover : nullptr);
    prof_end(pool, GB_PROF_PLAN, s);
    pool->launches += 1;
    gb_status st = check_launch(pool, "step_begin");
    if (st != GB_OK) return st;
    pool->step_tokens = n_tokens;
  } else if (n_tokens != pool->step_tokens) {
    return fail(pool, GB_ERR_STATE, "token count differs from the one layer 0 reserved");
  }
  const int runs = (n_tokens + pool->cfg.page_size - 1) / pool->cfg.page_size + 1;  // pages a beam's new tokens meet
  const dim3 grid(pool->cfg.max_beams, std::min(2 * runs, 65535));
  prof_begin(pool, GB_PROF_APPEND, s);  // an empty interval when the attention launch appends
  if (!fused) {
    launch_pdl(k_append, grid, 256, 0, s, pool->view, layer, n_tokens, static_cast<const char*>(k),
               static_cast<const char*>(v));
    pool->launches += 1;
  }
  prof_end(pool, GB_PROF_APPEND, s);
  gb_status st = check_launch(pool, "append");
  if (st != GB_OK) return st;
  pool->next_layer = (layer + 1) % pool->cfg.num_layers;
  return GB_OK;
}

extern "C" gb_status gb_append_kv(gb_pool* pool, int layer, int n_tokens, const void* k_dev,
                                  const void* v_dev, gb_stream_t stream) {
  if (!pool) return GB_ERR_INVALID;
  return append_layer(pool, layer, n_tokens, k_dev, v_dev, false, reinterpret_cast<cudaStream_t>(stream));
}

static bool overlap(const void* a, size_t an, const void* b, size_t bn) {
  const char *x = static_cast<const char*>(a), *y = static_cast<const char*>(b);
  return x < y + bn && y < x + an;
}

extern "C" gb_status gb_decode_attention(gb_pool* pool, int layer, const void* q_dev,
                                         const void* k_new_dev, const void* v_new_dev, float scale,
                                         float* out_dev, int flags, gb_stream_t stream) {
  if (!pool) return GB_ERR_INVALID;
  if (!q_dev || !out_dev) return fail(pool, GB_ERR_INVALID, "decode: null pointer");
  if (flags < GB_PATH_AUTO || flags > GB_PATH_GROUPED) return fail(pool, GB_ERR_INVALID, "decode: bad flags");
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  gb_status st = append_layer(pool, layer, 1, k_new_dev, v_new_dev, true, s);
  if (st != GB_OK) return st;
  // The launch writes a pair's output while other pairs' new rows are still to be read.
  const size_t rows = new_rows_bytes(pool->cfg);
  const size_t outb = (size_t)pool->cfg.max_beams * pool->cfg.num_q_heads * pool->cfg.head_dim * sizeof(float);
  if (overlap(out_dev, outb, k_new_dev, rows) || overlap(out_dev, outb, v_new_dev, rows)) {
    char* copy = reinterpret_cast<char*>(pool->view.mlp_scratch);
    if (cudaMemcpyAsync(copy, k_new_dev, rows, cudaMemcpyDeviceToDevice, s) != cudaSuccess ||
        cudaMemcpyAsync(copy + rows, v_new_dev, rows, cudaMemcpyDeviceToDevice, s) != cudaSuccess)
      return check_launch(pool, "new rows");
    k_new_dev = copy;
    v_new_dev = copy + rows;
  }
  // Mode 1: shared-prefix segments go through the grouped tensor-core kernel and the
  // per-beam kernel reads only each beam's remainder; mode 0: every beam reads everything.
  // In mode 1 one attention kernel runs both: the grouped and the per-beam roles on their
  // shares of the SMs (decode_ctas), or one after the other on every SM.
  const int mode = (flags == GB_PATH_PER_BEAM || !pool->view.grouped) ? 0 : 1;
  prof_begin(pool, GB_PROF_ATTENTION, s);
  if (launch_decode(pool, layer, q_dev, k_new_dev, v_new_dev, scale, out_dev, mode, flags != GB_PATH_GROUPED, s) !=
      cudaSuccess)
    return check_launch(pool, "decode");
  return check_launch(pool, "decode");
}

extern "C" gb_status gb_release(gb_pool* pool, const int32_t* slots_dev, int n, gb_stream_t stream) {
  if (!pool) return GB_ERR_INVALID;
  if (n < 0 || (n > 0 && !slots_dev)) return fail(pool, GB_ERR_INVALID, "release: bad arguments");
  if (pool->next_layer != 0) return fail(pool, GB_ERR_STATE, "release inside an open step");
  if (n == 0) return GB_OK;
  k_release<<<1, 1024, 0, reinterpret_cast<cudaStream_t>(stream)>>>(pool->view, slots_dev, n);
  pool->launches += 1;
  gb_status st = check_launch(pool, "release");
  if (st != GB_OK) return st;
  if (rebuild_segments(pool, reinterpret_cast<cudaStream_t>(stream)) != cudaSuccess)
    return check_launch(pool, "segments");
  return GB_OK;
}

extern "C" gb_status gb_pool_status(gb_pool* pool, int* device_status, gb_stream_t stream) {
  if (!pool || !device_status) return GB_ERR_INVALID;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  int v = 0;
  if (cudaMemcpyAsync(&v, pool->view.ctl + kCtlStatus, sizeof(int), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
      cudaStreamSynchronize(s) != cudaSuccess)
    return check_launch(pool, "status");
  *device_status = v;
  return GB_OK;
}

extern "C" gb_status gb_pool_set_profile_events(gb_pool* pool, int which, void* start_event, void* stop_event) {
  if (!pool || which < 0 || which >= GB_PROF_SLOTS) return GB_ERR_INVALID;
  pool->prof_start[which] = static_cast<cudaEvent_t>(start_event);
  pool->prof_stop[which] = static_cast<cudaEvent_t>(stop_event);
  return GB_OK;
}

extern "C" gb_status gb_pool_read_step_stats(gb_pool* pool, int32_t* out, int max_steps, int* n_out,
                                             gb_stream_t stream) {
  if (!pool || !out || !n_out || max_steps < 0) return GB_ERR_INVALID;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  std::vector<int> ring((size_t)kStatsRing * kStatsWords);
  int steps = 0;
  if (cudaMemcpyAsync(&steps, pool->view.ctl + kCtlSteps, sizeof(int), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
      cudaMemcpyAsync(ring.data(), pool->view.stats, ring.size() * sizeof(int), cudaMemcpyDeviceToHost, s) !=
          cudaSuccess ||
      cudaStreamSynchronize(s) != cudaSuccess)
    return check_launch(pool, "read_step_stats");
  const int n = std::min({max_steps, steps, kStatsRing});
  for (int i = 0; i < n; ++i) {
    const int step = steps - n + i;
    std::memcpy(out + (size_t)i * kStatsWords, ring.data() + (size_t)(step % kStatsRing) * kStatsWords,
                kStatsWords * sizeof(int));
  }
  *n_out = n;
  return GB_OK;
}

extern "C" gb_status gb_pool_launch_count(gb_pool* pool, uint64_t* count) {
  if (!pool || !count) return GB_ERR_INVALID;
  *count = pool->launches;
  return GB_OK;
}

extern "C" gb_status gb_pool_wait_selftest(gb_pool* pool, gb_stream_t stream) {
  if (!pool) return GB_ERR_INVALID;
  if (launch_wait_selftest(pool, reinterpret_cast<cudaStream_t>(stream)) != cudaSuccess)
    return check_launch(pool, "wait_selftest");
  pool->launches += 1;
  return check_launch(pool, "wait_selftest");
}

extern "C" gb_status gb_pool_clear_status(gb_pool* pool, gb_stream_t stream) {
  if (!pool) return GB_ERR_INVALID;
  k_clear_status<<<1, 1, 0, reinterpret_cast<cudaStream_t>(stream)>>>(pool->view);
  pool->launches += 1;
  return check_launch(pool, "clear_status");
}

extern "C" gb_status gb_pool_read_state(gb_pool* pool, const gb_pool_state* st, gb_stream_t stream) {
  if (!pool || !st) return GB_ERR_INVALID;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  const PoolView& v = pool->view;
  const size_t B = (size_t)v.max_beams;
  struct Copy { void* dst; const void* src; size_t bytes; } copies[] = {
      {st->tables, v.tables, B * v.max_pages * sizeof(int)},
      {st->seq_len, v.seq_len, B * sizeof(int)},
      {st->active, v.active, B * sizeof(int)},
      {st->gen, v.gen, B * sizeof(int)},
      {st->nsteps, v.nsteps, B * sizeof(int)},
      {st->mean, v.mean, B * sizeof(float)},
      {st->lineage, v.lineage, B * sizeof(unsigned)},
      {st->refcnt, v.refcnt, (size_t)v.num_pages * sizeof(int)},
      {st->free_bits, v.free_bits, (size_t)v.words * sizeof(unsigned)},
      {st->seg_cover, v.seg_cover, B * sizeof(int)},
      {st->seg_nseg, v.seg_nseg, B * sizeof(int)},
  };
  for (const Copy& c : copies) {
    if (!c.dst) continue;
    if (cudaMemcpyAsync(c.dst, c.src, c.bytes, cudaMemcpyDeviceToHost, s) != cudaSuccess)
      return check_launch(pool, "read_state");
  }
  if (cudaStreamSynchronize(s) != cudaSuccess) return check_launch(pool, "read_state");
  return GB_OK;
}
