// The log-sum-exp merge of a layer-step's partial attention records, run at the end of the
// attention launch itself rather than as a launch of its own: with bounded waits (k_attention,
// k_decode_mma), as described here, or without any (k_decode_pool, merge_completed below).
//
// Each (beam b, KV head h) pair has R = nseg + npb records: on the grouped path, nseg records
// of the beam's shared-prefix segments, and npb split-KV records of the per-beam warps whose
// chunk range meets the pair's chunks (warp w's record of the pair is number w + b * Hkv + h).
// A grouped CTA counts itself in the launch's kCntGrpDone once all of its records are written; a
// per-beam warp counts each record it writes in pair[b * Hkv + h] (release: fence, then
// the add).  After its own work, every warp of the merging CTAs takes pairs from the counter
// kCntPairNext until none is left, so the warps that finish first take the pairs and the
// last ones to finish find none.  Per pair it folds the segment records first (a bounded wait
// until every grouped CTA has finished, long past on a large step), then waits (bounded) until
// pair[p] == npb and folds the split-KV records, so what remains after the pair's last
// record is one batch of loads: running max M of the records' m, acc = sum o * 2^(m - M),
// L = sum l * 2^(m - M), out[b][h * G + g][:] = acc / L.
//
// The waits end because every CTA they wait on gets an SM: the callers only let CTAs merge
// that are resident together with the ones they wait on, or that wait only on CTAs which never
// wait (k_attention).  Each wait is bounded and gives up as soon as the pool's status word is
// set.  The counters are one of two sets; a launch zeroes the other one (Counters, internal.cuh).
#pragma once
#include <cuda_runtime.h>
#include <math.h>
#include "internal.cuh"
#include "ptx.cuh"

namespace gb {

// A per-beam warp has written the record of pair bh: make the writes visible, then count it.
__device__ __forceinline__ void record_arrive(const Counters& k, int bh, int lane) {
  fence_acq_rel_gpu();
  __syncwarp();
  if (lane == 0) atomicAdd(&k.pair[bh], 1);
}

// A grouped CTA has written all of its records (called by every thread of the CTA).
__device__ __forceinline__ void grouped_cta_done(const Counters& k) {
  __syncthreads();
  if (threadIdx.x == 0) {
    fence_acq_rel_gpu();
    atomicAdd(&k.c[kCntGrpDone], 1);
  }
}

// Wait, with the whole warp polling, until pair p has npb split-KV records and ng grouped
// CTAs have finished.  False on a timeout or when an error status is set.
__device__ __forceinline__ bool wait_pair_records(const PoolView& v, const Counters& k, int p, int npb, int ng) {
  const uint64_t t0 = globaltimer_ns();
  unsigned ns = 32;
  while (true) {
    const int a = npb > 0 ? ld_acquire_gpu(&k.pair[p]) : 0;
    const int g = ng > 0 ? ld_acquire_gpu(&k.c[kCntGrpDone]) : 0;
    if (__all_sync(0xffffffffu, a >= npb && g >= ng)) return true;
    if (__any_sync(0xffffffffu, *reinterpret_cast<volatile int*>(&v.ctl[kCtlStatus]) != GB_OK ||
                                    globaltimer_ns() - t0 > kWaitLimitNs))
      return false;
    __nanosleep(ns);
    ns = ns < 512 ? 2 * ns : ns;
  }
}

// The running state of one pair's merge (one warp; lane l owns the float4 elements l + 32 j of the
// pair's G heads of D dims, so with D = 128 element j belongs to head j).
template <int G, int D>
struct MergeState {
  static constexpr int N = G * D / 128;
  float M[N], L[N];
  float4 acc[N];
};

template <int G, int D>
__device__ __forceinline__ void merge_init(MergeState<G, D>& st) {
#pragma unroll
  for (int g = 0; g < MergeState<G, D>::N; ++g) {
    st.M[g] = -INFINITY;
    st.L[g] = 0.f;
    st.acc[g] = make_float4(0.f, 0.f, 0.f, 0.f);
  }
}

// Fold the records rec0, rec0 + stride, ... (cnt of them) into the state.  The records exist:
// the caller waited for them.
template <int G, int D>
__device__ __forceinline__ void merge_fold(MergeState<G, D>& st, const float* rec0, size_t stride, int cnt) {
  constexpr int GD = G * D, N = MergeState<G, D>::N;
  constexpr int RB = N >= 8 ? 1 : 16 / N;  // records per batch of loads: 8-16 float4 in flight per lane
  const int lane = threadIdx.x & 31;
  for (int r0 = 0; r0 < cnt; r0 += RB) {
    float4 x[RB][N];
    float mk[RB][N], lk[RB][N];
#pragma unroll
    for (int k = 0; k < RB; ++k) {
      if (r0 + k < cnt) {
        // L2 loads: the records were written by other SMs during this launch.
        const float* rec = rec0 + (size_t)(r0 + k) * stride;
#pragma unroll
        for (int g = 0; g < N; ++g) {
          const int head = 4 * (lane + 32 * g) / D;
          x[k][g] = __ldcg(reinterpret_cast<const float4*>(rec) + lane + 32 * g);
          mk[k][g] = __ldcg(rec + GD + head);
          lk[k][g] = __ldcg(rec + GD + G + head);
        }
      } else {
#pragma unroll
        for (int g = 0; g < N; ++g) {
          x[k][g] = make_float4(0.f, 0.f, 0.f, 0.f);
          mk[k][g] = -INFINITY;  // a record that saw no token (or none at all) adds nothing
          lk[k][g] = 0.f;
        }
      }
    }
#pragma unroll
    for (int g = 0; g < N; ++g) {
      float mnew = st.M[g];
#pragma unroll
      for (int k = 0; k < RB; ++k) mnew = fmaxf(mnew, mk[k][g]);
      if (mnew == -INFINITY) continue;
      if (mnew > st.M[g]) {  // M = -inf the first time: acc and L are still 0
        const float a = st.M[g] == -INFINITY ? 0.f : exp2f(st.M[g] - mnew);
        st.acc[g].x *= a;
        st.acc[g].y *= a;
        st.acc[g].z *= a;
        st.acc[g].w *= a;
        st.L[g] *= a;
        st.M[g] = mnew;
      }
#pragma unroll
      for (int k = 0; k < RB; ++k) {
        const float sc = mk[k][g] == -INFINITY ? 0.f : exp2f(mk[k][g] - st.M[g]);
        st.acc[g].x = fmaf(x[k][g].x, sc, st.acc[g].x);
        st.acc[g].y = fmaf(x[k][g].y, sc, st.acc[g].y);
        st.acc[g].z = fmaf(x[k][g].z, sc, st.acc[g].z);
        st.acc[g].w = fmaf(x[k][g].w, sc, st.acc[g].w);
        st.L[g] = fmaf(lk[k][g], sc, st.L[g]);
      }
    }
  }
}

// out[b][h * G + g][:] = acc / L.
template <int G, int D>
__device__ __forceinline__ void merge_write(const PoolView& v, const MergeState<G, D>& st, int b, int h,
                                            float* __restrict__ out) {
  const int lane = threadIdx.x & 31;
  float* ob = out + ((size_t)b * v.Hq + (size_t)h * G) * D;
  const bool vec_out = (reinterpret_cast<uintptr_t>(out) & 15) == 0;
#pragma unroll
  for (int g = 0; g < MergeState<G, D>::N; ++g) {
    const float4 res = make_float4(st.acc[g].x / st.L[g], st.acc[g].y / st.L[g], st.acc[g].z / st.L[g],
                                   st.acc[g].w / st.L[g]);
    float* d = ob + 4 * (lane + 32 * g);
    if (vec_out) {
      *reinterpret_cast<float4*>(d) = res;
    } else {
      d[0] = res.x;
      d[1] = res.y;
      d[2] = res.z;
      d[3] = res.w;
    }
  }
}

// Zero the output rows of pair (b, h) (an inactive beam, or a failed wait).
template <int G, int D = 128>
__device__ __forceinline__ void zero_pair(const PoolView& v, int b, int h, float* __restrict__ out) {
  float* ob = out + ((size_t)b * v.Hq + (size_t)h * G) * D;
  for (int e = threadIdx.x & 31; e < G * D; e += 32) ob[e] = 0.f;
}

// A step that was refused (no pages) has no attention: its outputs are zero.
template <int G, int D = 128>
__device__ __forceinline__ void zero_all_pairs(const PoolView& v, int cta, int nctas, float* __restrict__ out) {
  const int nw = blockDim.x >> 5;
  for (int p = cta * nw + (int)(threadIdx.x >> 5); p < v.max_beams * v.Hkv; p += nctas * nw)
    zero_pair<G, D>(v, p / v.Hkv, p % v.Hkv, out);
}

// The merge phase of an attention launch, run by every warp of the merging CTAs after its own
// work: `mode` selects the plan (0 per-beam, 1 with segments), W = warps of the per-beam
// role, ng = CTAs of the grouped role (0 without one), out = [max_beams][Hq][128] fp32.
// `claim`: the warps take pairs from the counter kCntPairNext as they finish (for CTAs
// that start at different times) and fold a pair's segment records before they wait for its
// split-KV records; otherwise merging CTA `cta` of `nctas` takes the pairs
// p = cta + nctas * (warp + k * warps per CTA) and waits for all of a pair's records at once.
template <int G>
__device__ __forceinline__ void combine_pairs(const PoolView& v, const Counters& cnt, int mode, int W, int ng,
                                              bool claim, int cta, int nctas, float* __restrict__ out) {
  constexpr int D = 128;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int npairs = v.max_beams * v.Hkv;
  const int* off = plan_off(v, mode);
  const int* nn = plan_n(v, mode);
  const int Tot = off[v.max_beams];
  const int c = Tot > 0 ? (Tot + W - 1) / W : 1;  // chunks per per-beam warp
  const size_t rf = (size_t)v.record_floats;
  for (int k = 0;; ++k) {
    int p = cta + nctas * (warp + k * nw);
    if (claim) {
      if (lane == 0) p = atomicAdd(&cnt.c[kCntPairNext], 1);
      p = __shfl_sync(0xffffffffu, p, 0);
    }
    if (p >= npairs) break;
    const int b = p / v.Hkv, h = p - b * v.Hkv;
    const bool act = v.active[b] != 0;
    const int n = act ? nn[b] : 0;
    const int nseg = (act && mode == 1 && v.grouped) ? v.seg_nrec[b] : 0;
    const int o0 = off[b] + h * n;
    const int first = o0 / c;
    const int npb = n > 0 ? (o0 + n - 1) / c - first + 1 : 0;
    if (npb + nseg == 0) {
      zero_pair<G>(v, b, h, out);
      continue;
    }
    const float* grec = v.grec + ((size_t)b * kMaxSegRecords * v.Hkv + h) * rf;  // [b][record][Hkv]
    const float* prec = v.partials + (size_t)(first + p) * rf;                     // first + p, ...
    MergeState<G, D> st;
    merge_init(st);
    bool good;
    if (claim) {
      good = nseg == 0 || wait_pair_records(v, cnt, p, 0, ng);
      if (good && nseg > 0) merge_fold(st, grec, (size_t)v.Hkv * rf, nseg);
      good = good && (npb == 0 || wait_pair_records(v, cnt, p, npb, 0));
      if (good && npb > 0) merge_fold(st, prec, rf, npb);
    } else {
      good = wait_pair_records(v, cnt, p, npb, nseg > 0 ? ng : 0);
      if (good) {
        merge_fold(st, prec, rf, npb);
        merge_fold(st, grec, (size_t)v.Hkv * rf, nseg);
      }
    }
    if (good) {
      merge_write(v, st, b, h, out);
    } else {
      if (lane == 0) set_status(v.ctl, GB_ERR_TIMEOUT);  // kept if already set
      zero_pair<G, D>(v, b, h, out);
    }
  }
}

// Merge w records in shared memory, `stride` floats apart, into ob[g][:]: out = sum o 2^(m - M) /
// sum l 2^(m - M), threads t of nt.  A record holds head g's D values at g HS, its m at G HS + g and its l
// at G HS + G + g; one without tokens has m = -inf and l = 0, and one whose warp's wait ran out has
// l < 0 (its heads' outputs are zero).
template <int G, int D, int HS>
__device__ __forceinline__ void merge_team(const float* recs, int stride, int w, int t, int nt, float* __restrict__ ob) {
  for (int e = t; e < G * D / 4; e += nt) {
    const int g = 4 * e / D, d = 4 * e % D;
    float M = -INFINITY;
    bool good = true;
    for (int k = 0; k < w; ++k) {
      M = fmaxf(M, recs[k * stride + G * HS + g]);
      good = good && !(recs[k * stride + G * HS + G + g] < 0.f);
    }
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    float l = 0.f;
    for (int k = 0; k < w; ++k) {
      const float m = recs[k * stride + G * HS + g];
      if (m == -INFINITY) continue;
      const float sc = exp2f(m - M);
      const float4 x = *reinterpret_cast<const float4*>(recs + k * stride + g * HS + d);
      acc.x = fmaf(x.x, sc, acc.x);
      acc.y = fmaf(x.y, sc, acc.y);
      acc.z = fmaf(x.z, sc, acc.z);
      acc.w = fmaf(x.w, sc, acc.w);
      l = fmaf(recs[k * stride + G * HS + G + g], sc, l);
    }
    float* od = ob + 4 * e;
    od[0] = good ? acc.x / l : 0.f;
    od[1] = good ? acc.y / l : 0.f;
    od[2] = good ? acc.z / l : 0.f;
    od[3] = good ? acc.w / l : 0.f;
  }
}

// A pair of more records than this (two batches of merge_fold's loads) is merged by the whole CTA of the
// warp that completes it, see merge_long.
template <int G, int D>
constexpr int kMergeAlone = 2 * (MergeState<G, D>::N >= 8 ? 1 : 16 / MergeState<G, D>::N);

// The merge of a launch whose warps each took chunks [w c, w c + c) of the Tot chunks of the flat list
// (s_off, s_n: its offsets and chunks per beam), run by every warp after its own: no warp waits.  A
// warp counts itself at the first and the last pair of its range (release: fence, then the add), and the
// one that completes a pair's count merges the pair; the pairs between those two are its own.  `good`:
// the warp wrote all of its records; a pair that misses one gets zeros (the count's high half).  Pairs
// of many records are left in p_long (room for two a warp), counted in *n_long, for merge_long.
template <int G, int D>
__device__ __forceinline__ void merge_completed(const PoolView& v, const Counters& cnt, const int* s_off,
                                                const int* s_n, int Tot, int c, int w, bool good, int* n_long,
                                                int* p_long, float* __restrict__ out) {
  const int lane = threadIdx.x & 31;
  const int x0 = (int)min((long long)w * c, (long long)Tot), x1 = min(x0 + c, Tot);
  if (x0 >= x1) return;
  auto beam_of = [&](int x) {  // the beam of chunk x
    int lo = 0, hi = v.max_beams;  // invariant: s_off[lo] <= x < s_off[hi]
    while (hi - lo > 1) {
      const int mid = (lo + hi) >> 1;
      if (s_off[mid] <= x) lo = mid; else hi = mid;
    }
    return lo;
  };
  const int x = lane == 0 ? x0 : x1 - 1, lo = beam_of(x);
  auto records = [&](int b, int h, int* first) {
    const int n = s_n[b], o = s_off[b] + h * n;
    *first = o / c;
    return (o + n - 1) / c - *first + 1;
  };
  int h = (x - s_off[lo]) / s_n[lo], first;
  const int p = lo * v.Hkv + h, need = records(lo, h, &first);
  const int p0 = __shfl_sync(0xffffffffu, p, 0), p1 = __shfl_sync(0xffffffffu, p, 1);
  fence_acq_rel_gpu();  // this warp's records before its counts
  __syncwarp();
  int seen = 0;
  if (lane == 0 || (lane == 1 && p1 != p0)) seen = atomicAdd(&cnt.pair[p], good ? 1 : 0x10001);
  const bool last = (seen & 0xffff) == need - 1, bad = !good || (seen >> 16) != 0;
  const unsigned m_last = __ballot_sync(0xffffffffu, last), m_bad = __ballot_sync(0xffffffffu, bad);
  fence_acq_rel_gpu();  // the other warps' records after their counts
  int b = __shfl_sync(0xffffffffu, lo, 0);
  h = p0 - b * v.Hkv;
  for (int q = p0; q <= p1; ++q, ++h) {
    if (h == v.Hkv) {  // on to the next beam that has chunks
      b = beam_of(s_off[b + 1]);
      h = 0;
      q = b * v.Hkv;
    }
    const int l = q == p0 ? 0 : 1;  // the lane that counted this pair, at either end of the range
    const bool own = q != p0 && q != p1;
    if (!own && !((m_last >> l) & 1u)) continue;
    if (own ? !good : ((m_bad >> l) & 1u) != 0) {
      zero_pair<G, D>(v, b, h, out);
      continue;
    }
    const int npb = records(b, h, &first);
    if (npb > kMergeAlone<G, D>) {
      if (lane == 0) p_long[atomicAdd(n_long, 1)] = q;
      continue;
    }
    MergeState<G, D> st;
    merge_init(st);
    merge_fold(st, v.partials + (size_t)(first + q) * v.record_floats, (size_t)v.record_floats, npb);
    merge_write(v, st, b, h, out);
  }
}

// The pairs with many records, by the whole CTA (called by all of its threads after a barrier): each warp
// folds every Warps-th record, and the warps' states are merged through shared memory (recs, a record every
// `stride` floats).  With one warp folding them all, a step of one beam x 4000 tokens with 8 heads per KV
// head spent 60 of its 75 us here.
template <int G, int D, int Warps>
__device__ __forceinline__ void merge_long(const PoolView& v, const int* s_off, const int* s_n, int c, int n_long,
                                           const int* p_long, float* recs, int stride, float* __restrict__ out) {
  constexpr int GD = G * D;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int i = 0; i < n_long; ++i) {
    const int q = p_long[i], b = q / v.Hkv, h = q - b * v.Hkv, n = s_n[b], o = s_off[b] + h * n;
    const int first = o / c, npb = (o + n - 1) / c - first + 1;
    MergeState<G, D> st;
    merge_init(st);
    merge_fold(st, v.partials + (size_t)(first + q + warp) * v.record_floats, (size_t)Warps * v.record_floats,
               npb > warp ? (npb - warp + Warps - 1) / Warps : 0);
    float* rec = recs + warp * stride;
#pragma unroll
    for (int g = 0; g < MergeState<G, D>::N; ++g) {
      const int e = 4 * (lane + 32 * g);
      *reinterpret_cast<float4*>(rec + e) = st.acc[g];
      if (e % D == 0) {
        rec[GD + e / D] = st.M[g];
        rec[GD + G + e / D] = st.L[g];
      }
    }
    __syncthreads();
    merge_team<G, D, D>(recs, stride, Warps, (int)threadIdx.x, Warps * 32, out + (size_t)q * GD);
    __syncthreads();
  }
}

}  // namespace gb
