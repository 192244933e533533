// The attention of a small step, merged inside each CTA.
//
// When a step's whole per-beam work is a few chunks per warp of the GPU, reading it is not what
// takes the time: the grouped role's set-up, the partial records in global memory and the waits of
// their merge are (a layer-step of 13 beams x 340 tokens took 21 us for 10 MB).  Here a team of
// w = 1, 2, 3, 4, 6 or 12 warps of one CTA takes a (beam, KV head) pair at a time, splits the beam's
// whole context (shared pages included: they come from L2) into w runs of chunks, and merges the
// warps' softmax states through shared memory: no records, no counters, no waits between CTAs.
// The arithmetic of a chunk is the per-beam role's (decode_mma.cuh), but for the probabilities, which
// enter P.V as two bf16 terms: a run of a few chunks rounded to one against its first chunk's maximum is up
// to 20% less exact than the roles, whose tiles hold 128 tokens and whose runs are other ones.  Which
// steps take this form is in step_form.cuh.
#pragma once
#include "decode_mma.cuh"

namespace gb {

__device__ __forceinline__ void team_sync(int team, int threads) {
  asm volatile("bar.sync %0, %1;" ::"r"(1 + team), "r"(threads) : "memory");
}

// All pairs of the pool by teams of w warps, CTA `cta` of `nctas`; kMmaWarps * 32 threads.  Shared memory: the warps'
// stages and barriers as in decode_mma_body; a warp's record for its team's merge lies over its
// own stages, which are idle by then.
template <int G>
__device__ __forceinline__ void local_attention(const PoolView& v, const CUtensorMap* tm_p, const CUtensorMap* tmh_p,
                                                int layer, const __nv_bfloat16* q, const NewRows& nw,
                                                float qscale, int w, int cta, int nctas,
                                                float* __restrict__ out, bool early) {
  using S = DecodeMmaSmem;
  constexpr int HS = 132;  // floats per head of a record: 128 and a pad, so that the stores below
                           // (4 head pairs x 8 rows) fall on 32 banks
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* smem = smem_raw + ((1024 - (smem_addr(smem_raw) & 1023)) & 1023);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int r = lane >> 2, c = lane & 3;
  const uint32_t stage0 = smem_addr(smem) + warp * kMmaStages * kMmaStageBytes;
  const uint32_t bar0 = smem_addr(smem) + S::STAGES + warp * kMmaStages * 8;
  static_assert((G * HS + 2 * G) * 4 <= kMmaStages * kMmaStageBytes, "a record fits the warp's stages");

  const int npairs = v.max_beams * v.Hkv;
  const int tpc = kMmaWarps / w, team = warp / w, wi = warp - team * w;

  if (lane == 0) {
    for (int s = 0; s < kMmaStages; ++s) mbar_init(bar0 + 8 * s, 1);
    fence_mbar_init();
  }
  __syncwarp();
  uint32_t koff[4], voff[4];
  ldsm_offsets(koff, voff, lane);
  const uint64_t pol = policy_evict_normal();  // siblings read the shared pages again
  const int pg8 = v.P >> 3, layer_pages = layer * v.num_pages;
  int stage = 0;
  uint32_t parity = 0;
  bool alive = true;  // false once a wait ran out: no more loads, the pairs' outputs are zero
  bool wait = early;  // the first pair's loads go out before the wait

  for (int p = cta + nctas * team; p < npairs; p += nctas * tpc) {
    const int b = p / v.Hkv, h = p - b * v.Hkv;
    const int n = plan_n(v, 0)[b], L = v.seq_len[b], old = v.cow_old[b];
    float* ob = out + ((size_t)b * v.Hq + (size_t)h * G) * 128;
    if (n == 0) {
      // Vacant slots: the run of them among the team's next 32 pairs at once, shared out among its warps
      // (1024 slots, 8 of them active: a round trip for each was 15 us of a layer-step's 24).
      enter(wait);
      wait = false;
      const int pl = p + lane * nctas * tpc;
      const bool end = pl >= npairs || plan_n(v, 0)[pl / v.Hkv] != 0;
      const unsigned ends = __ballot_sync(0xffffffffu, end);
      const int run = ends != 0 ? __ffs(ends) - 1 : 32;  // >= 1: this one
      for (int i = wi; i < run; i += w) {
        const int z = p + i * nctas * tpc;
        zero_pair<G>(v, z / v.Hkv, z % v.Hkv, out);
      }
      p += (run - 1) * nctas * tpc;
      continue;
    }
    const int i0 = wi * n / w, i1 = (wi + 1) * n / w;
    const int* tb = v.tables + (size_t)b * v.max_pages;
    const int tail = (L - 1) / v.P;
    const int special = old >= 0 ? tail * v.P / kChunk : n - 1;  // first chunk that is appended to or copied
    PairState st;
    uint4 nrow = make_uint4(0u, 0u, 0u, 0u);
    int npage = 0, pw = 0, pages = 0;
    auto load_pages = [&](int i) {  // lane l: the page of chunk i + l
      pw = i;
      const int pi = (i + lane) * kChunk / v.P;
      pages = i + lane >= i1 ? 0 : old >= 0 && pi == tail ? old : tb[pi];
    };
    auto issue = [&](int i, int s) {
      if (i >= pw + 32) load_pages(i);
      int page = __shfl_sync(0xffffffffu, pages, i - pw);
      if (lane == 0) {
        if (page < 0 || page >= v.num_pages) {
          set_status(v.ctl, GB_ERR_INVALID);
          page = 0;
        }
        const int tok = i * kChunk;
        const int wrow = ((layer_pages + page) * 2 * v.Hkv + h) * pg8 + ((tok & (v.P - 1)) >> 3);
        const bool half = i == n - 1 && L - tok <= 8;
        mbar_arrive_expect_tx(bar0 + 8 * s, half ? kMmaStageBytes / 2 : kMmaStageBytes);
        tma_chunk(stage0 + s * kMmaStageBytes, half ? tmh_p : tm_p, wrow, bar0 + 8 * s, pol);
      }
    };
    load_pages(i0);
    int ii = i0;  // next chunk to load
    for (int s = 0; s < kMmaStages && ii < i1 && alive; ++s, ++ii) issue(ii, (stage + s) % kMmaStages);
    enter(wait);
    wait = false;
    pair_begin<G, true>(st, v, q, b, h, r, c);
    if (i0 < i1 && i1 == n) {  // this warp holds the pair's last chunk
      nrow = (lane < 16 ? nw.k : nw.v)[(size_t)p * 16 + (lane & 15)];
      npage = tb[tail];
    }
    for (int i = i0; i < i1 && alive; ++i) {
      if (!mbar_wait_bounded(bar0 + 8 * stage, parity, kWaitLimitNs)) {
        if (lane == 0) set_status(v.ctl, GB_ERR_TIMEOUT);
        for (int s = 1; s < kMmaStages; ++s) {  // a bounded chance for the copies in flight
          const int k = stage + s;
          if (i + s < ii)
            mbar_wait_bounded(bar0 + 8 * (k % kMmaStages), parity ^ (k >= kMmaStages ? 1u : 0u), kWaitLimitNs / 4);
        }
        alive = false;
        break;
      }
      const int tok0 = i * kChunk, nvalid = min(kChunk, L - tok0);
      if (i >= special) {
        unsigned char* vs = smem + (stage0 + stage * kMmaStageBytes - smem_addr(smem));
        if (i == n - 1) chunk_append(v, layer, h, L, nvalid, nrow, npage, vs, lane);
        if (old >= 0) chunk_copied(v, layer, b, h, L, tok0, vs, lane);
      }
      chunk_attend<G, true>(st, stage0 + stage * kMmaStageBytes, koff, voff, nvalid, qscale, r, c);
      __syncwarp();
      if (ii < i1) {
        if (lane == 0) fence_proxy_async_smem();
        issue(ii++, stage);
      }
      if (++stage == kMmaStages) {
        stage = 0;
        parity ^= 1u;
      }
    }
    pair_finish<G, true>(st);
    if (w == 1) {
      if (2 * c < G) {
        float* o0 = ob + 2 * c * 128 + r;
#pragma unroll
        for (int mt = 0; mt < 8; ++mt) {
          o0[16 * mt] = alive ? st.o[mt][0] / st.l0 : 0.f;
          o0[16 * mt + 128] = alive ? st.o[mt][1] / st.l1 : 0.f;
          o0[16 * mt + 8] = alive ? st.o[mt][2] / st.l0 : 0.f;
          o0[16 * mt + 136] = alive ? st.o[mt][3] / st.l1 : 0.f;
        }
      }
      continue;
    }
    // The warp's record, then the team's merge (merge_team).
    __syncwarp();
    float* rec = reinterpret_cast<float*>(smem + warp * kMmaStages * kMmaStageBytes);
    if (2 * c < G) {
      float* o0 = rec + 2 * c * HS + r;
#pragma unroll
      for (int mt = 0; mt < 8; ++mt) {
        o0[16 * mt] = st.o[mt][0];
        o0[16 * mt + HS] = st.o[mt][1];
        o0[16 * mt + 8] = st.o[mt][2];
        o0[16 * mt + HS + 8] = st.o[mt][3];
      }
      if (r == 0) {
        rec[G * HS + 2 * c] = st.m0;
        rec[G * HS + 2 * c + 1] = st.m1;
        rec[G * HS + G + 2 * c] = alive ? st.l0 : -1.f;
        rec[G * HS + G + 2 * c + 1] = alive ? st.l1 : -1.f;
      }
    }
    team_sync(team, w * 32);
    merge_team<G, 128, HS>(reinterpret_cast<const float*>(smem + team * w * kMmaStages * kMmaStageBytes),
                           kMmaStages * kMmaStageBytes / 4, w, wi * 32 + lane, w * 32, ob);
    fence_proxy_async_smem();  // the records' memory is refilled by TMA for the next pair
    team_sync(team, w * 32);
  }
  enter(wait);
}

}  // namespace gb
