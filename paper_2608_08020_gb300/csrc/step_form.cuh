// Which form a decode step's attention takes (local.cuh): decided once per step by the planner, so that
// the launch of each layer reads one word.  Computed by every CTA of the launch, the choice's dozen
// divisions were on its critical path twice (the grid's second half starts when the first has left):
// 0.8 us of a small layer-step's 6.
#pragma once
#include "internal.cuh"

namespace gb {

// Warps per team for the local form of a step with `pairs` active (beam, KV head) pairs of `chunks`
// chunks each on `nctas` CTAs: 1, 2, 3, 4, 6 or 12, whichever minimises rounds of pairs x (chunks per
// warp + what a pair costs beside its chunks: page ids, query rows and the first load, then the merge
// of a team).  *cost gets that, in the time of a chunk.  Called by a whole warp.
__device__ __forceinline__ int local_team(int pairs, int chunks, int nctas, int* cost) {
  static_assert(kMmaWarps == 12, "team sizes divide the CTA's warps");
  const int lane = threadIdx.x & 31;
  unsigned key = 0xffffffffu;
  if (lane < 6) {
    const int w = lane < 4 ? lane + 1 : 6 * (lane - 3), teams = nctas * (kMmaWarps / w);
    key = (unsigned)(((pairs + teams - 1) / teams) * ((chunks + w - 1) / w + 3 + (w > 1 ? 1 : 0))) * 8u + (unsigned)lane;
  }
  key = __reduce_min_sync(0xffffffffu, key);
  const int i = (int)(key & 7u);
  *cost = (int)(key >> 3);
  return i < 4 ? i + 1 : 6 * (i - 3);
}

// Whether the local form beats the two roles on the default path.  Both times (us) are fits over 77
// layer-steps measured both ways (13 trees of 13 to 300 beams, G = 2 to 8, contexts 114 to 16836), per
// SM warp or SM: the local form 2.4 + 0.81 per unit of cost; the roles 12 + 1.6 per chunk they read +
// 3.8 per grouped unit + 0.18 per segment record of a pair and query head (their merge).  The choice
// loses 0.5% on average against the better of the two, 18% at worst (where both take 95-112 us);
// limits on the chunks alone lost 2.4% and 26%.  Local / roles, us: 12 / 25 (39 beams x 748 tokens),
// 32 / 37 (39 x 2057), 44 / 41 (39 x 2993), 46 / 47 (57 x 2880), 41 / 83 (256 x 313), 44 / 54
// (13 x 8979, G = 8), 52 / 39 (64 x 2565, prompt 1795).  Above 72 chunks per warp, outside the fits,
// the roles are ahead (256 x 1100 and up, 2% of a search).
__device__ __forceinline__ bool local_step(const PoolView& v, int all, int rest, int cost, int pairs, int seg_tile_tok,
                                           int seg_units) {
  const float sm = 1.f / v.num_sms, w = sm / kMmaWarps;
  if (all * w > 72.f) return false;
  const float tile = (float)seg_tile_tok * v.Hkv / kChunk, unit = tile / fmaxf((float)seg_units * v.Hkv, 1.f);
  const float records = unit > 0.f ? (float)(all - rest) / pairs / unit : 0.f;
  return 2.4f + 0.81f * cost < 12.f + 1.6f * (rest + tile) * w + 3.8f * seg_units * v.Hkv * sm + 0.18f * records * v.G;
}

// The same for the per-beam path, whose other form splits the whole contexts evenly over all warps
// of the GPU.  Where beams share pages, siblings of neighbouring teams read them at about the same
// time here, and from L2: 79 against 117 us per layer-step for 64 beams x 4000 tokens, 188 / 326
// (193 x 2962), 101 / 160 (40 x 8000, whose pairs fill 73% of the teams' rounds), 370 / 448
// (256 x 4000), 265 / 256-303 (152 x 4000).  So a tree whose beams share a third of their contexts
// takes this form unless uneven rounds cost it more than 1.6 times; one that shares little has
// nothing to gain but an even split.  A small step takes it unless its rounds are uneven (0.82 us per
// unit of cost against 1.2 per chunk and warp): 156 pairs 30 / 33 us at 18 chunks per warp, 41 / 41 at
// 26, 52 / 48 at 34.
__device__ __forceinline__ bool local_step_per_beam(const PoolView& v, int all, int rest, int cost, int seg_count,
                                                    int seg_tok) {
  const float a = (float)all / (kMmaWarps * v.num_sms);
  if (a <= 44.f && cost <= 16.f + 1.4f * a) return true;
  if (!v.grouped || seg_count == 0) return false;
  const long long unshared = rest + (long long)seg_tok * v.Hkv / kChunk;
  return 2ll * all >= 3 * unshared && cost <= 1.6f * (a + 6.f);
}

// The step's two forms: warps per team of the local form, or 0, on the default path and on the
// per-beam path.  all / rest: chunks x KV heads of the active beams' whole contexts and of what the
// segments leave.  Called by a whole warp, lane 0 writes.
__device__ __forceinline__ void choose_forms(const PoolView& v, int all, int rest, int nact, int seg_tile_tok, int seg_units,
                                             int seg_count, int seg_tok) {
  const int pairs = max(nact, 1) * v.Hkv;
  int cost;
  const int team = local_team(pairs, (all + pairs - 1) / pairs, v.num_sms, &cost);
  if ((threadIdx.x & 31) != 0) return;
  v.ctl[kCtlTeam] = local_step(v, all, rest, cost, pairs, seg_tile_tok, seg_units) ? team : 0;
  v.ctl[kCtlTeamPerBeam] = local_step_per_beam(v, all, rest, cost, seg_count, seg_tok) ? team : 0;
}

}  // namespace gb
