// The history-aware sequence scorer (Appendix, "Evaluating Search Generalization",
// Eq. 4-6) run incrementally over the search: each thought step adds one position to
// every trace's step sequence, and the scorer's own key/value cache lives in a second
// beam pool (the step pool: one token per thought step), so a branched trace shares
// its parent's scorer history the way it shares its KV (forked block tables).
//
// Per step and layer, on the C slots of the step pool:
//   x_t  = GELU(W_in LN(h_t))                                   (Eq. 4)
//   u    = LN1(x);  q, k, v = W_qkv u, RoPE on q and k at the position t
//   a    = paged causal attention of q over the trace's cached k/v plus (k, v)
//          (gb_decode_attention on the step pool: it appends k, v first)
//   x   += W_o a;   u = LN2(x);   x += W_2 (SiLU(W_1 u) * W_3 u)  (Eq. 5)
//   y_t  = sigmoid(w_out . LN(x) + b_out)                        (Eq. 6)
// Every product runs on tcgen05 (bf16 operands, fp32 accumulation).  W_in, whose K is the
// generator's hidden size, is the split-K GEMM of gemm.cu; the others are, up to d_model 512,
// k_fused_gemm, which builds its A operand itself (LayerNorm of the residual stream, or the
// attention output rounded to bf16) and finishes the product (RoPE, residual add, SwiGLU) in the
// same launch, and above that the split-K GEMM and an epilogue (split_products).  The residual
// stream x is fp32; the operands of the products (LayerNorm outputs, q/k/v, attention outputs,
// SwiGLU outputs) are rounded to bf16.
//
// Model shape: L = the step pool's layers, Hq query heads and Hkv key/value heads of
// 128 dims (the step pool's head counts, bf16 K/V), d_model = Hq * 128.  LayerNorm
// eps 1e-5; GELU the exact (erf) form; rotary pairs (i, i + 64) with angle
// t * 10000^(-i/64); softmax scale 1/sqrt(128).
#include "internal.cuh"
#include "ptx.cuh"
#include "tc.cuh"

namespace gb {
namespace {

constexpr int kHd = 128;               // head dim of the scorer's attention
constexpr int kRowThreads = 256;       // epilogue CTAs: one per row
constexpr float kLnEps = 1e-5f;
constexpr int kPerLayer = 8;           // tensors per layer in the weight buffer
constexpr int kSplitBudget = 8;        // partial buffer: kSplitBudget x C x (widest product)

enum LayerTensor { kLn1G, kLn1B, kWqkv, kWo, kLn2G, kLn2B, kW13, kW2 };

struct Dims {
  int H, F, d, L, Hq, Hkv, G, Nqkv, C, Nmax, Umax;
};

size_t a256(size_t x) { return (x + 255) & ~size_t(255); }

bool make_dims(const gb_pool* p, const gb_scorer_config* cfg, Dims* s) {
  const gb_pool_config& c = p->cfg;
  if (!cfg || cfg->hidden_dim <= 0 || cfg->hidden_dim % 64 || cfg->ffn_dim <= 0 || cfg->ffn_dim % 64) return false;
  if (c.kv_dtype != GB_BF16 || c.head_dim != kHd) return false;
  s->H = cfg->hidden_dim;
  s->F = cfg->ffn_dim;
  s->L = c.num_layers;
  s->Hq = c.num_q_heads;
  s->Hkv = c.num_kv_heads;
  s->G = s->Hq / s->Hkv;
  s->d = s->Hq * kHd;
  s->Nqkv = (s->Hq + 2 * s->Hkv) * kHd;
  s->C = c.max_beams;
  s->Nmax = s->d > s->Nqkv ? s->d : s->Nqkv;
  s->Nmax = s->Nmax > 2 * s->F ? s->Nmax : 2 * s->F;
  s->Umax = s->H > s->d ? s->H : s->d;
  s->Umax = s->Umax > s->F ? s->Umax : s->F;
  return true;
}

int n_tensors(const Dims& s) { return 3 + kPerLayer * s.L + 4; }

// Byte sizes of the weight tensors in buffer order.
void tensor_sizes(const Dims& s, size_t* b) {
  int i = 0;
  b[i++] = 4 * (size_t)s.H;                 // ln_in gain
  b[i++] = 4 * (size_t)s.H;                 // ln_in bias
  b[i++] = 2 * (size_t)s.d * s.H;           // W_in [d][H]
  for (int l = 0; l < s.L; ++l) {
    b[i++] = 4 * (size_t)s.d;               // ln1 gain, bias
    b[i++] = 4 * (size_t)s.d;
    b[i++] = 2 * (size_t)s.Nqkv * s.d;      // W_qkv [(Hq + 2 Hkv) 128][d]: q heads, k heads, v heads
    b[i++] = 2 * (size_t)s.d * s.d;         // W_o [d][d]
    b[i++] = 4 * (size_t)s.d;               // ln2 gain, bias
    b[i++] = 4 * (size_t)s.d;
    b[i++] = 2 * (size_t)2 * s.F * s.d;     // W_13 [2F][d]: W_1 rows then W_3 rows
    b[i++] = 2 * (size_t)s.d * s.F;         // W_2 [d][F]
  }
  b[i++] = 4 * (size_t)s.d;                 // ln_out gain, bias
  b[i++] = 4 * (size_t)s.d;
  b[i++] = 4 * (size_t)s.d;                 // w_out
  b[i++] = 4;                               // b_out
}

size_t weight_offsets(const Dims& s, size_t* off) {
  size_t sz[3 + kPerLayer * 64 + 4];
  tensor_sizes(s, sz);
  size_t o = 0;
  for (int i = 0; i < n_tensors(s); ++i) {
    if (off) off[i] = o;
    o += a256(sz[i]);
  }
  return o;
}

struct Ws {
  size_t u, x, q, kn, vn, att, part, seedk, seedv, total;
  size_t part_floats;
};

Ws ws_layout(const Dims& s) {
  Ws w;
  size_t o = 0;
  auto take = [&](size_t bytes) {
    const size_t r = o;
    o += a256(bytes);
    return r;
  };
  w.u = take(2 * (size_t)s.C * s.Umax);
  w.x = take(4 * (size_t)s.C * s.d);
  w.q = take(2 * (size_t)s.C * s.d);
  w.kn = take(2 * (size_t)s.C * s.Hkv * kHd);
  w.vn = take(2 * (size_t)s.C * s.Hkv * kHd);
  w.att = take(4 * (size_t)s.C * s.d);
  w.part_floats = (size_t)kSplitBudget * s.C * s.Nmax;
  w.part = take(4 * w.part_floats);
  w.seedk = take(2 * (size_t)s.L * s.Hkv * kHd);
  w.seedv = take(2 * (size_t)s.L * s.Hkv * kHd);
  w.total = o;
  return w;
}

// Fixed-order block sum (xor butterfly in each warp, then the warps in order); every
// thread gets the total.  `red` holds 33 floats.
__device__ __forceinline__ float block_sum(float v, float* red) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (lane == 0) red[warp] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    float t = 0.f;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += red[w];
    red[32] = t;
  }
  __syncthreads();
  const float t = red[32];
  __syncthreads();
  return t;
}

__device__ __forceinline__ bool row_live(const int* active, int m) { return active == nullptr || active[m] != 0; }

// Input LayerNorm of Eq. 4: u[m] = LN_in(h[m]) (bf16 h, H wide, H % 64 == 0).  Inactive
// rows give zeros.  16-byte loads and stores (8 values); the row is staged in shared memory.
__global__ void __launch_bounds__(kRowThreads) k_ln_in(const __nv_bfloat16* __restrict__ h, int H,
                                                       const float* __restrict__ g, const float* __restrict__ b,
                                                       const int* active,
                                                       __nv_bfloat16* __restrict__ u) {
  pdl_wait();
  pdl_launch_dependents();
  extern __shared__ float row[];
  __shared__ float red[33];
  const int m = blockIdx.x, nv = H / 8;
  uint4* out = reinterpret_cast<uint4*>(u + (size_t)m * H);
  if (!row_live(active, m)) {
    for (int i = threadIdx.x; i < nv; i += blockDim.x) out[i] = make_uint4(0, 0, 0, 0);
    return;
  }
  const uint4* in = reinterpret_cast<const uint4*>(h + (size_t)m * H);
  float s = 0.f;
  for (int i = threadIdx.x; i < nv; i += blockDim.x) {
    const uint4 q = in[i];
    const __nv_bfloat162* p2 = reinterpret_cast<const __nv_bfloat162*>(&q);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float2 f = __bfloat1622float2(p2[j]);
      row[8 * i + 2 * j] = f.x;
      row[8 * i + 2 * j + 1] = f.y;
      s += f.x + f.y;
    }
  }
  const float mu = block_sum(s, red) / (float)H;
  float v = 0.f;
  for (int i = threadIdx.x; i < H; i += blockDim.x) {
    const float c = row[i] - mu;
    v = fmaf(c, c, v);
  }
  const float r = 1.0f / sqrtf(block_sum(v, red) / (float)H + kLnEps);
  for (int i = threadIdx.x; i < nv; i += blockDim.x) {
    uint4 q;
    __nv_bfloat162* p2 = reinterpret_cast<__nv_bfloat162*>(&q);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int e = 8 * i + 2 * j;
      p2[j] = __floats2bfloat162_rn((row[e] - mu) * r * g[e] + b[e], (row[e + 1] - mu) * r * g[e + 1] + b[e + 1]);
    }
    out[i] = q;
  }
}

// x = GELU(z) of Eq. 4 (exact, erf), z = the sum of the product's K-split partials.
__global__ void __launch_bounds__(kRowThreads) k_gelu_epilogue(const float* P, int splits, int n4,
                                                               float* __restrict__ x) {
  pdl_wait();
  pdl_launch_dependents();
  const int i = blockIdx.x * kRowThreads + threadIdx.x;
  if (i >= n4) return;
  float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
  for (int k = 0; k < splits; ++k) {
    const float4 p = reinterpret_cast<const float4*>(P)[(size_t)k * n4 + i];
    z = make_float4(z.x + p.x, z.y + p.y, z.z + p.z, z.w + p.w);
  }
  auto gelu = [](float t) { return 0.5f * t * (1.0f + erff(t * 0.70710678118654752f)); };
  reinterpret_cast<float4*>(x)[i] = make_float4(gelu(z.x), gelu(z.y), gelu(z.z), gelu(z.w));
}

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Output head (Eq. 6), one warp per row: score = sigmoid(w_out . LN(x) + b_out); 0 for inactive rows.
__global__ void __launch_bounds__(kRowThreads) k_head(const float* x, int M, int d,
                                                      const float* __restrict__ g, const float* __restrict__ b,
                                                      const float* __restrict__ w_out, const float* __restrict__ b_out,
                                                      const int* active, float* __restrict__ score) {
  pdl_wait();
  pdl_launch_dependents();
  const int m = blockIdx.x * (kRowThreads / 32) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (m >= M) return;
  if (!row_live(active, m)) {
    if (lane == 0) score[m] = 0.f;
    return;
  }
  const float4* row = reinterpret_cast<const float4*>(x + (size_t)m * d);
  float s = 0.f, v = 0.f, dot = 0.f;
  for (int i = lane; i < d / 4; i += 32) s += (row[i].x + row[i].y) + (row[i].z + row[i].w);
  const float mu = warp_sum(s) / (float)d;
  for (int i = lane; i < d / 4; i += 32) {
    const float4 y = row[i];
    v = fmaf(y.x - mu, y.x - mu, v);
    v = fmaf(y.y - mu, y.y - mu, v);
    v = fmaf(y.z - mu, y.z - mu, v);
    v = fmaf(y.w - mu, y.w - mu, v);
  }
  const float r = 1.0f / sqrtf(warp_sum(v) / (float)d + kLnEps);
  for (int i = lane; i < d / 4; i += 32) {
    const float4 y = row[i], gg = reinterpret_cast<const float4*>(g)[i], bb = reinterpret_cast<const float4*>(b)[i],
                 w = reinterpret_cast<const float4*>(w_out)[i];
    dot = fmaf((y.x - mu) * r * gg.x + bb.x, w.x, dot);
    dot = fmaf((y.y - mu) * r * gg.y + bb.y, w.y, dot);
    dot = fmaf((y.z - mu) * r * gg.z + bb.z, w.z, dot);
    dot = fmaf((y.w - mu) * r * gg.w + bb.w, w.w, dot);
  }
  const float y = warp_sum(dot) + b_out[0];
  if (lane == 0) score[m] = 1.0f / (1.0f + expf(-y));
}

// ---- products with their operand and epilogue in one launch -------------------------------------
//
// Grid (row tiles of mt = 32, 64 or 128 slots) x (64-column tiles).  A CTA of 256 threads builds its
// rows' A operand in shared memory (128-byte swizzle, pass_k of K at a time), loads its 64 rows of
// the weights, multiplies (128 x 64 x 16 tcgen05.mma into tensor memory; the accumulator's rows past
// mt, whatever the shared memory there gave them, are never read) and finishes its tile.  At these sizes (64 slots, d = 512: 32 MFLOP and 0.5-2 MiB of weights
// a product) a product is latency: the chain of LayerNorm, GEMM with K-split partials in global
// memory and epilogue was three launches of 6-9 us each.  So K is not split, the LayerNorm is
// recomputed by every column tile (its rows come from L2), and the weights, which do not depend on
// the previous launch, are loaded before waiting for it.  mt is the smallest that keeps the grid
// within the SMs: fewer rows per CTA shorten its own chain.
enum AMode { kALn, kAF32, kABf16 };              // LayerNorm of fp32 rows (K <= kFK); fp32 rows; bf16 rows
enum EMode { kEQkv, kEResid, kESwiglu };         // RoPE and q/k/v in bf16; x += z; SwiGLU in bf16

constexpr int kFThreads = 256, kFN = 64;
constexpr int kFK = 512;                                    // K a warp's registers hold of a row at a time
constexpr int kFBBlock = kFN * 128;                         // 64 of K of the weights: 64 rows x 128 bytes
constexpr int kFOperands = 192 * 1024;                      // A (mt rows x pass_k) and the weights (64 x pass_k)
constexpr int kFCtl = kFOperands;                           // mbarrier, tensor-memory address
constexpr int kFSmem = kFCtl + 16;
constexpr int kFTile = kFN + 1;                             // epilogue tile [mt][65] over the A operand
static_assert(kFSmem <= 232448 - 1024, "shared memory per block");
// K per pass: what fits beside the weights, one pass up to 1024 for the 32-row tiles of small steps.
__host__ __device__ constexpr int pass_k(int mt) { return mt == 32 ? 1024 : 512; }
static_assert(32 * 1024 * 2 + kFN * 1024 * 2 <= kFOperands && 128 * 512 * 2 + kFN * 512 * 2 <= kFOperands, "operands");

struct FusedArgs {
  const void* a;            // [M][K]
  const float *g, *b;       // LayerNorm gain and bias (kALn)
  const __nv_bfloat16* w;   // weights, rows of K
  int M, K, mt;
  const int* active;
  float* x;                 // kEResid: [M][d]
  int d;
  __nv_bfloat16 *q, *kn, *vn;  // kEQkv
  int Hq, Hkv, pos_shift;
  const int* pos_of;
  __nv_bfloat16* u;         // kESwiglu: [M][F]
  int F;
  int* ctl;
};

// Weight row of column n of column tile t.  A rotary tile holds 32 (i, i + 64) pairs of one head, a
// SwiGLU tile 32 columns of W_1 and the same of W_3, so each tile finishes on its own.
template <int E>
__device__ __forceinline__ int weight_row(const FusedArgs& p, int t, int n) {
  if (E == kEQkv) {
    const int rot = 2 * (p.Hq + p.Hkv);
    if (t < rot) return (t >> 1) * kHd + (t & 1) * 32 + (n & 31) + (n >> 5) * (kHd / 2);
    return (p.Hq + p.Hkv) * kHd + (t - rot) * kFN + n;
  }
  if (E == kESwiglu) return t * 32 + (n & 31) + (n >> 5) * p.F;
  return t * kFN + n;
}

template <int A, int E>
__global__ void __launch_bounds__(kFThreads, 1) k_fused_gemm(FusedArgs p) {
  extern __shared__ __align__(1024) unsigned char sm[];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int m0 = blockIdx.x * p.mt, t = blockIdx.y;
  const uint32_t sbase = smem_addr(sm), bar = sbase + kFCtl;
  if (sbase & 1023) {
    if (tid == 0) set_status(p.ctl, GB_ERR_UNSUPPORTED);
    return;
  }
  if (tid == 0) {
    mbar_init(bar, 1);
    fence_mbar_init();
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(bar + 8), "r"(kFN));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  const int fk = pass_k(p.mt), a_block = p.mt * 128;  // A block: 64 of K, mt rows x 128 bytes
  const uint32_t b_base = (uint32_t)(p.mt * fk * 2);
  auto load_b = [&](int k0) {
    const int pc = min(fk, p.K - k0) / 8;  // 16-byte pieces per row
    for (int n = warp; n < kFN; n += kFThreads / 32) {  // a warp per row: 512 contiguous bytes at a time
      const __nv_bfloat16* src = p.w + (size_t)weight_row<E>(p, t, n) * p.K + k0;
      for (int c = lane; c < pc; c += 32)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(sbase + b_base + (c >> 3) * kFBBlock +
                                                                       swz(n, (c & 7) * 8)),
                     "l"(src + 8 * c)
                     : "memory");
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  load_b(0);
  pdl_wait();
  pdl_launch_dependents();

  const float* af = static_cast<const float*>(p.a);
  auto live_row = [&](int r) { return r < p.mt && m0 + r < p.M && row_live(p.active, m0 + r); };
  bool ok = true;
  int pass = 0;
  uint32_t tmem = 0;
  for (int k0 = 0; k0 < p.K; k0 += fk, ++pass) {
    const int kpass = min(fk, p.K - k0);
    if (pass > 0) {  // the previous pass's operands have been read
      ok = ok && mbar_wait_bounded(bar, (pass - 1) & 1, kWaitLimitNs);
      load_b(k0);
    }
    // A: row r = warp + 8 j of the tile, four rows in flight per warp, 512 of K at a time.
    for (int h0 = 0; h0 < kpass; h0 += kFK) {
      const int kw = min(kFK, kpass - h0), kh = k0 + h0;
      unsigned char* sa = sm + (h0 >> 6) * a_block;
      if (A == kABf16) {
        const __nv_bfloat16* ab = static_cast<const __nv_bfloat16*>(p.a);
        for (int r0 = warp; r0 < p.mt; r0 += kFThreads / 32 * 4) {
          uint4 v[4][kFK / 256];
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int r = r0 + kFThreads / 32 * u;
            const bool live = live_row(r);
#pragma unroll
            for (int i = 0; i < kFK / 256; ++i) {
              const int c = 8 * lane + 256 * i;
              v[u][i] = live && c < kw ? *reinterpret_cast<const uint4*>(ab + (size_t)(m0 + r) * p.K + kh + c)
                                       : make_uint4(0u, 0u, 0u, 0u);
            }
          }
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int r = r0 + kFThreads / 32 * u;
#pragma unroll
            for (int i = 0; i < kFK / 256; ++i) {
              const int c = 8 * lane + 256 * i;
              if (r < p.mt && c < kw) *reinterpret_cast<uint4*>(sa + (c >> 6) * a_block + swz(r, c & 63)) = v[u][i];
            }
          }
        }
      } else {
        float4 gg[kFK / 128], bb[kFK / 128];
        if (A == kALn) {
#pragma unroll
          for (int i = 0; i < kFK / 128; ++i) {
            const int c = 4 * lane + 128 * i;
            gg[i] = c < kw ? *reinterpret_cast<const float4*>(p.g + kh + c) : make_float4(0.f, 0.f, 0.f, 0.f);
            bb[i] = c < kw ? *reinterpret_cast<const float4*>(p.b + kh + c) : make_float4(0.f, 0.f, 0.f, 0.f);
          }
        }
        for (int r0 = warp; r0 < p.mt; r0 += kFThreads / 32 * 4) {
          float4 v[4][kFK / 128];
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int r = r0 + kFThreads / 32 * u;
            const bool live = live_row(r);
#pragma unroll
            for (int i = 0; i < kFK / 128; ++i) {
              const int c = 4 * lane + 128 * i;
              v[u][i] = live && c < kw ? *reinterpret_cast<const float4*>(af + (size_t)(m0 + r) * p.K + kh + c)
                                       : make_float4(0.f, 0.f, 0.f, 0.f);
            }
          }
          // The four rows' statistics together: their shuffles are independent chains.
          float mu[4] = {0.f, 0.f, 0.f, 0.f}, rs[4] = {1.f, 1.f, 1.f, 1.f};
          if (A == kALn) {
            float s[4], q[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int u = 0; u < 4; ++u) {
              s[u] = 0.f;
#pragma unroll
              for (int i = 0; i < kFK / 128; ++i) s[u] += (v[u][i].x + v[u][i].y) + (v[u][i].z + v[u][i].w);
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1)
#pragma unroll
              for (int u = 0; u < 4; ++u) s[u] += __shfl_xor_sync(0xffffffffu, s[u], o);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
              mu[u] = s[u] / (float)p.K;
#pragma unroll
              for (int i = 0; i < kFK / 128; ++i)
                if (4 * lane + 128 * i < kw) {
                  q[u] = fmaf(v[u][i].x - mu[u], v[u][i].x - mu[u], q[u]);
                  q[u] = fmaf(v[u][i].y - mu[u], v[u][i].y - mu[u], q[u]);
                  q[u] = fmaf(v[u][i].z - mu[u], v[u][i].z - mu[u], q[u]);
                  q[u] = fmaf(v[u][i].w - mu[u], v[u][i].w - mu[u], q[u]);
                }
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1)
#pragma unroll
              for (int u = 0; u < 4; ++u) q[u] += __shfl_xor_sync(0xffffffffu, q[u], o);
#pragma unroll
            for (int u = 0; u < 4; ++u) rs[u] = 1.0f / sqrtf(q[u] / (float)p.K + kLnEps);
          }
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int r = r0 + kFThreads / 32 * u;
#pragma unroll
            for (int i = 0; i < kFK / 128; ++i) {
              const int c = 4 * lane + 128 * i;
              float4 y = v[u][i];
              if (A == kALn)
                y = make_float4((y.x - mu[u]) * rs[u] * gg[i].x + bb[i].x, (y.y - mu[u]) * rs[u] * gg[i].y + bb[i].y,
                                (y.z - mu[u]) * rs[u] * gg[i].z + bb[i].z, (y.w - mu[u]) * rs[u] * gg[i].w + bb[i].w);
              const __nv_bfloat162 lo = __floats2bfloat162_rn(y.x, y.y), hi = __floats2bfloat162_rn(y.z, y.w);
              if (r < p.mt && c < kw)
                *reinterpret_cast<uint2*>(sa + (c >> 6) * a_block + swz(r, c & 63)) =
                    make_uint2(*reinterpret_cast<const uint32_t*>(&lo), *reinterpret_cast<const uint32_t*>(&hi));
            }
          }
        }
      }
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    fence_proxy_async_smem();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    tmem = *reinterpret_cast<volatile uint32_t*>(sm + kFCtl + 8);
    if (tid == 0 && ok) {
      constexpr uint32_t ID = idesc(128, kFN, false);
      for (int kb = 0; kb < kpass / 64; ++kb)
#pragma unroll
        for (int kk = 0; kk < 4; ++kk)
          mma(tmem, sdesc(sbase + kb * a_block + kk * 32, 16, 1024),
              sdesc(sbase + b_base + kb * kFBBlock + kk * 32, 16, 1024), ID, (pass > 0 || kb > 0 || kk > 0) ? 1u : 0u);
      mma_commit(bar);
    }
  }
  ok = ok && mbar_wait_bounded(bar, (pass - 1) & 1, kWaitLimitNs);
  ok = __syncthreads_and(ok) != 0;
  tc_fence_after();
  float* tile = reinterpret_cast<float*>(sm);  // [mt][65]
  if (ok && warp < p.mt / 32) {
#pragma unroll
    for (int c0 = 0; c0 < kFN; c0 += 32) {
      float z[32];
      tmem_ld32(tmem + ((uint32_t)(warp * 32) << 16) + c0, z);
#pragma unroll
      for (int i = 0; i < 32; ++i) tile[(warp * 32 + lane) * kFTile + c0 + i] = z[i];
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kFN));
  if (!ok) {
    if (tid == 0) set_status(p.ctl, GB_ERR_TIMEOUT);
    return;
  }

  const int rows = min(p.mt, p.M - m0);
  if (E == kEQkv) {
    const int rot = 2 * (p.Hq + p.Hkv);
    if (t < rot) {
      // Rotate the pairs (i, i + 64) by pos * 10000^(-i/64); inactive rows give zeros.
      const int head = t >> 1, i = (t & 1) * 32 + lane;
      const float inv = powf(10000.0f, -(float)i / (float)(kHd / 2));
      for (int r = warp; r < rows; r += kFThreads / 32) {
        const int m = m0 + r;
        float a = 0.f, c = 0.f;
        if (row_live(p.active, m)) {
          const float x1 = tile[r * kFTile + lane], x2 = tile[r * kFTile + 32 + lane];
          const float pos = p.pos_of ? (float)(p.pos_of[m] + p.pos_shift) : 0.f;
          float sn, cs;
          sincosf(pos * inv, &sn, &cs);
          a = x1 * cs - x2 * sn;
          c = x1 * sn + x2 * cs;
        }
        __nv_bfloat16* dst =
            head < p.Hq ? p.q + ((size_t)m * p.Hq + head) * kHd : p.kn + ((size_t)m * p.Hkv + head - p.Hq) * kHd;
        dst[i] = __float2bfloat16_rn(a);
        dst[i + kHd / 2] = __float2bfloat16_rn(c);
      }
    } else {
      for (int i = tid; i < rows * kFN; i += kFThreads) {
        const int r = i / kFN, c = i % kFN, m = m0 + r;
        p.vn[(size_t)m * p.Hkv * kHd + (t - rot) * kFN + c] =
            __float2bfloat16_rn(row_live(p.active, m) ? tile[r * kFTile + c] : 0.f);
      }
    }
  } else if (E == kEResid) {
    for (int i = tid; i < rows * kFN; i += kFThreads) {
      const int r = i / kFN, c = i % kFN, m = m0 + r;
      if (row_live(p.active, m)) p.x[(size_t)m * p.d + t * kFN + c] += tile[r * kFTile + c];
    }
  } else {
    for (int i = tid; i < rows * 32; i += kFThreads) {
      const int r = i / 32, c = i % 32, m = m0 + r;
      if (!row_live(p.active, m)) continue;
      const float g1 = tile[r * kFTile + c], g3 = tile[r * kFTile + 32 + c];
      p.u[(size_t)m * p.F + t * 32 + c] = __float2bfloat16_rn(g1 / (1.0f + expf(-g1)) * g3);
    }
  }
}

// Attention of the first position alone (the seed row): softmax over one key is 1, so
// query head h returns the value of KV head h / G.
__global__ void k_first_position_attention(const __nv_bfloat16* vn, int Hq, int G,
                                           float* __restrict__ att) {
  pdl_wait();
  pdl_launch_dependents();
  for (int j = threadIdx.x; j < Hq * kHd; j += blockDim.x) att[j] = __bfloat162float(vn[(j / kHd / G) * kHd + j % kHd]);
}

// ---- products with K-split partials (split_products) ----------------------------------------------
//
// d_model above 512: a product is k_gemm_partials (gemm.cu) and an epilogue that sums its partials,
// one CTA per row, four columns per thread (16-byte loads, the splits in flight together).

// Columns n .. n + 3 of row m, the splits in order.
__device__ __forceinline__ float4 sum_partials(const float* P, int splits, int M, int N, int m, int n) {
  float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 4
  for (int k = 0; k < splits; ++k) {
    const float4 y = *reinterpret_cast<const float4*>(P + ((size_t)k * M + m) * N + n);
    z = make_float4(z.x + y.x, z.y + y.y, z.z + y.z, z.w + y.w);
  }
  return z;
}

__device__ __forceinline__ void store_bf16x4(__nv_bfloat16* d, float a, float b, float c, float e) {
  __nv_bfloat162 p[2] = {__floats2bfloat162_rn(a, b), __floats2bfloat162_rn(c, e)};
  *reinterpret_cast<uint2*>(d) = *reinterpret_cast<const uint2*>(p);
}

enum RowMode { kGeluLn = 0, kResidLn = 1, kResid = 2 };

// Epilogue of a d-wide product: x = GELU(z) (kGeluLn) or x += z, then u = LN(x) in bf16 (not kResid,
// which the head follows).  Inactive rows: u = 0.
template <int Mode>
__global__ void __launch_bounds__(kRowThreads) k_row_epilogue(const float* P, int splits, int M, int d,
                                                              float* __restrict__ x, const float* __restrict__ g,
                                                              const float* __restrict__ b, const int* active,
                                                              __nv_bfloat16* __restrict__ u) {
  pdl_wait();
  pdl_launch_dependents();
  extern __shared__ float row[];
  __shared__ float red[33];
  const int m = blockIdx.x, n4 = d / 4;
  __nv_bfloat16* um = u + (size_t)m * d;
  if (!row_live(active, m)) {
    if (Mode != kResid)
      for (int i = threadIdx.x; i < n4; i += blockDim.x) store_bf16x4(um + 4 * i, 0.f, 0.f, 0.f, 0.f);
    return;
  }
  float4* xm = reinterpret_cast<float4*>(x + (size_t)m * d);
  float4* row4 = reinterpret_cast<float4*>(row);
  float s = 0.f;
  for (int i = threadIdx.x; i < n4; i += blockDim.x) {
    float4 z = sum_partials(P, splits, M, d, m, 4 * i);
    if (Mode == kGeluLn) {
      z.x = 0.5f * z.x * (1.0f + erff(z.x * 0.70710678118654752f));
      z.y = 0.5f * z.y * (1.0f + erff(z.y * 0.70710678118654752f));
      z.z = 0.5f * z.z * (1.0f + erff(z.z * 0.70710678118654752f));
      z.w = 0.5f * z.w * (1.0f + erff(z.w * 0.70710678118654752f));
    } else {
      const float4 y = xm[i];
      z = make_float4(y.x + z.x, y.y + z.y, y.z + z.z, y.w + z.w);
    }
    xm[i] = z;
    row4[i] = z;
    s += (z.x + z.y) + (z.z + z.w);
  }
  if (Mode == kResid) return;
  const float mu = block_sum(s, red) / (float)d;
  float v = 0.f;
  for (int i = threadIdx.x; i < n4; i += blockDim.x) {  // the elements this thread wrote
    const float4 y = row4[i];
    v = fmaf(y.x - mu, y.x - mu, v);
    v = fmaf(y.y - mu, y.y - mu, v);
    v = fmaf(y.z - mu, y.z - mu, v);
    v = fmaf(y.w - mu, y.w - mu, v);
  }
  const float r = 1.0f / sqrtf(block_sum(v, red) / (float)d + kLnEps);
  for (int i = threadIdx.x; i < n4; i += blockDim.x) {
    const float4 y = row4[i], gg = reinterpret_cast<const float4*>(g)[i], bb = reinterpret_cast<const float4*>(b)[i];
    store_bf16x4(um + 4 * i, (y.x - mu) * r * gg.x + bb.x, (y.y - mu) * r * gg.y + bb.y, (y.z - mu) * r * gg.z + bb.z,
                 (y.w - mu) * r * gg.w + bb.w);
  }
}

// Epilogue of the q/k/v product: the (i, i + 64) pairs of every q and k head are rotated by
// pos * 10000^(-i/64) with pos = pos_of[m] + pos_shift (0 without pos_of).
__global__ void __launch_bounds__(kRowThreads) k_qkv_epilogue(const float* P, int splits, int M, int Hq,
                                                              int Hkv, const int* pos_of, int pos_shift,
                                                              const int* active,
                                                              __nv_bfloat16* __restrict__ q,
                                                              __nv_bfloat16* __restrict__ kn,
                                                              __nv_bfloat16* __restrict__ vn) {
  pdl_wait();
  pdl_launch_dependents();
  const int m = blockIdx.x, N = (Hq + 2 * Hkv) * kHd;
  const bool live = row_live(active, m);
  const float pos = pos_of && live ? (float)(pos_of[m] + pos_shift) : 0.f;
  constexpr int kQuads = kHd / 8;  // groups of four pairs per head
  for (int j = threadIdx.x; j < (Hq + Hkv) * kQuads; j += blockDim.x) {
    const int head = j / kQuads, i = 4 * (j % kQuads);
    float a[4] = {0.f, 0.f, 0.f, 0.f}, c[4] = {0.f, 0.f, 0.f, 0.f};
    if (live) {
      const float4 y1 = sum_partials(P, splits, M, N, m, head * kHd + i);
      const float4 y2 = sum_partials(P, splits, M, N, m, head * kHd + i + kHd / 2);
      const float x1[4] = {y1.x, y1.y, y1.z, y1.w}, x2[4] = {y2.x, y2.y, y2.z, y2.w};
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        float sn, cs;
        sincosf(pos * powf(10000.0f, -(float)(i + e) / (float)(kHd / 2)), &sn, &cs);
        a[e] = x1[e] * cs - x2[e] * sn;
        c[e] = x1[e] * sn + x2[e] * cs;
      }
    }
    __nv_bfloat16* dst = head < Hq ? q + ((size_t)m * Hq + head) * kHd : kn + ((size_t)m * Hkv + head - Hq) * kHd;
    store_bf16x4(dst + i, a[0], a[1], a[2], a[3]);
    store_bf16x4(dst + i + kHd / 2, c[0], c[1], c[2], c[3]);
  }
  for (int j = 4 * threadIdx.x; j < Hkv * kHd; j += 4 * blockDim.x) {
    const float4 z = live ? sum_partials(P, splits, M, N, m, (Hq + Hkv) * kHd + j) : make_float4(0.f, 0.f, 0.f, 0.f);
    store_bf16x4(vn + (size_t)m * Hkv * kHd + j, z.x, z.y, z.z, z.w);
  }
}

// SwiGLU epilogue: u[m][n] = SiLU(z[m][n]) * z[m][F + n] in bf16 (z = W_13 u, F wide halves).
__global__ void __launch_bounds__(kRowThreads) k_swiglu_epilogue(const float* P, int splits, int M, int F,
                                                                 const int* active,
                                                                 __nv_bfloat16* __restrict__ u) {
  pdl_wait();
  pdl_launch_dependents();
  const int m = blockIdx.x;
  const bool live = row_live(active, m);
  auto act = [](float g1, float g3) { return g1 / (1.0f + expf(-g1)) * g3; };
  for (int n = 4 * threadIdx.x; n < F; n += 4 * blockDim.x) {
    float4 y = make_float4(0.f, 0.f, 0.f, 0.f);
    if (live) {
      const float4 g1 = sum_partials(P, splits, M, 2 * F, m, n), g3 = sum_partials(P, splits, M, 2 * F, m, F + n);
      y = make_float4(act(g1.x, g3.x), act(g1.y, g3.y), act(g1.z, g3.z), act(g1.w, g3.w));
    }
    store_bf16x4(u + (size_t)m * F + n, y.x, y.y, y.z, y.w);
  }
}

// Attention outputs (fp32) to the bf16 operand of W_o.
__global__ void __launch_bounds__(kRowThreads) k_to_bf16(const float* a, int n4, __nv_bfloat16* __restrict__ u) {
  pdl_wait();
  pdl_launch_dependents();
  const int i = blockIdx.x * kRowThreads + threadIdx.x;
  if (i >= n4) return;
  const float4 y = reinterpret_cast<const float4*>(a)[i];
  store_bf16x4(u + 4 * (size_t)i, y.x, y.y, y.z, y.w);
}

struct Run {
  gb_pool* pool;
  Dims s;
  const char* w;
  size_t off[3 + kPerLayer * 64 + 4];
  char* ws;
  Ws L;
  cudaStream_t st;
  int launches = 0;

  template <class T>
  const T* wt(int i) const { return reinterpret_cast<const T*>(w + off[i]); }
  int layer_tensor(int l, int t) const { return 3 + kPerLayer * l + t; }
  int tail(int t) const { return 3 + kPerLayer * s.L + t; }
  __nv_bfloat16* u() const { return reinterpret_cast<__nv_bfloat16*>(ws + L.u); }
  float* x() const { return reinterpret_cast<float*>(ws + L.x); }
  float* part() const { return reinterpret_cast<float*>(ws + L.part); }

  // P = A [M][K] . B [N][K]^T as K-split partials; returns the split count (0 on failure).
  int gemm(const void* A, int M, const void* B, int N, int K) {
    const int splits = gemm_splits(M, N, K, pool->num_sms, L.part_floats);
    if (splits == 0) return 0;
    if (gemm_partials(A, M, B, N, K, splits, part(), pool->view.ctl, true, st) != cudaSuccess) return 0;
    ++launches;
    return splits;
  }

  // One fused product of `tiles` 64-column tiles.
  template <int A, int E>
  bool fused(FusedArgs p, int tiles) {
    p.ctl = pool->view.ctl;
    p.mt = 32;
    while (p.mt < 128 && (p.M + p.mt - 1) / p.mt * tiles > pool->num_sms) p.mt *= 2;
    if (set_max_dynamic_smem(reinterpret_cast<const void*>(k_fused_gemm<A, E>), kFSmem) != cudaSuccess) return false;
    ++launches;
    return launch_pdl(k_fused_gemm<A, E>, dim3((p.M + p.mt - 1) / p.mt, tiles), kFThreads, kFSmem, st, p) == cudaSuccess;
  }

  // A row of `floats` in dynamic shared memory beside the kernel's static words (red) may pass the 48 KiB
  // that a launch gets without asking.
  template <class K>
  static bool row_smem(K* kernel, int floats) {
    return floats * sizeof(float) + 256 <= 48 * 1024 ||
           set_max_dynamic_smem(reinterpret_cast<const void*>(kernel), 48 * 1024) == cudaSuccess;
  }

  template <int Mode>
  bool rows(int splits, int M, const float* g, const float* b, const int* active) {
    if (!row_smem(k_row_epilogue<Mode>, s.d)) return false;
    launch_pdl(k_row_epilogue<Mode>, M, kRowThreads, s.d * sizeof(float), st, static_cast<const float*>(part()), splits,
               M, s.d, x(), g, b, active, u());
    ++launches;
    return true;
  }

  // How a layer's products run: above d_model 512 a fused product's CTAs would each normalise rows of
  // several passes (and W_2's K runs with it).
  bool split_products() const { return s.d > kFK; }

  bool layer_split(int l, int M, bool step, const int* active, __nv_bfloat16* q, __nv_bfloat16* kn, __nv_bfloat16* vn,
                   float* att) {
    const float* P = part();
    int sp = gemm(u(), M, wt<__nv_bfloat16>(layer_tensor(l, kWqkv)), s.Nqkv, s.d);
    if (!sp) return false;
    launch_pdl(k_qkv_epilogue, M, kRowThreads, 0, st, P, sp, M, s.Hq, s.Hkv,
               step ? static_cast<const int*>(pool->view.seq_len) : nullptr, l > 0 ? -1 : 0, active, q, kn, vn);
    ++launches;
    if (!step && l + 1 == s.L) return true;  // the seed needs only each layer's k and v
    if (!attend(l, step, q, kn, vn, att)) return false;
    const int n4 = M * (s.d / 4);
    launch_pdl(k_to_bf16, (n4 + kRowThreads - 1) / kRowThreads, kRowThreads, 0, st, static_cast<const float*>(att), n4, u());
    ++launches;
    sp = gemm(u(), M, wt<__nv_bfloat16>(layer_tensor(l, kWo)), s.d, s.d);
    if (!sp) return false;
    if (!rows<kResidLn>(sp, M, wt<float>(layer_tensor(l, kLn2G)), wt<float>(layer_tensor(l, kLn2B)), active)) return false;
    sp = gemm(u(), M, wt<__nv_bfloat16>(layer_tensor(l, kW13)), 2 * s.F, s.d);
    if (!sp) return false;
    launch_pdl(k_swiglu_epilogue, M, kRowThreads, 0, st, P, sp, M, s.F, active, u());
    ++launches;
    sp = gemm(u(), M, wt<__nv_bfloat16>(layer_tensor(l, kW2)), s.d, s.F);
    if (!sp) return false;
    if (l + 1 < s.L)
      return rows<kResidLn>(sp, M, wt<float>(layer_tensor(l + 1, kLn1G)), wt<float>(layer_tensor(l + 1, kLn1B)), active);
    return rows<kResid>(sp, M, nullptr, nullptr, active);
  }

  // Attention of layer l over each trace's history, or of the first position alone.
  bool attend(int l, bool step, __nv_bfloat16* q, __nv_bfloat16* kn, __nv_bfloat16* vn, float* att) {
    if (step)
      return gb_decode_attention(pool, l, q, kn, vn, 0.08838834764831845f, att, GB_PATH_AUTO,
                                 reinterpret_cast<gb_stream_t>(st)) == GB_OK;
    launch_pdl(k_first_position_attention, 1, kRowThreads, 0, st, static_cast<const __nv_bfloat16*>(vn), s.Hq, s.G, att);
    ++launches;
    return true;
  }

  // The layer stack on M rows.  step = true: rows are the step pool's slots, attention
  // runs over each trace's cached history (and appends to it); RoPE positions are the
  // slots' sequence lengths.  step = false: one row at position 0 (the seed), whose
  // per-layer k and v go to the seed buffers.
  bool layers(int M, bool step, const int* active, float* score) {
    float* att = reinterpret_cast<float*>(ws + L.att);
    __nv_bfloat16* q = reinterpret_cast<__nv_bfloat16*>(ws + L.q);
    FusedArgs base{};
    base.M = M;
    base.active = active;
    base.x = x();
    base.d = s.d;
    for (int l = 0; l < s.L; ++l) {
      __nv_bfloat16* kn = reinterpret_cast<__nv_bfloat16*>(ws + (step ? L.kn : L.seedk)) +
                          (step ? 0 : (size_t)l * s.Hkv * kHd);
      __nv_bfloat16* vn = reinterpret_cast<__nv_bfloat16*>(ws + (step ? L.vn : L.seedv)) +
                          (step ? 0 : (size_t)l * s.Hkv * kHd);
      if (split_products()) {
        if (!layer_split(l, M, step, active, q, kn, vn, att)) return false;
        continue;
      }
      // q, k, v = RoPE(W_qkv LN1(x)).  Layer 0 opens the step pool's step, which advances every
      // length by one: the new position is seq_len before layer 0 and seq_len - 1 after it.
      FusedArgs p = base;
      p.a = x();
      p.g = wt<float>(layer_tensor(l, kLn1G));
      p.b = wt<float>(layer_tensor(l, kLn1B));
      p.w = wt<__nv_bfloat16>(layer_tensor(l, kWqkv));
      p.K = s.d;
      p.q = q;
      p.kn = kn;
      p.vn = vn;
      p.Hq = s.Hq;
      p.Hkv = s.Hkv;
      p.pos_of = step ? pool->view.seq_len : nullptr;
      p.pos_shift = l > 0 ? -1 : 0;
      if (!fused<kALn, kEQkv>(p, s.Nqkv / kFN)) return false;
      if (!step && l + 1 == s.L) break;  // the seed needs only each layer's k and v
      if (!attend(l, step, q, kn, vn, att)) return false;
      p = base;  // x += W_o a
      p.a = att;
      p.w = wt<__nv_bfloat16>(layer_tensor(l, kWo));
      p.K = s.d;
      if (!fused<kAF32, kEResid>(p, s.d / kFN)) return false;
      p = base;  // u = SiLU(W_1 LN2(x)) * W_3 LN2(x)
      p.a = x();
      p.g = wt<float>(layer_tensor(l, kLn2G));
      p.b = wt<float>(layer_tensor(l, kLn2B));
      p.w = wt<__nv_bfloat16>(layer_tensor(l, kW13));
      p.K = s.d;
      p.u = u();
      p.F = s.F;
      if (!fused<kALn, kESwiglu>(p, s.F / 32)) return false;
      p = base;  // x += W_2 u
      p.a = u();
      p.w = wt<__nv_bfloat16>(layer_tensor(l, kW2));
      p.K = s.F;
      if (!fused<kABf16, kEResid>(p, s.d / kFN)) return false;
    }
    if (step) {
      launch_pdl(k_head, (M + kRowThreads / 32 - 1) / (kRowThreads / 32), kRowThreads, 0, st,
                 static_cast<const float*>(x()), M, s.d, wt<float>(tail(0)), wt<float>(tail(1)), wt<float>(tail(2)),
                 wt<float>(tail(3)), active, score);
      ++launches;
    }
    return true;
  }

  // Eq. 4 on M rows of h.
  bool input(const void* h, int M, const int* active) {
    if (!row_smem(k_ln_in, s.H)) return false;
    launch_pdl(k_ln_in, M, kRowThreads, s.H * sizeof(float), st, reinterpret_cast<const __nv_bfloat16*>(h), s.H,
               wt<float>(0), wt<float>(1), active, u());
    ++launches;
    const int sp = gemm(u(), M, wt<__nv_bfloat16>(2), s.d, s.H);
    if (!sp) return false;
    if (split_products())  // with LN1 of layer 0
      return rows<kGeluLn>(sp, M, wt<float>(layer_tensor(0, kLn1G)), wt<float>(layer_tensor(0, kLn1B)), active);
    const int n4 = M * (s.d / 4);
    launch_pdl(k_gelu_epilogue, (n4 + kRowThreads - 1) / kRowThreads, kRowThreads, 0, st,
               static_cast<const float*>(part()), sp, n4, x());
    ++launches;
    return true;
  }
};

gb_status prepare(gb_pool* pool, const gb_scorer_config* cfg, const void* weights, void* ws, gb_stream_t stream,
                  Run* r) {
  if (!pool) return GB_ERR_INVALID;
  if (!make_dims(pool, cfg, &r->s)) return fail(pool, GB_ERR_UNSUPPORTED, "scorer: needs a bf16 step pool with 128-dim heads and sizes in multiples of 64");
  if (r->s.L > 64) return fail(pool, GB_ERR_UNSUPPORTED, "scorer: at most 64 layers");
  if (!weights || !ws || ((uintptr_t)weights & 255) || ((uintptr_t)ws & 255))
    return fail(pool, GB_ERR_INVALID, "scorer: weights and workspace must be 256-byte aligned device buffers");
  if (r->s.d * sizeof(float) > 48 * 1024 || r->s.H * sizeof(float) > 48 * 1024)
    return fail(pool, GB_ERR_UNSUPPORTED, "scorer: hidden_dim and d_model up to 12288");
  if (pool->next_layer != 0) return fail(pool, GB_ERR_STATE, "scorer: step pool has an open step");
  r->pool = pool;
  r->w = reinterpret_cast<const char*>(weights);
  weight_offsets(r->s, r->off);
  r->ws = reinterpret_cast<char*>(ws);
  r->L = ws_layout(r->s);
  r->st = reinterpret_cast<cudaStream_t>(stream);
  return GB_OK;
}

}  // namespace
}  // namespace gb

using namespace gb;

extern "C" gb_status gb_scorer_sizes(gb_pool* step_pool, const gb_scorer_config* cfg, size_t* weight_bytes,
                                     size_t* workspace_bytes, size_t* offsets, int max_offsets, int* n_offsets) {
  if (!step_pool) return GB_ERR_INVALID;
  Dims s;
  if (!make_dims(step_pool, cfg, &s)) return fail(step_pool, GB_ERR_UNSUPPORTED, "scorer: unsupported shape");
  if (s.L > 64) return fail(step_pool, GB_ERR_UNSUPPORTED, "scorer: at most 64 layers");
  size_t off[3 + kPerLayer * 64 + 4];
  const size_t wb = weight_offsets(s, off);
  if (weight_bytes) *weight_bytes = wb;
  if (workspace_bytes) *workspace_bytes = ws_layout(s).total;
  if (n_offsets) *n_offsets = n_tensors(s);
  if (offsets) {
    if (max_offsets < n_tensors(s)) return fail(step_pool, GB_ERR_INVALID, "scorer: offsets array too short");
    for (int i = 0; i < n_tensors(s); ++i) offsets[i] = off[i];
  }
  return GB_OK;
}

extern "C" gb_status gb_scorer_seed(gb_pool* step_pool, const gb_scorer_config* cfg, const void* weights_dev,
                                    void* workspace_dev, const void* h0_dev, int n_beams, gb_stream_t stream) {
  Run r;
  gb_status st = prepare(step_pool, cfg, weights_dev, workspace_dev, stream, &r);
  if (st != GB_OK) return st;
  if (!h0_dev || ((uintptr_t)h0_dev & 15)) return fail(step_pool, GB_ERR_INVALID, "scorer_seed: h0 must be 16-byte aligned");
  if (step_pool->seeded) return fail(step_pool, GB_ERR_STATE, "scorer_seed: step pool already seeded");
  if (n_beams < 1 || n_beams > r.s.C) return fail(step_pool, GB_ERR_INVALID, "scorer_seed: bad beam count");
  const bool ok = r.input(h0_dev, 1, nullptr) && r.layers(1, false, nullptr, nullptr);
  step_pool->launches += r.launches;
  st = check_launch(step_pool, "scorer_seed");
  if (st != GB_OK) return st;
  if (!ok) return fail(step_pool, GB_ERR_CUDA, "scorer_seed: a launch failed");
  return gb_pool_seed(step_pool, n_beams, 1, r.ws + r.L.seedk, r.ws + r.L.seedv, stream);
}

extern "C" gb_status gb_scorer_step(gb_pool* step_pool, const gb_scorer_config* cfg, const void* weights_dev,
                                    void* workspace_dev, const void* hidden_dev, float* score_out_dev,
                                    gb_stream_t stream) {
  Run r;
  gb_status st = prepare(step_pool, cfg, weights_dev, workspace_dev, stream, &r);
  if (st != GB_OK) return st;
  if (!hidden_dev || ((uintptr_t)hidden_dev & 15) || !score_out_dev)
    return fail(step_pool, GB_ERR_INVALID, "scorer_step: hidden (16-byte aligned) and score_out required");
  if (!step_pool->seeded) return fail(step_pool, GB_ERR_STATE, "scorer_step: step pool not seeded");
  const int* active = step_pool->view.active;
  prof_begin(step_pool, GB_PROF_PROBE, r.st);
  const bool ok = r.input(hidden_dev, r.s.C, active) && r.layers(r.s.C, true, active, score_out_dev);
  if (ok) prof_end(step_pool, GB_PROF_PROBE, r.st);
  step_pool->launches += r.launches;
  st = check_launch(step_pool, "scorer_step");
  if (st != GB_OK) return st;
  return ok ? GB_OK : fail(step_pool, GB_ERR_CUDA, "scorer_step: a launch failed");
}
