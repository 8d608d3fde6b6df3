// Kernels of the prompt pass, the weight repacking and the batch's first arg-max (sm_100a).
//
// Prompt pass (all prompt tokens of a chunk at once):
//   embed_rmsnorm -> [ qkv GEMM (rotates, fills the cache) -> attn_prefill -> o GEMM (+= residual) ->
//   rmsnorm -> gate/up GEMM (SwiGLU) -> down GEMM (+= residual) -> rmsnorm ] x layers ->
//   gather_last_rmsnorm -> LM-head GEMM (fp32 partials) -> lmhead_tile_argmax -> bookkeeping
// (short chunks: the four GEMMs leave partials, and a kernel behind each does what the epilogues do)
// The decode step itself is one persistent kernel (ss_decode_mega.cuh) and shares the small helpers here.
//
// Every kernel starts with griddepcontrol.launch_dependents / griddepcontrol.wait so that the
// next kernel's prologue (for a GEMM: its first weight tiles) overlaps this kernel's body.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <math_constants.h>

#include "ss_gemm.cuh"

namespace ss {

using bf16 = __nv_bfloat16;

// Per-batch device state (arrays of max_batch entries unless noted).
struct RowState {
  int32_t* ctx_len;      // tokens whose keys/values are cached
  int32_t* cur_tok;      // last emitted token, fed by the next step
  int32_t* gen;          // tokens generated so far
  int32_t* active;       // 1 while the row is generating
  int32_t* finished;     // 1 once EOS was emitted
  int32_t* eos_at;       // 0 = natural EOS, t >= 1 = forced EOS at generated index t
  int32_t* row_key;      // the row's key in the sampling counter (its query id inside a group)
  int32_t* out_tokens;   // [max_batch][max_new]
  int32_t* block_table;  // [max_batch][max_pages]
  int32_t* scalars;      // [0] = cap, [1] = n_active
  int max_pages, max_new;
};

struct KvLayout {
  bf16* pool;            // [layer][page][K|V][head][page_tok][Dh]
  size_t layer_stride;   // elements between layers
  size_t page_elems;     // elements per page: 2*H*page_tok*Dh
  int n_pages, H, Dh;
};

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
// Sum over the block; every thread gets the result.  `red` holds >= 32 floats.
__device__ __forceinline__ float block_sum(float v, float* red) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
  v = warp_sum(v);
  __syncthreads();
  if (lane == 0) red[warp] = v;
  __syncthreads();
  float t = (lane < nw) ? red[lane] : 0.f;
  t = warp_sum(t);
  return t;
}

// ------------------------------------------------------------------------------------ weight repacking
// Row-major [rows, K] bf16 -> the GEMM's streaming layout: 32 KiB blocks in (tile, k-block) order, each
// the exact shared-memory image of a 256-row x 64-column tile under the 128-byte swizzle (row r at
// r*128 bytes, its 16-byte chunk c stored at chunk position c ^ (r & 7)).  Each half of a block is
// the image of a 128-row tile, which is what the prompt-pass GEMM loads.  One thread per 16-byte chunk.
// row_off places the source at a row offset of the destination matrix (q,k,v are stacked).  `half`, `step` say where a
// source row goes in it: rows that one thread of an epilogue (or of the decode step) wants together become neighbours.
//   half = 0: row r goes to row_off + r * step (step 1; 2 for gate and up, which alternate)
//   half > 0: the two halves of every 2 * half rows alternate (q and k: the two dimensions of a rotation)
static __global__ void __launch_bounds__(256)
repack_weights_kernel(const uint4* __restrict__ src, long long rows, int K, uint8_t* __restrict__ dst, int row_off,
                      int kb, int half, int step) {
  const int chunks_per_row = K >> 3;
  const long long id = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (id >= rows * chunks_per_row) return;
  const long long sr = id / chunks_per_row;
  const int cc = (int)(id - sr * chunks_per_row);
  long long n = row_off + sr * step;
  if (half > 0) {
    const long long i = sr % (2 * half);
    n = row_off + (sr - i) + (i < half ? 2 * i : 2 * (i - half) + 1);
  }
  const long long tile = n / kTileN;
  const int r = (int)(n % kTileN), k = cc >> 3, c = cc & 7;
  uint8_t* blk = dst + ((size_t)tile * kb + k) * (size_t)kBlockBytes;
  *reinterpret_cast<uint4*>(blk + r * 128 + ((c ^ (r & 7)) << 4)) = src[id];
}

// ------------------------------------------------------------------------------------ rotations
// rope[pos][i] = (cos, sin) of pos * inv_freq[i]: grid (positions), block Dh / 2.  Filled once per context; the kernels
// that rotate read it instead of evaluating a sine and a cosine per (token, head, pair).
static __global__ void rope_table_kernel(const float* __restrict__ inv_freq, float2* __restrict__ rope) {
  float sn, cs;
  sincosf((float)blockIdx.x * inv_freq[threadIdx.x], &sn, &cs);
  rope[(size_t)blockIdx.x * blockDim.x + threadIdx.x] = make_float2(cs, sn);
}

// ------------------------------------------------------------------------------------ embedding + first norm
// A row of d floats (d a multiple of 64, at most 8192) is held by 256 threads as up to 8 x 4 values each: read once,
// normalised from registers.  (Element by element with a second pass over the row: 15 us for a handful of tokens, a chain
// of dependent round trips, and 171 us for 16281 tokens, 0.35 of the copy bandwidth; now 5 and 58 us.)
constexpr int kRowVec = 8;
__device__ __forceinline__ float row_sum_squares(const float4 (&v)[kRowVec], int d4, float* red) {
  float ss = 0.f;
#pragma unroll
  for (int k = 0; k < kRowVec; ++k)
    if (threadIdx.x + k * 256 < d4) ss += v[k].x * v[k].x + v[k].y * v[k].y + v[k].z * v[k].z + v[k].w * v[k].w;
  return block_sum(ss, red);
}
__device__ __forceinline__ void store_normed(const float4 (&v)[kRowVec], int d4, float inv, const bf16* __restrict__ g, bf16* __restrict__ x) {
#pragma unroll
  for (int k = 0; k < kRowVec; ++k) {
    const int i = threadIdx.x + k * 256;
    if (i < d4) {
      const uint2 gb = __ldg(reinterpret_cast<const uint2*>(g) + i);
      const float2 g0 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&gb.x));
      const float2 g1 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&gb.y));
      uint2 o;
      o.x = pack_bf16x2(v[k].x * inv * g0.x, v[k].y * inv * g0.y);
      o.y = pack_bf16x2(v[k].z * inv * g1.x, v[k].w * inv * g1.y);
      reinterpret_cast<uint2*>(x)[i] = o;
    }
  }
}

// h[t] = E[token]; x[t] = RMSNorm(h[t]) * g over T prompt tokens.
static __global__ void __launch_bounds__(256)
embed_rmsnorm_kernel(const int32_t* __restrict__ tokens, const bf16* __restrict__ E, const bf16* __restrict__ g, float* __restrict__ h,
                     bf16* __restrict__ x, int d, float eps, int vocab) {
  __shared__ float red[32];
  pdl_launch_dependents();
  pdl_wait();
  const size_t r = blockIdx.x;
  int tok = tokens[r];
  if (tok < 0 || tok >= vocab) tok = 0;
  const int d4 = d >> 2;
  float4 v[kRowVec];
#pragma unroll
  for (int k = 0; k < kRowVec; ++k) {
    const int i = threadIdx.x + k * 256;
    if (i < d4) {
      const uint2 e = __ldg(reinterpret_cast<const uint2*>(E + (size_t)tok * d) + i);
      const float2 e0 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&e.x));
      const float2 e1 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&e.y));
      v[k] = make_float4(e0.x, e0.y, e1.x, e1.y);
      reinterpret_cast<float4*>(h + r * d)[i] = v[k];
    }
  }
  const float inv = rsqrtf(row_sum_squares(v, d4, red) / d + eps);
  store_normed(v, d4, inv, g, x + r * d);
}

// ------------------------------------------------------------------------------------ LM head argmax
// Stage 1, grid (n_tiles of the vocabulary, rows / kArgmaxRows), block 128 (thread = vocabulary row of the tile):
// logits from partials for the block's rows of the batch, optional dump, and the tile's best (value, id)
// per batch row; the lowest id wins a tie; EOS is left out when the row has a forced-EOS schedule.
// Stage 2 (inside bookkeeping_kernel) picks the best tile per row.
__device__ __forceinline__ uint32_t float_order_key(float f) {      // monotone float -> uint32
  const uint32_t u = __float_as_uint(f);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

// ---- sampling at a temperature (Sec. 4.2 generates at T = 0.5) ------------------------------------------
// A draw from softmax(logits / T) is taken as argmax_v(logit_v / T + g_v) with Gumbel noise g_v = -log(-log(u_v)):
// every u_v comes from the counter-based generator Philox4x32-10 (Salmon et al., SC'11) at counter
// (vocabulary id, index of the generated token, row key, 0) and key (seed), so the arg-max machinery -- per
// tile, then over tiles, in any order -- yields the same token as a sequential draw would.
struct SampleCfg {
  float inv_temp;        // 1 / T, or 0 for greedy decoding
  uint32_t seed_lo, seed_hi;
};

__device__ __forceinline__ uint32_t philox4x32_10_word0(uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3, uint32_t k0,
                                                        uint32_t k1) {
  constexpr uint32_t M0 = 0xD2511F53u, M1 = 0xCD9E8D57u, W0 = 0x9E3779B9u, W1 = 0xBB67AE85u;
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    const uint32_t hi0 = __umulhi(M0, c0), lo0 = M0 * c0;
    const uint32_t hi1 = __umulhi(M1, c2), lo1 = M1 * c2;
    c0 = hi1 ^ c1 ^ k0;
    c1 = lo1;
    c2 = hi0 ^ c3 ^ k1;
    c3 = lo0;
    k0 += W0;
    k1 += W1;
  }
  return c0;
}
// The value whose arg-max decides the token: logit / T + Gumbel noise, or the logit itself (greedy).
__device__ __forceinline__ float sampled_value(float logit, const SampleCfg& sc, int v, int gen_index, int row_key) {
  const uint32_t w = philox4x32_10_word0((uint32_t)v, (uint32_t)gen_index, (uint32_t)row_key, 0u, sc.seed_lo, sc.seed_hi);
  const float u = ((float)(w >> 9) + 0.5f) * (1.0f / 8388608.0f);      // 24 significant bits, never 0 or 1
  return fmaf(logit, sc.inv_temp, -logf(-logf(u)));
}
__device__ __forceinline__ float decision_value(float logit, const SampleCfg& sc, int v, int gen_index, int row_key) {
  return sc.inv_temp == 0.f ? logit : sampled_value(logit, sc, v, gen_index, row_key);
}

constexpr int kArgmaxRows = 8;             // one after the other in a block: 100 rows by one block each took 92 us
static __global__ void __launch_bounds__(128)
lmhead_tile_argmax_kernel(const float* __restrict__ partial, SplitInfo sp, RowState st, float* __restrict__ dump_logits,
                          float* __restrict__ tile_val, int32_t* __restrict__ tile_idx, int B, int vocab, int n_tiles,
                          int eos_id, SampleCfg sc) {
  __shared__ uint32_t s_key[4][kArgmaxRows];
  __shared__ int s_id[4][kArgmaxRows];
  pdl_launch_dependents();
  pdl_wait();
  const int tile = blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int v = tile * 128 + threadIdx.x;
  const int r_lo = blockIdx.y * kArgmaxRows, r_hi = min(B, r_lo + kArgmaxRows);
  for (int r = r_lo; r < r_hi; ++r) {
    uint32_t key = 0;                              // below every real key
    if (st.active[r]) {
      if (v < vocab) {
        const float lg = sum_partials(partial, sp, v, r);
        if (dump_logits) dump_logits[(size_t)r * vocab + v] = lg;
        if (!(st.eos_at[r] > 0 && v == eos_id))
          key = float_order_key(decision_value(lg, sc, v, st.gen[r] + 1, st.row_key[r]));
      }
      const uint32_t best = __reduce_max_sync(0xffffffffu, key);
      const uint32_t who = __ballot_sync(0xffffffffu, key == best);
      if (lane == 0) {
        s_key[warp][r - r_lo] = best;
        s_id[warp][r - r_lo] = tile * 128 + warp * 32 + (__ffs(who) - 1);     // lowest lane = lowest id
      }
    }
  }
  __syncthreads();
  const int k = threadIdx.x, r = r_lo + k;
  if (r < r_hi && st.active[r]) {
    uint32_t bk = s_key[0][k];
    int bi = s_id[0][k];
#pragma unroll
    for (int w = 1; w < 4; ++w)
      if (s_key[w][k] > bk) { bk = s_key[w][k]; bi = s_id[w][k]; }     // warps ascend in id: '>' keeps the lowest
    tile_val[(size_t)r * n_tiles + tile] = __uint_as_float(bk);       // order key, bit-cast
    tile_idx[(size_t)r * n_tiles + tile] = bi;
  }
}

// ------------------------------------------------------------------------------------ step bookkeeping
// One block of 1024 threads; warp w serves rows w, w+32, ...: final argmax over the vocabulary
// tiles, then the row's state update.  is_prefill: the prompt has just been cached (ctx_len set
// by the host) and this is generated token 1; otherwise the fed token becomes part of the cache.
static __global__ void __launch_bounds__(1024)
bookkeeping_kernel(RowState st, const float* __restrict__ tile_val, const int32_t* __restrict__ tile_idx, int n_tiles,
                   const int32_t* __restrict__ forced, int32_t* __restrict__ next_tokens, int32_t* __restrict__ dump_choice,
                   int B, int eos_id, int is_prefill) {
  __shared__ int s_still;
  pdl_launch_dependents();
  pdl_wait();
  if (threadIdx.x == 0) s_still = 0;
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int still = 0;
  for (int r = warp; r < B; r += 32) {
    int tok = eos_id;
    if (st.active[r]) {
      uint32_t bk = 0;
      int bi = 0x7fffffff;
      for (int t = lane; t < n_tiles; t += 32) {
        const uint32_t k = __float_as_uint(tile_val[(size_t)r * n_tiles + t]);
        const int id = tile_idx[(size_t)r * n_tiles + t];
        if (k > bk || (k == bk && id < bi)) { bk = k; bi = id; }
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const uint32_t ok = __shfl_xor_sync(0xffffffffu, bk, o);
        const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
        if (ok > bk || (ok == bk && oi < bi)) { bk = ok; bi = oi; }
      }
      if (lane == 0) {
        if (!is_prefill) st.ctx_len[r] += 1;
        const int cap = st.scalars[0];
        const int gidx = st.gen[r] + 1;               // 1-based index of the token being emitted
        tok = (bi == 0x7fffffff) ? 0 : bi;
        if (dump_choice) dump_choice[r] = tok;
        if (st.eos_at[r] > 0 && gidx == st.eos_at[r]) tok = eos_id;
        if (forced) tok = forced[r];
        st.out_tokens[(size_t)r * st.max_new + (gidx - 1)] = tok;
        st.gen[r] = gidx;
        st.cur_tok[r] = tok;
        if (tok == eos_id) { st.finished[r] = 1; st.active[r] = 0; }
        else if (gidx >= cap) { st.active[r] = 0; }
        else still += 1;
      }
    }
    if (lane == 0 && next_tokens) next_tokens[r] = tok;
  }
  if (lane == 0 && still) atomicAdd(&s_still, still);
  __syncthreads();
  if (threadIdx.x == 0) st.scalars[1] = s_still;
}

// ------------------------------------------------------------------------------------ prompt-pass kernels
// x[t] = RMSNorm(h[t]) * g over T tokens.
static __global__ void __launch_bounds__(256)
rmsnorm_kernel(const float* __restrict__ h, const bf16* __restrict__ g, bf16* __restrict__ x, int d, float eps) {
  __shared__ float red[32];
  pdl_launch_dependents();
  pdl_wait();
  const size_t r = blockIdx.x;
  const int d4 = d >> 2;
  float4 v[kRowVec];
#pragma unroll
  for (int k = 0; k < kRowVec; ++k)
    if (threadIdx.x + k * 256 < d4) v[k] = reinterpret_cast<const float4*>(h + r * d)[threadIdx.x + k * 256];
  const float inv = rsqrtf(row_sum_squares(v, d4, red) / d + eps);
  store_normed(v, d4, inv, g, x + r * d);
}

// Gather each sequence's last token: h_last[s] = h[last[s]]; x_last[s] = RMSNorm(h_last[s]) * g.
static __global__ void __launch_bounds__(256)
gather_last_rmsnorm_kernel(const float* __restrict__ h, const int32_t* __restrict__ last_tok, float* __restrict__ h_out,
                           const bf16* __restrict__ g, bf16* __restrict__ x_out, float* __restrict__ dump_hidden,
                           int d, float eps) {
  __shared__ float red[32];
  pdl_launch_dependents();
  pdl_wait();
  const size_t s = blockIdx.x, t = (size_t)last_tok[s];
  const int d4 = d >> 2;
  float4 v[kRowVec];
#pragma unroll
  for (int k = 0; k < kRowVec; ++k) {
    const int i = threadIdx.x + k * 256;
    if (i < d4) {
      v[k] = reinterpret_cast<const float4*>(h + t * d)[i];
      reinterpret_cast<float4*>(h_out + s * d)[i] = v[k];
      if (dump_hidden) {                             // the caller's buffer: no alignment beyond a float's
        float* o = dump_hidden + s * d + (size_t)i * 4;
        o[0] = v[k].x; o[1] = v[k].y; o[2] = v[k].z; o[3] = v[k].w;
      }
    }
  }
  const float inv = rsqrtf(row_sum_squares(v, d4, red) / d + eps);
  store_normed(v, d4, inv, g, x_out + s * d);
}

// ---- short prompts (chunks of at most kShortTokens tokens): every projection is split over all SMs along K as well and
// leaves fp32 partials [slot][token][128 rows]; these kernels add them (four consecutive outputs per thread) and do what
// the epilogues of the paired GEMM do.  With a CTA per 128-row tile the o and down projections ran on 32 CTAs of 148 and
// took 50 us each for 61 tokens (7B shape); the whole prompt pass of 8 layers went from 1.89 to 0.91 ms.  Up to 256 tokens the
// paired GEMM has one token tile, so 16 to 86 units for 74 pairs: 150 / 200 / 256 tokens, 6 layers, 842 / 888 / 981
// against 1306 / 1357 / 1406 us (300 tokens paired: 1591).
constexpr int kShortTokens = 256;

// Partials of outputs n0 .. n0 + 3 (inside one 128-row tile) for token tok, added in CTA order.
// t: the tile's table entry.
__device__ __forceinline__ float4 sum_partials4(const float* __restrict__ partial, const SplitInfo& s, const int4 t, int n0, int tok) {
  const size_t slot_stride = (size_t)s.NT * 128, cta_stride = slot_stride * s.max_seg;
  const size_t off = (size_t)tok * 128 + (n0 & 127);
  float4 x = __ldcg(reinterpret_cast<const float4*>(partial + (size_t)t.x * slot_stride + off));
  for (int c = t.y; c <= t.z; c += 4) {
    float4 u[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) u[j] = __ldcg(reinterpret_cast<const float4*>(partial + (size_t)min(c + j, t.z) * cta_stride + off));
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (c + j <= t.z) { x.x += u[j].x; x.y += u[j].y; x.z += u[j].z; x.w += u[j].w; }
  }
  return x;
}

// grid (T, ceil(3d / 1024)), block 256
static __global__ void __launch_bounds__(256)
short_qkv_kernel(const float* __restrict__ partial, SplitInfo sp, GemmArgs a) {
  pdl_launch_dependents();
  const int t = blockIdx.x, n = (blockIdx.y * 256 + threadIdx.x) * 4;
  if (n >= 3 * a.d) return;
  const int sec = n / a.d, in = n - sec * a.d, hd = in / a.Dh, e = in - hd * a.Dh;
  const int4 seg = __ldg(reinterpret_cast<const int4*>(sp.tiles) + (n >> 7));
  pdl_wait();
  float4 x = sum_partials4(partial, sp, seg, n, t);
  if (sec < 2) {
    const float2* rope = a.rope + (size_t)a.tok_pos[t] * (a.Dh >> 1) + (e >> 1);
    const float2 c0 = __ldg(rope), c1 = __ldg(rope + 1);
    x = make_float4(x.x * c0.x - x.y * c0.y, x.y * c0.x + x.x * c0.y, x.z * c1.x - x.w * c1.y, x.w * c1.x + x.z * c1.y);
  }
  const uint2 w = make_uint2(pack_bf16x2(x.x, x.y), pack_bf16x2(x.z, x.w));
  *reinterpret_cast<uint2*>(reinterpret_cast<bf16*>(a.out) + (size_t)t * 3 * a.d + n) = w;
  if (sec > 0) {
    const int slot = a.tok_slot[t];
    *reinterpret_cast<uint2*>(reinterpret_cast<bf16*>(a.kv_layer) + (size_t)(slot / kPageTokens) * a.page_elems +
                              ((size_t)((sec - 1) * a.H + hd) * kPageTokens + slot % kPageTokens) * a.Dh + e) = w;
  }
}

// h[t] += projection; x[t] = RMSNorm(h[t]) * g.  grid (T), block 1024: few blocks, so every thread has only one or two
// groups of four outputs, and what does not depend on the projection is read before the wait for it.
static __global__ void __launch_bounds__(1024)
short_residual_kernel(const float* __restrict__ partial, SplitInfo sp, float* __restrict__ h, const bf16* __restrict__ g,
                      bf16* __restrict__ x, int d, float eps) {
  __shared__ float red[32];
  pdl_launch_dependents();
  const size_t t = blockIdx.x;
  const int d4 = d >> 2;
  uint2 gb[2];
  int4 seg[2];
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    const int i = min((int)threadIdx.x + k * 1024, d4 - 1);
    gb[k] = __ldg(reinterpret_cast<const uint2*>(g) + i);
    seg[k] = __ldg(reinterpret_cast<const int4*>(sp.tiles) + (i >> 5));
  }
  pdl_wait();
  float4 v[2];
  float ss = 0.f;
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    const int i = threadIdx.x + k * 1024;
    if (i < d4) {
      const float4 h4 = __ldcg(reinterpret_cast<const float4*>(h + t * d) + i), p = sum_partials4(partial, sp, seg[k], i * 4, (int)t);
      v[k] = make_float4(h4.x + p.x, h4.y + p.y, h4.z + p.z, h4.w + p.w);
      reinterpret_cast<float4*>(h + t * d)[i] = v[k];
      ss += v[k].x * v[k].x + v[k].y * v[k].y + v[k].z * v[k].z + v[k].w * v[k].w;
    }
  }
  const float inv = rsqrtf(block_sum(ss, red) / d + eps);
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    const int i = threadIdx.x + k * 1024;
    if (i < d4) {
      const float2 g0 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&gb[k].x));
      const float2 g1 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&gb[k].y));
      reinterpret_cast<uint2*>(x + t * d)[i] = make_uint2(pack_bf16x2(v[k].x * inv * g0.x, v[k].y * inv * g0.y),
                                                          pack_bf16x2(v[k].z * inv * g1.x, v[k].w * inv * g1.y));
    }
  }
}

// grid (T, ceil(2F / 1024)), block 256
static __global__ void __launch_bounds__(256)
short_swiglu_kernel(const float* __restrict__ partial, SplitInfo sp, bf16* __restrict__ act, int F) {
  pdl_launch_dependents();
  const int t = blockIdx.x, n = (blockIdx.y * 256 + threadIdx.x) * 4;
  if (n >= 2 * F) return;
  const int4 seg = __ldg(reinterpret_cast<const int4*>(sp.tiles) + (n >> 7));
  pdl_wait();
  const float4 x = sum_partials4(partial, sp, seg, n, t);               // gate, up, gate, up
  *reinterpret_cast<uint32_t*>(act + (size_t)t * F + (n >> 1)) =
      pack_bf16x2(x.x / (1.f + __expf(-x.x)) * x.y, x.z / (1.f + __expf(-x.z)) * x.w);
}

// Causal attention over one prompt on tcgen05.  CTA = (128 queries, head, sequence), one thread per query row; keys and
// values come 128 at a time by TMA (128-byte swizzle) straight from the packed q,k,v operand.  Scores S = Q K^T (M = 128
// queries, N = 128 keys) land in tensor memory, every thread reads its row, takes the running maximum and the weights
// (fp32; rounded to bf16 as the A operand of the second product, as before), and O = P V (values as the MN-major B
// operand, so nothing is transposed) is added to a running sum in registers.  P overwrites the keys at head size 128:
// 96 KiB of shared memory and 256 columns of tensor memory, so two CTAs share an SM and one computes while the other's
// loads and MMAs run.
// Why: the warp-level mma of the first version is a sixteenth of tcgen05's rate on this part and its operands went
// through a transposition in shared memory (630 -> 229 us per layer, 86 prompts of 96 to 288 tokens, 32 heads x 128).
constexpr int kAttnTile = 128;             // queries per CTA, keys per step
constexpr int kAttnBlock = kAttnTile * 128;    // one [128 rows x 64 columns] operand block: 16 KiB

template <int DH> constexpr int attn_prefill_smem() {
  return 2048 + (3 * (DH / 64) + (DH == 128 ? 0 : 2)) * kAttnBlock;
}

// Instruction descriptor as umma_idesc_bf16, with B (the values) MN-major.
__host__ __device__ constexpr uint32_t umma_idesc_bf16_b_mn(int n, int m) { return umma_idesc_bf16(n, m) | (1u << 16); }
// Shared-memory descriptor of an MN-major operand under the 128-byte swizzle: 64-element runs along N, rows (K) of 128
// bytes, 8-row groups 1024 bytes apart, the next 64 elements of N one block further.
__device__ __forceinline__ uint64_t smem_desc_mn_sw128(uint32_t saddr, uint32_t n_block_bytes) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr >> 4) & 0x3FFF);
  d |= (uint64_t)(n_block_bytes >> 4) << 16;
  d |= (uint64_t)(1024 >> 4) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)2 << 61;
  return d;
}
__device__ __forceinline__ void sts128(uint32_t addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
  asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(a), "r"(b), "r"(c), "r"(d) : "memory");
}

struct AttnPrefillSmem {
  uint64_t loaded, mma_done;
  uint32_t tmem_base, pad;
};

template <int DH>
__global__ void __launch_bounds__(128, 2)
attn_prefill_kernel(const __grid_constant__ CUtensorMap map_qkv, const int32_t* __restrict__ cu_seqlens, bf16* __restrict__ out, int d,
                    uint32_t* status, long long limit) {
  constexpr int NB = DH / 64;                      // 64-column blocks per operand row
  constexpr uint32_t kTmemCols = 256;              // scores, then outputs
  extern __shared__ uint8_t smem_raw[];
  AttnPrefillSmem* sm = reinterpret_cast<AttnPrefillSmem*>(smem_raw);
  const int hd = blockIdx.y, s = blockIdx.z;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  pdl_launch_dependents();
  const int seq0 = cu_seqlens[s], len = cu_seqlens[s + 1] - seq0;
  const int qt0 = (int)(gridDim.x - 1 - blockIdx.x) * kAttnTile;          // the longest rows first
  if (qt0 >= len) return;
  const uint32_t q_s = (smem_u32(smem_raw) + (uint32_t)sizeof(AttnPrefillSmem) + 1023u) & ~1023u;
  const uint32_t k_s = q_s + NB * kAttnBlock, v_s = k_s + NB * kAttnBlock;
  const uint32_t p_s = DH == 128 ? k_s : v_s + NB * kAttnBlock;
  const uint32_t loaded = smem_u32(&sm->loaded), mma_done = smem_u32(&sm->mma_done);
  if (threadIdx.x == 0) {
    mbar_init(loaded, 1);
    mbar_init(mma_done, 1);
    fence_barrier_init();
    tma_prefetch_desc(&map_qkv);
  }
  if (warp == 0) {
    tmem_alloc(smem_u32(&sm->tmem_base), kTmemCols);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = sm->tmem_base, tmem_row = tmem + ((uint32_t)(warp * 32) << 16);
  pdl_wait();

  uint64_t hint;
  asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(hint));
  auto load_kv = [&](int kt0, uint32_t more) {     // thread 0: the keys and values of a step
    mbar_expect_tx(loaded, 2u * NB * kAttnBlock + more);
    for (int b = 0; b < NB; ++b) {
      tma_load_2d(k_s + b * kAttnBlock, &map_qkv, loaded, d + hd * DH + b * 64, seq0 + kt0, hint);
      tma_load_2d(v_s + b * kAttnBlock, &map_qkv, loaded, 2 * d + hd * DH + b * 64, seq0 + kt0, hint);
    }
  };
  if (threadIdx.x == 0) {
    load_kv(0, NB * kAttnBlock);
    for (int b = 0; b < NB; ++b) tma_load_2d(q_s + b * kAttnBlock, &map_qkv, loaded, hd * DH + b * 64, seq0 + qt0, hint);
  }

  const int row = threadIdx.x, pos = qt0 + row;    // this thread's query
  const float qscale = rsqrtf((float)DH) * 1.4426950408889634f;
  float o[DH];
#pragma unroll
  for (int e = 0; e < DH; ++e) o[e] = 0.f;
  float m = -CUDART_INF_F, l = 0.f;
  const int k_end = min(len, qt0 + kAttnTile);     // causal: keys up to the tile's last query
  uint32_t n_load = 0, n_mma = 0;
  bool ok = true;
  for (int kt0 = 0; kt0 < k_end; kt0 += kAttnTile) {
    ok = mbar_wait(loaded, n_load++ & 1u, status, kStatusProducerTimeout, limit);
    if (ok && threadIdx.x == 0) {
      tc_fence_after();
      const uint32_t idesc = umma_idesc_bf16(kAttnTile);
#pragma unroll
      for (int kk = 0; kk < DH / 16; ++kk) {
        const uint32_t at = (uint32_t)((kk >> 2) * kAttnBlock);
        umma_bf16(tmem, smem_desc_sw128(q_s + at) + (uint64_t)((kk & 3) * 2), smem_desc_sw128(k_s + at) + (uint64_t)((kk & 3) * 2), idesc,
                  kk ? 1u : 0u);
      }
      umma_commit(mma_done);
    }
    ok = ok && mbar_wait(mma_done, n_mma++ & 1u, status, kStatusMmaTimeout, limit);
    if (!__syncthreads_and(ok)) { ok = false; break; }
    tc_fence_after();
    // keys this row may see in the step: all, or up to its own position (rows beyond the prompt are never stored)
    const int vis = min(kAttnTile, pos - kt0 + 1);
    float mx = m;
#pragma unroll 1
    for (int c = 0; c < kAttnTile; c += 64) {
      uint32_t v[64];
      tmem_ld64(tmem_row + c, v);
#pragma unroll
      for (int j = 0; j < 64; ++j) mx = fmaxf(mx, c + j < vis ? __uint_as_float(v[j]) * qscale : -CUDART_INF_F);
    }
    const float mr = mx == -CUDART_INF_F ? 0.f : mx;       // no finite score so far: weights of 0, not NaN
    const float keep = exp2f(m - mr);
    m = mx;
    l *= keep;
#pragma unroll 1
    for (int c = 0; c < kAttnTile; c += 64) {
      uint32_t v[64];
      tmem_ld64(tmem_row + c, v);
      // the row's line of the K-major operand block: eight 16-byte chunks, chunk i at place i ^ (row & 7)
      const uint32_t line = p_s + (uint32_t)((c >> 6) * kAttnBlock + row * 128);
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        uint32_t w[4];
#pragma unroll
        for (int h = 0; h < 4; ++h) {
          const int j = i * 8 + h * 2;
          const float p0 = c + j < vis ? exp2f(__uint_as_float(v[j]) * qscale - mr) : 0.f;
          const float p1 = c + j + 1 < vis ? exp2f(__uint_as_float(v[j + 1]) * qscale - mr) : 0.f;
          l += p0 + p1;
          w[h] = pack_bf16x2(p0, p1);
        }
        sts128(line + (uint32_t)((i ^ (row & 7)) * 16), w[0], w[1], w[2], w[3]);
      }
    }
    if (kt0 + row >= len) {
      // values behind the prompt's end belong to another row: a weight of 0 times what they may hold must stay 0
      for (int b = 0; b < NB; ++b)
#pragma unroll
        for (int i = 0; i < 8; ++i) sts128(v_s + (uint32_t)(b * kAttnBlock + row * 128 + i * 16), 0u, 0u, 0u, 0u);
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    tc_fence_before();
    __syncthreads();
    if (threadIdx.x == 0) {
      tc_fence_after();
      const uint32_t idesc = umma_idesc_bf16_b_mn(DH, kAttnTile);
#pragma unroll
      for (int kk = 0; kk < kAttnTile / 16; ++kk)
        umma_bf16(tmem + kAttnTile, smem_desc_sw128(p_s + (uint32_t)((kk >> 2) * kAttnBlock)) + (uint64_t)((kk & 3) * 2),
                  smem_desc_mn_sw128(v_s + (uint32_t)(kk * 2048), kAttnBlock), idesc, kk ? 1u : 0u);
      umma_commit(mma_done);
    }
    ok = mbar_wait(mma_done, n_mma++ & 1u, status, kStatusMmaTimeout, limit);
    if (!__syncthreads_and(ok)) { ok = false; break; }
    if (threadIdx.x == 0 && kt0 + kAttnTile < k_end) load_kv(kt0 + kAttnTile, 0);
    tc_fence_after();
#pragma unroll
    for (int c = 0; c < DH; c += 64) {
      uint32_t v[64];
      tmem_ld64(tmem_row + kAttnTile + c, v);
#pragma unroll
      for (int j = 0; j < 64; ++j) o[c + j] = fmaf(o[c + j], keep, __uint_as_float(v[j]));
    }
    tc_fence_before();
  }
  if (ok) {
    // the row's bf16 output through the query's shared memory (read by the last MMA), so that rows are stored as whole lines
    const float il = 1.f / l;
#pragma unroll
    for (int b = 0; b < NB; ++b)
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const float* x = o + b * 64 + i * 8;
        sts128(q_s + (uint32_t)(b * kAttnBlock + row * 128 + (i ^ (row & 7)) * 16), pack_bf16x2(x[0] * il, x[1] * il),
               pack_bf16x2(x[2] * il, x[3] * il), pack_bf16x2(x[4] * il, x[5] * il), pack_bf16x2(x[6] * il, x[7] * il));
      }
    __syncwarp();
    constexpr int LPR = DH / 8;                    // lanes per output row, 16 bytes each
    for (int i = 0; i < 32; i += 32 / LPR) {
      const int rr = warp * 32 + i + lane / LPR, ch = lane % LPR;
      uint4 v;
      asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                   : "r"(q_s + (uint32_t)((ch >> 3) * kAttnBlock + rr * 128 + (((ch & 7) ^ (rr & 7)) * 16))) : "memory");
      if (qt0 + rr < len) *reinterpret_cast<uint4*>(out + (size_t)(seq0 + qt0 + rr) * d + hd * DH + ch * 8) = v;
    }
  } else {
    // a wait ran out: copies and MMAs in flight get a bounded time to end before their memory is given up
    const long long t0 = clock64();
    while (clock64() - t0 < 2000000LL) { }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    tmem_dealloc(tmem, kTmemCols);
  }
}

}  // namespace ss
