// Weight-streaming GEMM for sm_100a:  D[n_out, tok] = W[n_out, K] . X[tok, K]^T   (bf16 in, fp32 accumulate)
//
// gemm_wx_kernel: for few tokens (the LM head behind a prompt pass, short prompt chunks, ss_logits_noalloc; the decode
// step has a GEMM of its own).  The weight matrix is the tcgen05 "A" operand (128 rows per tile), the activations are "B"
// (one tile of 16..256 tokens), so a handful of tokens still fills the 128-lane tensor-memory accumulator while every
// weight byte crosses HBM exactly once.  Both operands arrive by TMA (128-byte swizzle) into a multi-stage shared-memory
// ring; one elected thread issues tcgen05.mma; four warps drain the accumulator from tensor memory.
// Work decomposition: the (tile, k-block) iteration space is cut into gridDim.x equal contiguous ranges.  A range that ends
// inside a tile produces a partial sum; all segments are written as fp32 partials which the consumer kernel adds in CTA
// order.
//
// gemm_wx_pair_kernel: for more tokens than one tile, on pairs of CTAs; it finishes the projection in its epilogue.
//
// Programmatic dependent launch: weights never depend on the previous kernel, so the producer
// fills the ring with weight tiles BEFORE griddepcontrol.wait and only then loads activations.
// Every wait on an mbarrier is bounded; on expiry the kernel records a status word and leaves.
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "ss_internal.h"

namespace ss {

// ------------------------------------------------------------------------------------ PTX wrappers
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
// Bounded wait: gives up after `limit` SM cycles, records `code` and returns false.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, uint32_t* status, uint32_t code, long long limit) {
  if (mbar_try_wait(bar, parity)) return true;
  const long long t0 = clock64();
  for (;;) {
    if (mbar_try_wait(bar, parity)) return true;
    if (clock64() - t0 > limit) {
      atomicCAS(status, 0u, code);
      return false;
    }
  }
}
// Bounded wait, by one thread, for a word that another SM sets with release.
__device__ __forceinline__ bool flag_wait(const uint32_t* flag, uint32_t* status, long long limit) {
  const long long t0 = clock64();
  for (;;) {
    uint32_t f;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(f) : "l"(flag) : "memory");
    if (f != 0u) return true;
    if (clock64() - t0 > limit) {
      atomicCAS(status, 0u, (uint32_t)kStatusFlagTimeout);
      return false;
    }
  }
}

__device__ __forceinline__ void fence_barrier_init() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, uint32_t bar, int x, int y,
                                            uint64_t hint) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint"
      " [%0], [%1, {%3, %4}], [%2], %5;"
      :
      : "r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(x), "r"(y), "l"(hint)
      : "memory");
}
// Linear bulk copy global -> shared (both 16-byte aligned, size a multiple of 16).
__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar, uint64_t hint) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], %4;"
      :
      : "r"(dst), "l"(reinterpret_cast<uint64_t>(src)), "r"(bytes), "r"(bar), "l"(hint)
      : "memory");
}
__device__ __forceinline__ void tma_prefetch_desc(const CUtensorMap* map) {
  asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(map)) : "memory");
}

__device__ __forceinline__ void tmem_alloc(uint32_t dst_smem, uint32_t cols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(dst_smem), "r"(cols) : "memory");
}
__device__ __forceinline__ void tmem_relinquish() {
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t cols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(cols) : "memory");
}
// D[tmem] (+)= A[smem] * B[smem], bf16 x bf16 -> fp32, M = 128, N from the instruction descriptor, K = 16.
__device__ __forceinline__ void umma_bf16(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                          uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      :
      : "r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// Arrives on the mbarrier once every tcgen05.mma issued so far by this thread has completed.
__device__ __forceinline__ void umma_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
// 32 lanes x 8 consecutive fp32 columns: thread i of the warp gets lane (base + i), columns c..c+7.
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, float (&v)[8]) {
  uint32_t r0, r1, r2, r3, r4, r5, r6, r7;
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3), "=r"(r4), "=r"(r5), "=r"(r6), "=r"(r7)
               : "r"(taddr)
               : "memory");
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
  v[0] = __uint_as_float(r0); v[1] = __uint_as_float(r1); v[2] = __uint_as_float(r2); v[3] = __uint_as_float(r3);
  v[4] = __uint_as_float(r4); v[5] = __uint_as_float(r5); v[6] = __uint_as_float(r6); v[7] = __uint_as_float(r7);
}
// 32 lanes x 32 consecutive fp32 columns.
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float (&v)[32]) {
  uint32_t r[32];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
        "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
        "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr)
      : "memory");
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}

// 32 lanes x 64 consecutive fp32 columns in one load.
__device__ __forceinline__ void tmem_ld64(uint32_t taddr, uint32_t (&r)[64]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x64.b32 {"
      "%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, "
      "%32, %33, %34, %35, %36, %37, %38, %39, %40, %41, %42, %43, %44, %45, %46, %47, "
      "%48, %49, %50, %51, %52, %53, %54, %55, %56, %57, %58, %59, %60, %61, %62, %63}, [%64];\n"
      "tcgen05.wait::ld.sync.aligned;"
      :
        "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
        "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
        "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31]),
        "=r"(r[32]), "=r"(r[33]), "=r"(r[34]), "=r"(r[35]), "=r"(r[36]), "=r"(r[37]), "=r"(r[38]), "=r"(r[39]),
        "=r"(r[40]), "=r"(r[41]), "=r"(r[42]), "=r"(r[43]), "=r"(r[44]), "=r"(r[45]), "=r"(r[46]), "=r"(r[47]),
        "=r"(r[48]), "=r"(r[49]), "=r"(r[50]), "=r"(r[51]), "=r"(r[52]), "=r"(r[53]), "=r"(r[54]), "=r"(r[55]),
        "=r"(r[56]), "=r"(r[57]), "=r"(r[58]), "=r"(r[59]), "=r"(r[60]), "=r"(r[61]), "=r"(r[62]), "=r"(r[63])
      : "r"(taddr)
      : "memory");
}

// ---- forms for a pair of CTAs on neighbouring SMs working on one accumulator tile (cta_group::2) ---------------
// TMA tile load whose bytes are counted on the mbarrier of the pair's first CTA (the one that issues the MMAs):
// both CTAs execute it with the address of their own copy of the barrier; clearing the CTA-rank bit of the
// shared-window address makes it the first CTA's.  Every CTA loads only its own operand halves.
constexpr uint32_t kPairLeaderMask = 0xFEFFFFFFu;
__device__ __forceinline__ void tma_load_2d_pair(uint32_t dst, const CUtensorMap* map, uint32_t bar, int x, int y,
                                                 uint64_t hint) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint"
      " [%0], [%1, {%3, %4}], [%2], %5;"
      :
      : "r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(bar & kPairLeaderMask), "r"(x), "r"(y), "l"(hint)
      : "memory");
}
__device__ __forceinline__ void tmem_alloc_pair(uint32_t dst_smem, uint32_t cols) {
  asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(dst_smem), "r"(cols) : "memory");
}
__device__ __forceinline__ void tmem_relinquish_pair() {
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc_pair(uint32_t taddr, uint32_t cols) {
  asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(cols) : "memory");
}
// D[tmem of both CTAs] (+)= A * B with M = 256 (128 rows from each CTA's shared memory), N from the descriptor
// (half of the B rows from each CTA), K = 16.  Issued by one thread of the pair's first CTA.
__device__ __forceinline__ void umma_bf16_pair(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                               uint32_t accumulate) {
  const uint32_t z = 0;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, {%5, %5, %5, %5, %5, %5, %5, %5}, p;\n\t}"
      :
      : "r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate), "r"(z)
      : "memory");
}
// Arrives on the same-named mbarrier of both CTAs of the pair once every MMA issued so far has completed.
__device__ __forceinline__ void umma_commit_pair(uint32_t bar) {
  const uint16_t mask = 3;
  asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
               ::"r"(bar), "h"(mask) : "memory");
}
__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t cluster_cta_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}

// Shared-memory matrix descriptor: K-major tile, 128-byte swizzle, rows of 128 bytes,
// 8-row groups 1024 bytes apart.
__device__ __forceinline__ uint64_t smem_desc_sw128(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr >> 4) & 0x3FFF);          // start address
  d |= (uint64_t)1 << 16;                          // leading byte offset (unused with swizzle)
  d |= (uint64_t)(1024 >> 4) << 32;                // stride byte offset between 8-row groups
  d |= (uint64_t)1 << 46;                          // descriptor version (sm_100)
  d |= (uint64_t)2 << 61;                          // layout: SWIZZLE_128B
  return d;
}
// Instruction descriptor: fp32 accumulate, bf16 A and B, both K-major, M = m (128 or 64), N = n.
// Accumulator row i of an M = 128 instruction is tensor-memory lane i; of an M = 64 instruction it is lane
// (i % 16) + 32 * (i / 16), i.e. the first 16 lanes of each warp's lane quarter.
__host__ __device__ constexpr uint32_t umma_idesc_bf16(int n, int m = 128) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(m >> 4) << 24);
}

// ------------------------------------------------------------------------------------ split bookkeeping
__host__ __device__ __forceinline__ long long split_begin(const SplitInfo& s, int c) {
  return (long long)c * s.total / s.gridx;
}
// CTA whose range holds iteration x.
__host__ __device__ __forceinline__ int split_owner(const SplitInfo& s, long long x) {
  int c = (int)(x * s.gridx / s.total);
  while (c + 1 < s.gridx && split_begin(s, c + 1) <= x) ++c;
  return c;
}
// Sum of the fp32 partials of output row n (of n_out) for token `tok`, in CTA order; the tile's segments come from the
// precomputed table.
__device__ __forceinline__ float sum_partials(const float* __restrict__ partial, const SplitInfo& s, int n, int tok) {
  const int4 t = __ldg(reinterpret_cast<const int4*>(s.tiles) + (n >> 7));
  const size_t slot_stride = (size_t)s.NT * 128;
  const size_t off = (size_t)tok * 128 + (n & 127);
  float acc = partial[(size_t)t.x * slot_stride + off];
  const size_t cta_stride = slot_stride * s.max_seg;
  for (int c = t.y; c <= t.z; ++c) acc += partial[(size_t)c * cta_stride + off];
  return acc;
}

// ------------------------------------------------------------------------------------ the kernel
constexpr int kGemmThreads = 192;   // warp 0: TMA producer, warp 1: MMA issuer, warps 2..5: epilogue
constexpr int kGemmMaxStages = 16;

struct GemmSmemHeader {
  uint64_t full[kGemmMaxStages];
  uint64_t empty[kGemmMaxStages];
  uint64_t acc_full[2];
  uint64_t acc_empty[2];
  uint32_t tmem_base;
  uint32_t pad;
};

// internal linkage: the header is compiled into more than one translation unit
static __global__ void __launch_bounds__(kGemmThreads, 1)
gemm_wx_kernel(const __grid_constant__ CUtensorMap map_w, const __grid_constant__ CUtensorMap map_x, GemmArgs a) {
  extern __shared__ uint8_t smem_raw[];
  const GemmPlan& p = a.p;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int cta = blockIdx.x;

  // carve shared memory: header, then 1024-byte aligned stages
  GemmSmemHeader* hdr = reinterpret_cast<GemmSmemHeader*>(smem_raw);
  const uint32_t smem_base = smem_u32(smem_raw);
  const uint32_t stage0 = (smem_base + (uint32_t)sizeof(GemmSmemHeader) + 1023u) & ~1023u;
  const uint32_t a_bytes = kTileM * kTileK * 2;               // 16 KiB
  const uint32_t b_bytes = (uint32_t)p.NT * kTileK * 2;
  const uint32_t stage_bytes = a_bytes + b_bytes;

  const long long total = (long long)p.n_tiles * p.kb;
  const long long it0 = (long long)cta * total / p.gridx;
  const long long it1 = (long long)(cta + 1) * total / p.gridx;
  const int n_it = (int)(it1 - it0);

  if (threadIdx.x == 0) {
    pdl_launch_dependents();
    for (int s = 0; s < p.stages; ++s) {
      mbar_init(smem_u32(&hdr->full[s]), 1);
      mbar_init(smem_u32(&hdr->empty[s]), 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(smem_u32(&hdr->acc_full[b]), 1);
      mbar_init(smem_u32(&hdr->acc_empty[b]), 4);
    }
    fence_barrier_init();
    if (!a.w_tiled) tma_prefetch_desc(&map_w);
    tma_prefetch_desc(&map_x);
  }
  if (warp == 1) {
    tmem_alloc(smem_u32(&hdr->tmem_base), (uint32_t)p.tmem_cols);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = hdr->tmem_base;

  if (warp == 0) {
    // ===================== TMA producer =====================
    if (lane == 0) {
      // weights are streamed once: evict-first; activations are shared by all CTAs: evict-last
      uint64_t hint_w, hint_x;
      asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(hint_w));
      asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(hint_x));
      const int pre = n_it < p.stages ? n_it : p.stages;
      // Repacked weights: the 128-row tile `tile` at k-block `kblk` is one half of the 32 KiB block
      // (tile / 2, kblk), already in the swizzled shared-memory image.
      const uint8_t* w_tiled = reinterpret_cast<const uint8_t*>(a.w_tiled);
      auto w_block = [&](int tile, int kblk) {
        return w_tiled + ((size_t)(tile >> 1) * p.kb + kblk) * (size_t)kBlockBytes + (size_t)(tile & 1) * a_bytes;
      };
      // phase 1: weight tiles of the first ring fill, before the dependency resolves
      for (int i = 0; i < pre; ++i) {
        const long long it = it0 + i;
        const int tile = (int)(it / p.kb), kblk = (int)(it % p.kb);
        const uint32_t full = smem_u32(&hdr->full[i]);
        mbar_expect_tx(full, stage_bytes);
        if (w_tiled) bulk_load(stage0 + i * stage_bytes, w_block(tile, kblk), a_bytes, full, hint_w);
        else tma_load_2d(stage0 + i * stage_bytes, &map_w, full, kblk * kTileK, tile * kTileM, hint_w);
      }
      pdl_wait();
      for (int i = 0; i < pre; ++i) {
        const long long it = it0 + i;
        const int kblk = (int)(it % p.kb);
        tma_load_2d(stage0 + i * stage_bytes + a_bytes, &map_x, smem_u32(&hdr->full[i]), kblk * kTileK, 0, hint_x);
      }
      // phase 2: steady state (second and later passes over the ring)
      int stage = 0, issued = pre;
      uint32_t phase = 1u;
      for (int i = pre; i < n_it; ++i) {
        const long long it = it0 + i;
        const int tile = (int)(it / p.kb), kblk = (int)(it % p.kb);
        if (!mbar_wait(smem_u32(&hdr->empty[stage]), phase ^ 1u, a.status, kStatusProducerTimeout, a.wait_limit)) break;
        const uint32_t full = smem_u32(&hdr->full[stage]);
        mbar_expect_tx(full, stage_bytes);
        if (w_tiled) bulk_load(stage0 + stage * stage_bytes, w_block(tile, kblk), a_bytes, full, hint_w);
        else tma_load_2d(stage0 + stage * stage_bytes, &map_w, full, kblk * kTileK, tile * kTileM, hint_w);
        tma_load_2d(stage0 + stage * stage_bytes + a_bytes, &map_x, full, kblk * kTileK, 0, hint_x);
        if (++stage == p.stages) { stage = 0; phase ^= 1u; }
        ++issued;
      }
      if (issued < n_it) {
        // a wait ran out and the kernel is leaving: the copies still in flight (at most one ring) get a bounded
        // time to land before the CTA's shared memory is given up
        for (int s2 = 0; s2 < p.stages; ++s2) {
          const long long t0 = clock64();
          while (!mbar_try_wait(smem_u32(&hdr->full[s2]), 0u) && !mbar_try_wait(smem_u32(&hdr->full[s2]), 1u) &&
                 clock64() - t0 < 2000000LL) { }
        }
      }
    }
  } else if (warp == 1) {
    // ===================== MMA issuer =====================
    if (lane == 0) {
      pdl_wait();
      const uint32_t idesc = umma_idesc_bf16(p.NT);
      int stage = 0;
      uint32_t phase = 0;
      int seg = 0;
      bool ok = true;
      long long it = it0;
      while (it < it1 && ok) {
        const int tile = (int)(it / p.kb);
        long long seg_end = (long long)(tile + 1) * p.kb;
        if (seg_end > it1) seg_end = it1;
        const int buf = seg & 1;
        const uint32_t use = (uint32_t)(seg >> 1);
        // wait until the epilogue has drained this accumulator buffer (first use passes at once)
        ok = mbar_wait(smem_u32(&hdr->acc_empty[buf]), (use & 1u) ^ 1u, a.status, kStatusMmaTimeout, a.wait_limit);
        if (!ok) break;
        tc_fence_after();
        const uint32_t d_tmem = tmem_base + (uint32_t)(buf * p.NT);
        bool first = true;
        for (; it < seg_end; ++it) {
          ok = mbar_wait(smem_u32(&hdr->full[stage]), phase, a.status, kStatusMmaTimeout, a.wait_limit);
          if (!ok) break;
          tc_fence_after();
          const uint32_t sa = stage0 + stage * stage_bytes;
          const uint64_t da = smem_desc_sw128(sa), db = smem_desc_sw128(sa + a_bytes);
#pragma unroll
          for (int k = 0; k < kTileK / 16; ++k) {
            // +32 bytes per 16-element K step inside the 128-byte swizzled row
            umma_bf16(d_tmem, da + (uint64_t)(k * 2), db + (uint64_t)(k * 2), idesc, (first && k == 0) ? 0u : 1u);
          }
          first = false;
          umma_commit(smem_u32(&hdr->empty[stage]));      // frees the stage when these MMAs retire
          if (++stage == p.stages) { stage = 0; phase ^= 1u; }
        }
        if (!ok) break;
        umma_commit(smem_u32(&hdr->acc_full[buf]));
        ++seg;
      }
    }
  } else {
    // ===================== epilogue (4 warps, one TMEM lane quarter each) =====================
    pdl_wait();
    const int quarter = warp & 3;                 // warps 2,3,4,5 -> lane quarters 2,3,0,1
    const int row = quarter * 32 + lane;          // row inside the 128-row tile
    int seg = 0;
    long long it = it0;
    const int n_valid = a.n_tok < p.NT ? a.n_tok : p.NT;
    while (it < it1) {
      const int tile = (int)(it / p.kb);
      long long seg_end = (long long)(tile + 1) * p.kb;
      if (seg_end > it1) seg_end = it1;
      const int buf = seg & 1;
      const uint32_t use = (uint32_t)(seg >> 1);
      bool ok = mbar_wait(smem_u32(&hdr->acc_full[buf]), use & 1u, a.status, kStatusEpilogueTimeout, a.wait_limit);
      ok = __all_sync(0xffffffffu, ok);           // warp-uniform, and reconverges the warp
      if (!ok) break;
      tc_fence_after();
      const uint32_t taddr = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(buf * p.NT);
      const size_t slot = (size_t)cta * p.max_seg + seg;
      float* dst = a.partial + slot * p.NT * 128 + row;
      for (int c = 0; c < p.NT; c += 8) {
        float v[8];
        tmem_ld8(taddr + c, v);
#pragma unroll
        for (int j = 0; j < 8; ++j)
          if (c + j < n_valid) dst[(size_t)(c + j) * 128] = v[j];
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&hdr->acc_empty[buf]));
      it = seg_end;
      ++seg;
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem_base, (uint32_t)p.tmem_cols);
  }
}

// ------------------------------------------------------------------------------------ the paired kernel
// The prompt-pass GEMM on pairs of CTAs (a cluster of two neighbouring SMs, tcgen05 cta_group::2): the pair
// computes a tile of 256 rows x NT tokens, CTA r of the pair holding weight rows 128 r .. 128 r + 127 (its half of a
// 32 KiB block of the tiled layout) and its half of the tile's tokens in its shared memory, and
// rows 128 r .. of the accumulator in its tensor memory.  One thread of the first CTA issues the MMAs for both.
// Why: with one CTA per tile, 48 KiB written into shared memory and 48 KiB read out of it by the tensor core per
// k-block exceed what the shared memory of one SM moves in the 512 cycles the four MMAs take; in the pair every
// CTA stages 32 KiB per k-block for the same arithmetic.
constexpr int kPairTokens = 256;                                 // largest token tile of the pair (half of it per CTA)
constexpr int kPairThreads = 320;                                // warp 0: TMA producer, warp 1: MMA issuer, warps 2..9: epilogue

// Remote arrival on the first CTA's copy of a barrier (used by the partner's epilogue warps).
__device__ __forceinline__ void mbar_arrive_leader(uint32_t bar) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar & kPairLeaderMask) : "memory");
}

// ---- epilogues that finish a projection.  Weight rows that belong together (the two dimensions of a rotation, gate and
// up of a feature, neighbouring value dimensions) are neighbours in the tiled layout, i.e. on neighbouring lanes of the
// accumulator.  Of 32 tokens the even lane of two takes the first 16 and the odd lane the others: each hands the other
// lane the values it needs, 16 shuffles for 32 values, and then holds both rows of its 16 tokens.
// Writing the fp32 accumulators out for a kernel of its own to rotate (or gate) cost, per layer of 16281 tokens at the
// 7B shape, 222 (258) us of that kernel beside the write: at the copy bandwidth, so it had to go, not to be tuned.
__device__ __forceinline__ void pair_rows(const float (&v)[32], int lane, float (&lo)[16], float (&hi)[16]) {
  const bool odd = lane & 1;
#pragma unroll
  for (int j = 0; j < 16; ++j) {
    const float got = __shfl_xor_sync(0xffffffffu, odd ? v[j] : v[16 + j], 1);
    lo[j] = odd ? got : v[j];
    hi[j] = odd ? v[16 + j] : got;
  }
}
__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi) {
  const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&v);
}

// ---- work of a pair.  The units (256 weight rows, token tile) are numbered group of token tiles by group, inside a group
// with the token tile as the fast index: pairs that run side by side share weight blocks, and a group's activations stay
// in L2 from one round of pairs to the next.  The first `split_units` of them are cut, as one sequence of k-blocks, into
// `ranges` equal contiguous parts, one per pair, so that all pairs end together; the others go to the pairs in turn.
// A unit that is cut belongs to the pair with its first k-blocks; the others leave fp32 partials.  Ranges are dealt in
// reverse, so that an owner waits for pairs of lower index, which the hardware starts no later than the owner.
struct PairSegment {
  int wt, tt;        // weight tile (of 256 rows), token tile
  int k0, k1;        // k-blocks
  int unit;          // its number, where it is of the part that is cut
};
struct PairWalk {
  int it, it1, u;    // next and last k-block of the pair's range; next whole unit
  __device__ __forceinline__ PairWalk(const GemmPlan& p, int pair) {
    const int q = p.ranges - 1 - pair;
    it = it1 = 0;
    if (q >= 0) { it = pair_range(p, q); it1 = pair_range(p, q + 1); }
    u = p.split_units + pair;
  }
  static __device__ __forceinline__ int pair_range(const GemmPlan& p, int q) {
    return (int)((long long)q * p.split_units * p.kb / p.ranges);
  }
  __device__ __forceinline__ bool next(const GemmPlan& p, int n_pairs, PairSegment& s) {
    if (it < it1) {
      s.unit = it / p.kb;
      s.k0 = it - s.unit * p.kb;
      s.k1 = min(p.kb, s.k0 + it1 - it);
      it += s.k1 - s.k0;
    } else {
      const int n_wt = p.n_tiles >> 1;
      if (u >= n_wt * p.tok_tiles) return false;
      s.unit = u;
      s.k0 = 0;
      s.k1 = p.kb;
      u += n_pairs;
    }
    const int n_wt = p.n_tiles >> 1, per_group = p.group * n_wt;
    const int g = s.unit / per_group, in = s.unit - g * per_group, size = min(p.group, p.tok_tiles - g * p.group);
    s.wt = in / size;
    s.tt = g * p.group + in - s.wt * size;
    return true;
  }
};

// The accumulator of 32 tokens, and the partials that others left for it: contributions of the ranges q + 1 .. q + n_more.
// `part`: this warp's rows and the first of the 32 tokens in range q's slab; a slab is [CTA of the pair][token][128 rows].
struct PairParts {
  const float* part;
  size_t slab;
  int n_more;
};
__device__ __forceinline__ void load_acc(uint32_t taddr, int c, const PairParts& pp, float (&v)[32]) {
  tmem_ld32(taddr + c, v);
  for (int m = 1; m <= pp.n_more; ++m) {
    const float* src = pp.part + (size_t)m * pp.slab + (size_t)c * kTileM;
    float u[32];
#pragma unroll
    for (int j = 0; j < 32; ++j) u[j] = __ldcg(src + j * kTileM);
#pragma unroll
    for (int j = 0; j < 32; ++j) v[j] += u[j];
  }
}

// q, k, v: rotation (q, k), one rounding; operand of the prompt-pass attention, and keys and values into the pages.
__device__ __forceinline__ void epilogue_qkv(const GemmArgs& a, uint32_t taddr, const PairParts& pp, int n, int tok0, int c0, int n_valid, int lane) {
  const int sec = n / a.d, in = n - sec * a.d, hd = in / a.Dh, e = (in - hd * a.Dh) & ~1;      // sec, hd: warp-uniform
  const int first = (lane & 1) * 16;
  __nv_bfloat16* out = reinterpret_cast<__nv_bfloat16*>(a.out) + (size_t)sec * a.d + hd * a.Dh + e;
  __nv_bfloat16* kv = reinterpret_cast<__nv_bfloat16*>(a.kv_layer) + (size_t)((max(sec, 1) - 1) * a.H + hd) * kPageTokens * a.Dh + e;
  for (int c = c0; c < n_valid; c += 64) {
    const int mine = tok0 + min(c + lane, n_valid - 1);
    const int pos_l = __ldg(a.tok_pos + mine), slot_l = __ldg(a.tok_slot + mine);
    float v[32], lo[16], hi[16];
    load_acc(taddr, c, pp, v);
    pair_rows(v, lane, lo, hi);
    if (sec < 2) {
      const float2* rope = a.rope + (e >> 1);
#pragma unroll
      for (int j = 0; j < 16; ++j) {
        const int pos = __shfl_sync(0xffffffffu, pos_l, first + j);
        const float2 cs = __ldg(rope + (size_t)pos * (a.Dh >> 1));
        const float x0 = lo[j], x1 = hi[j];
        lo[j] = x0 * cs.x - x1 * cs.y;
        hi[j] = x1 * cs.x + x0 * cs.y;
      }
    }
#pragma unroll
    for (int j = 0; j < 16; ++j) {
      const int slot = __shfl_sync(0xffffffffu, slot_l, first + j);
      if (c + first + j < n_valid) {
        const uint32_t w = pack_bf16x2(lo[j], hi[j]);
        *reinterpret_cast<uint32_t*>(out + (size_t)(tok0 + c + first + j) * 3 * a.d) = w;
        if (sec > 0) *reinterpret_cast<uint32_t*>(kv + (size_t)(slot / kPageTokens) * a.page_elems + (slot % kPageTokens) * a.Dh) = w;
      }
    }
  }
}

// silu(gate) * up, one rounding.
__device__ __forceinline__ void epilogue_swiglu(const GemmArgs& a, uint32_t taddr, const PairParts& pp, int n, int tok0, int c0, int n_valid, int lane) {
  const int F = a.p.n_out >> 1, f = n >> 1, first = (lane & 1) * 16;
  __nv_bfloat16* out = reinterpret_cast<__nv_bfloat16*>(a.out) + (size_t)tok0 * F + f;
  for (int c = c0; c < n_valid; c += 64) {
    float v[32], gate[16], up[16];
    load_acc(taddr, c, pp, v);
    pair_rows(v, lane, gate, up);
#pragma unroll
    for (int j = 0; j < 16; ++j)
      if (f < F && c + first + j < n_valid)
        out[(size_t)(c + first + j) * F] = __float2bfloat16_rn(gate[j] / (1.f + __expf(-gate[j])) * up[j]);
  }
}

// Read-modify-write of the fp32 residual: 32 tokens' loads in flight per round trip.
__device__ __forceinline__ void epilogue_residual(const GemmArgs& a, uint32_t taddr, const PairParts& pp, int n, int tok0, int c0, int n_valid) {
  for (int c = c0; c < n_valid; c += 64) {
    float v[32], h[32];
    float* o = a.residual + (size_t)(tok0 + c) * a.p.n_out + n;
    if (n < a.p.n_out) {
#pragma unroll
      for (int j = 0; j < 32; ++j) h[j] = (c + j < n_valid) ? __ldcg(o + (size_t)j * a.p.n_out) : 0.f;
    }
    load_acc(taddr, c, pp, v);
    if (n < a.p.n_out) {
#pragma unroll
      for (int j = 0; j < 32; ++j)
        if (c + j < n_valid) o[(size_t)j * a.p.n_out] = h[j] + v[j];
    }
  }
}

// Persistent: gridDim.x / 2 pairs, each with the segments of its PairWalk.  Two accumulator buffers of 256 columns: the
// drain of one segment overlaps the MMAs of the next.  Eight epilogue warps per CTA: the drain of the last segment is the
// serial tail of every projection.
static __global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kPairThreads, 1)
gemm_wx_pair_kernel(const __grid_constant__ CUtensorMap map_w, const __grid_constant__ CUtensorMap map_x, const __grid_constant__ GemmArgs a) {
  extern __shared__ uint8_t smem_raw[];
  const GemmPlan& p = a.p;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cluster_cta_rank();          // 0: issues the MMAs; 1: its partner
  const int pair = blockIdx.x >> 1, n_pairs = gridDim.x >> 1;
  GemmSmemHeader* hdr = reinterpret_cast<GemmSmemHeader*>(smem_raw);
  const uint32_t stage0 = (smem_u32(smem_raw) + (uint32_t)sizeof(GemmSmemHeader) + 1023u) & ~1023u;
  const uint32_t a_bytes = kTileM * kTileK * 2, stage_bytes = a_bytes + (uint32_t)p.NT * kTileK;   // half of NT tokens
  PairWalk walk(p, pair);
  PairSegment s{};

  if (threadIdx.x == 0) {
    pdl_launch_dependents();
    for (int i = 0; i < p.stages; ++i) {
      mbar_init(smem_u32(&hdr->full[i]), 1);
      mbar_init(smem_u32(&hdr->empty[i]), 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(smem_u32(&hdr->acc_full[b]), 1);
      mbar_init(smem_u32(&hdr->acc_empty[b]), 16);   // eight epilogue warps of each CTA (used in the first CTA only)
    }
    fence_barrier_init();
    tma_prefetch_desc(&map_w);
    tma_prefetch_desc(&map_x);
  }
  if (warp == 1) {
    tmem_alloc_pair(smem_u32(&hdr->tmem_base), 2u * kPairTokens);
    tmem_relinquish_pair();
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();                                // both CTAs' barriers exist before either signals the other's
  tc_fence_after();
  const uint32_t tmem_base = hdr->tmem_base;

  if (warp == 0) {
    // ===================== TMA producer (one per CTA) =====================
    if (lane == 0) {
      // Weights of up to two token tiles are read once, or twice at the same time; with more tiles, pairs and groups that come to
      // a block later find it in L2 (16000 tokens, 6 layers: 37.4 ms evict-first, 34.9 normal; 512: 1490 and 1525 us).
      uint64_t hint_w, hint_x;
      if (p.tok_tiles <= 2) asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(hint_w));
      else asm volatile("createpolicy.fractional.L2::evict_normal.b64 %0, 1.0;" : "=l"(hint_w));
      asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(hint_x));
      // the tiled weights seen as lines of 128 bytes: this CTA's half of block (wt, k) starts at line
      // (wt * kb + k) * 256 + rank * 128 and is 128 lines long; the first CTA's barrier counts the bytes of all four
      // loads of a stage (two per CTA)
      auto load_w = [&](int stage, int i) {
        const uint32_t full = smem_u32(&hdr->full[stage]);
        if (rank == 0) mbar_expect_tx(full, 2u * stage_bytes);
        tma_load_2d_pair(stage0 + (uint32_t)stage * stage_bytes, &map_w, full, 0, (s.wt * p.kb + i) * kTileN + (int)rank * kTileM, hint_w);
      };
      auto load_x = [&](int stage, int i) {
        tma_load_2d_pair(stage0 + (uint32_t)stage * stage_bytes + a_bytes, &map_x, smem_u32(&hdr->full[stage]), i * kTileK,
                         s.tt * p.NT + (int)rank * (p.NT >> 1), hint_x);
      };
      int stage = 0, gi = 0;
      uint32_t phase = 0;
      bool ok = true;
      while (ok && walk.next(p, n_pairs, s)) {
        int i = s.k0;
        if (gi == 0) {
          // the weights of the first ring fill do not depend on the kernel in front
          const int pre = min(p.stages, s.k1 - s.k0);
          for (int j = 0; j < pre; ++j) load_w(j, i + j);
          pdl_wait();
          for (int j = 0; j < pre; ++j) load_x(j, i + j);
          i += pre;
          gi = pre;
          stage = pre == p.stages ? 0 : pre;
          phase = pre == p.stages ? 1u : 0u;
        }
        for (; i < s.k1; ++i, ++gi) {
          if (gi >= p.stages && !(ok = mbar_wait(smem_u32(&hdr->empty[stage]), phase ^ 1u, a.status, kStatusProducerTimeout, a.wait_limit))) break;
          load_w(stage, i);
          load_x(stage, i);
          if (++stage == p.stages) { stage = 0; phase ^= 1u; }
        }
      }
      if (!ok) {
        // a wait ran out: give the copies in flight a bounded time to land before the shared memory is given up
        const long long t0 = clock64();
        while (clock64() - t0 < 2000000LL) { }
      }
    }
  } else if (warp == 1) {
    // ===================== MMA issuer (first CTA of the pair only) =====================
    if (lane == 0 && rank == 0) {
      pdl_wait();                                        // the kernel in front does not count against the limit
      const uint32_t idesc = umma_idesc_bf16(p.NT, 256);
      int stage = 0;
      uint32_t phase = 0;
      bool ok = true;
      for (int r = 0; ok && walk.next(p, n_pairs, s); ++r) {
        const int buf = r & 1;
        // both CTAs' epilogues have drained this buffer (its first use passes at once)
        ok = mbar_wait(smem_u32(&hdr->acc_empty[buf]), ((uint32_t)(r >> 1) & 1u) ^ 1u, a.status, kStatusMmaTimeout, a.wait_limit);
        if (!ok) break;
        tc_fence_after();
        const uint32_t d_tmem = tmem_base + (uint32_t)(buf * kPairTokens);
        for (int i = s.k0; i < s.k1; ++i) {
          ok = mbar_wait(smem_u32(&hdr->full[stage]), phase, a.status, kStatusMmaTimeout, a.wait_limit);
          if (!ok) break;
          tc_fence_after();
          const uint32_t sa = stage0 + (uint32_t)stage * stage_bytes;
          const uint64_t da = smem_desc_sw128(sa), db = smem_desc_sw128(sa + a_bytes);
#pragma unroll
          for (int k = 0; k < kTileK / 16; ++k)
            umma_bf16_pair(d_tmem, da + (uint64_t)(k * 2), db + (uint64_t)(k * 2), idesc, (i == s.k0 && k == 0) ? 0u : 1u);
          umma_commit_pair(smem_u32(&hdr->empty[stage]));    // frees the stage in both CTAs when these MMAs retire
          if (++stage == p.stages) { stage = 0; phase ^= 1u; }
        }
        if (ok) umma_commit_pair(smem_u32(&hdr->acc_full[buf]));
      }
    }
  } else {
    // ===================== epilogue: this CTA's 128 rows x NT tokens ====================================
    // eight warps, two per tensor-memory lane quarter, which take the 32-token groups in turn
    pdl_wait();
    const int quarter = warp & 3, c0 = warp >= 6 ? 32 : 0;
    const int row = quarter * 32 + lane;
    const size_t slab = (size_t)2 * p.NT * kTileM;
    for (int r = 0; walk.next(p, n_pairs, s); ++r) {
      const int buf = r & 1;
      const int tok0 = s.tt * p.NT;
      const int n_valid = min(a.n_tok - tok0, p.NT);
      bool ok = mbar_wait(smem_u32(&hdr->acc_full[buf]), (uint32_t)(r >> 1) & 1u, a.status, kStatusEpilogueTimeout, a.wait_limit);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
      tc_fence_after();
      const uint32_t taddr = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(buf * kPairTokens);
      const int q = p.ranges - 1 - pair;
      float* mine = a.partial + ((size_t)max(q, 0) * 2 + rank) * p.NT * kTileM + row;
      // flags: one word per range, CTA and epilogue warp
      uint32_t* flag = a.pair_flag + (max(q, 0) * 2 + (int)rank) * 8 + (warp - 2);
      if (s.k0 > 0) {
        // the rest of a unit that another pair began
        for (int c = c0; c < n_valid; c += 64) {
          float v[32];
          tmem_ld32(taddr + c, v);
#pragma unroll
          for (int j = 0; j < 32; ++j) __stcg(mine + (size_t)(c + j) * kTileM, v[j]);
        }
        __syncwarp();
        if (lane == 0) asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(flag), "r"(1u) : "memory");
      } else {
        PairParts pp = {mine, slab, 0};
        if (s.k1 < p.kb) {
          // ranges behind this one until the unit's end
          while (PairWalk::pair_range(p, q + 1 + pp.n_more) < (s.unit + 1) * p.kb) ++pp.n_more;
          if (lane == 0)
            for (int m = 1; m <= pp.n_more && ok; ++m) ok = flag_wait(flag + m * 16, a.status, a.wait_limit);
          ok = __all_sync(0xffffffffu, ok);
          if (!ok) break;
          __syncwarp();                                     // lane 0's acquire holds for every lane's reads
        }
        const int n = (2 * s.wt + (int)rank) * kTileM + row;
        if (a.mode == kGemmQkv) {
          if (n < p.n_out) epilogue_qkv(a, taddr, pp, n, tok0, c0, n_valid, lane);        // warp-uniform: d is a multiple of 64
        } else if (a.mode == kGemmSwiglu) {
          epilogue_swiglu(a, taddr, pp, n, tok0, c0, n_valid, lane);
        } else {
          epilogue_residual(a, taddr, pp, n, tok0, c0, n_valid);
        }
        if (pp.n_more > 0) {
          // read: the flags are zero again for the next projection
          __syncwarp();
          for (int m = 1 + lane; m <= pp.n_more; m += 32) flag[m * 16] = 0u;
        }
      }
      // the buffer may be overwritten once all sixteen epilogue warps of the pair have read it
      tc_fence_before();
      __syncwarp();
      if (lane == 0) {
        if (rank == 0) mbar_arrive(smem_u32(&hdr->acc_empty[buf]));
        else mbar_arrive_leader(smem_u32(&hdr->acc_empty[buf]));
      }
    }
  }

  // neither CTA may give up its shared or tensor memory while the other's MMAs or copies can still touch it
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc_pair(tmem_base, 2u * kPairTokens);
  }
}

}  // namespace ss
