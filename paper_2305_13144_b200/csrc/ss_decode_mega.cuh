// One decode step as ONE persistent cooperative kernel (one CTA per SM).
//
// Why: a decode step at small batch is a chain of ~130 weight-streaming projections separated by
// tiny dependent stages.  As separate kernels every projection pays several microseconds of
// launch, ramp-up and drain during which HBM idles.  Here a dedicated producer warp streams the
// tiled weights of ALL projections of the step, in order, through one shared-memory ring; it
// never waits for activations, so while the other warps sit in a grid barrier or run a small
// stage, the ring keeps filling with the next projection's weights.
//
// Warp roles (352 threads):
//   warp 0      weight producer: linear bulk copies of 32 KiB (256-row tile, k-block) images into the ring
//   warp 1      MMA issuer: tcgen05.mma, accumulators in tensor memory (two buffers)
//   warp 2      activation loader: TMA loads of the [tokens x 64] activation block of each ring stage,
//               issued once the stage that produced the activations has passed its grid barrier
//   warps 3-10  workers: drain accumulators to fp32 partials, then run the stage between two
//               projections (partial sums in CTA order, RoPE, cache append, attention, residual,
//               SwiGLU, arg-max, bookkeeping), separated by grid barriers
//
// Operand roles: one tcgen05.mma costs about the same issue time whatever its shape, so the decode
// projections put the WEIGHTS on the wide side: D[token, row] += X[token, 16] . W[row, 16]^T with
// M = 64 or 128 token lanes and N = 256 weight rows (8 KiB of weights per instruction).  Token lanes
// beyond the batch compute on whatever shared memory follows the activation block; rows of D are
// independent, and those lanes are never read.  Larger batches' projections run on pairs of CTAs
// (tcgen05 cta_group::2, M = 256): the pair shares a range of weight blocks, each CTA holds half of a
// block's rows and its own half of the tokens.
//
// RMSNorm is applied lazily: the residual stage writes x' = bf16(h * g) and per-slice sums of
// squares; since a projection is linear, the consumer of its partial sums multiplies by
// rsqrt(mean h^2 + eps).  This lets a row be split over many CTAs without a cross-CTA reduction.
//
// Every wait (mbarrier, grid barrier, flag) is bounded; on expiry the kernel records a status word,
// raises a CTA-wide abort flag and all roles leave.  The worker warps leave together, behind a grid barrier: they meet in
// barriers of the CTA, which have no limit of their own, so none of them goes by the abort flag alone.
#pragma once

#include "ss_kernels.cuh"

namespace ss {

constexpr int kMegaThreads = 352;
constexpr int kMegaWorkers = 256;          // warps 3..10
constexpr int kMegaMaxStages = 8;          // ring depth bound (shared memory holds 4 at batch 16)
constexpr int kSegTabEntries = 256;        // tile-table entries kept in shared memory (the four per-layer projections)
constexpr int kRowSlice = 128;             // elements of a row handled by one residual work item (one warp, 4 per lane)
constexpr int kMaxSlices = 64;             // d_model <= 8192
constexpr int kKvPieceBytes = 4096;        // one bulk copy of the cache scan: the keys (or values) of one unit
constexpr int kKvMaxPieces = 4;            // pieces in flight per worker warp, at most
constexpr int kPgTab = 512;                // units whose page ids are kept in shared memory

struct MegaGemmShape {
  int n_tiles, kb, max_seg;
  int gsplit;              // CTAs (or pairs) that share the iteration space (the others idle through this projection)
  long long total;
  const TileSeg* tiles;
  float* partial;          // partial sums, [CTA or pair][max_seg][token][256]
  int smem_off;            // first entry of this projection's table in MegaSmem::seg_tab, or -1 (read it from `tiles`)
};

// Range of the (tile, k-block) iteration space owned by a CTA (or a pair).
__device__ __forceinline__ void mega_range(const MegaGemmShape& gs, int cta, long long& it0, long long& it1) {
  if (cta < gs.gsplit) {
    it0 = (long long)cta * gs.total / gs.gsplit;
    it1 = (long long)(cta + 1) * gs.total / gs.gsplit;
  } else {
    it0 = it1 = 0;
  }
}

struct MegaArgs {
  // model
  int n_layers, d, H, Dh, F, V, eos_id;
  float eps;
  const uint8_t* const* wptr;      // [4*L + 1] tiled weights in execution order (qkv, o, gate/up, down)*L, lm head
  const bf16* const* norm_ptr;     // [2*L + 1] gains: attn_norm(l), ffn_norm(l) ..., final
  const bf16* embed;
  const float2* rope;              // [position][Dh / 2] (cos, sin)
  MegaGemmShape shape[5];          // qkv, o, gate/up, down, lm head
  // batch
  int B, NT, stages;
  int x_rows;                      // activation rows per TMA load (the tensor map's box height): the batch, on pairs half of it
  const uint8_t* wbase;            // pairs: what map_w calls line 0
  RowState st;
  KvLayout kv;
  int kv_pieces;                   // shared-memory pieces per worker warp for the cache scan
  float* att_part;                 // [CTA][Dh + 4] (acc, max, sum, two unused) of the pair a CTA's range starts inside of
  unsigned long long* att_flag;    // [CTA] set to the running barrier's number once att_part[CTA] is complete
  // activations (decode buffers)
  float* h;                        // [B][d] residual stream
  bf16 *x, *o, *act;               // GEMM operands: x' [B][d], attention out [B][d], SwiGLU out [B][F]
  float* rowss;                    // [B][kMaxSlices] sums of squares of h per slice
  float* tile_val;
  int32_t* tile_idx;
  int n_tiles_lm;
  // options
  const int32_t* forced;
  int32_t* next_tokens;
  float *dump_logits, *dump_hidden;
  int32_t* dump_choice;
  SampleCfg sample;
  // sync
  unsigned long long* grid_ctr;    // monotone arrival counter
  unsigned long long grid_base;    // its value when this launch starts
  uint32_t* status;
  unsigned long long* trace;       // [2 + 4 * projections] global-timer stamps of CTA 0 (stage boundaries)
  long long wait_limit;            // SM cycles after which any wait inside the kernel gives up
};

__device__ __forceinline__ unsigned long long global_timer_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

struct MegaSmem {
  uint64_t full[kMegaMaxStages];
  uint64_t empty[kMegaMaxStages];
  uint64_t acc_full[2];
  uint64_t acc_empty[2];
  uint64_t mma_done;               // an abandoned step's last MMAs have ended
  uint32_t tmem_base;
  volatile int w_issued;           // ring iterations armed by the weight producer
  volatile int act_epoch;          // projections whose activation operand is complete
  volatile int abort;
  volatile int leave;              // set behind a grid barrier that found the flag up, or that nobody answered: the workers leave
  int prefix[kMaxBatch + 1];
  // attention, set up once per step (the lengths do not change between layers): every warp's slice of the cache scan
  int sl_begin[8], sl_n[8];        // its first unit and its units
  int sl_r[8], sl_hd[8], sl_u0[8]; // its first unit's row, head and place in the pair
  int sl_head[8];                  // pair the slice starts inside of, or -1
  int sl_tail[8];                  // pair that starts in the slice and goes on behind it, or -1
  int att_head;                    // pair the CTA's range starts inside of, or -1
  int att_cut;                     // some pair is cut between warps (or CTAs): there is something to merge
  int att_row0;                    // first row of the CTA's range: pg_tab holds the page of every unit from there on
  int max_units;
  int cost[kMaxBatch + 1];         // as prefix, in work: a row's units and kAttnPairCost
  uint64_t kv_full[8][kKvMaxPieces];
  int ctx_s[kMaxBatch];            // cached tokens of every row
  int pg_tab[kPgTab];
  int4 seg_tab[kSegTabEntries];    // tile tables of the per-layer projections (when they fit)
  uint8_t active_s[kMaxBatch];     // rows active in this step
};
// Scratch behind MegaSmem.  In the attention stage: every warp's rotated query, then two partials per warp.  In a drain:
// the transposition of 16 outputs of a warp's tokens (16 in the kernel of the small batches, else 32; rows padded to 20).
struct AttnScratch {
  float q_s[8][128];
  float slot[8][2][132];           // [warp][0: the pair it starts inside of, 1: the pair that goes on][acc[Dh], max, sum]
};
constexpr int kDrainPad = 20;
__host__ __device__ constexpr int mega_scratch_bytes(bool wide) {
  return wide ? 8 * 32 * kDrainPad * 4 : (int)sizeof(AttnScratch);
}
static_assert(sizeof(AttnScratch) >= 8 * 16 * kDrainPad * 4 && sizeof(AttnScratch) <= mega_scratch_bytes(true), "scratch");
static_assert(sizeof(MegaSmem) % 16 == 0, "the scratch is read as float4");
static_assert(sizeof(MegaSmem) + mega_scratch_bytes(true) + 1024 + 2 * (kBlockBytes + 128 * kTileK * 2) + 2 * 8 * kKvPieceBytes <= 227 * 1024 &&
              sizeof(MegaSmem) + mega_scratch_bytes(true) + 1024 + 4 * (kBlockBytes / 2 + 128 * kTileK * 2) + 2 * 8 * kKvPieceBytes <= 227 * 1024,
              "two ring stages (on pairs four) and two pieces per warp fit beside the wide kernels' scratch");

__device__ __forceinline__ void named_bar_workers() { asm volatile("bar.sync 1, 256;" ::: "memory"); }
__device__ __forceinline__ void fence_proxy_async_global() { asm volatile("fence.proxy.async.global;" ::: "memory"); }
__device__ __forceinline__ unsigned long long ld_acquire_u64(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}

// mbarrier wait that also gives up when the CTA aborts.
__device__ __forceinline__ bool mega_wait(uint32_t bar, uint32_t parity, MegaSmem* sm, uint32_t* status, uint32_t code,
                                          long long limit) {
  if (mbar_try_wait(bar, parity)) return true;
  const long long t0 = clock64();
  for (;;) {
    if (mbar_try_wait(bar, parity)) return true;
    if (sm->abort) return false;
    if (clock64() - t0 > limit) {
      atomicCAS(status, 0u, code);
      sm->abort = 1;
      return false;
    }
    __nanosleep(40);                 // a spinning role must not starve the warps that share its scheduler
  }
}

// Arrival on a grid-wide counter and the bounded poll for `target` arrivals, as one thread of a CTA does them.
// Returns false when the limit ran out before the counter got there, or the CTA's abort flag was up at the last look.
__device__ __forceinline__ bool arrive_and_poll(unsigned long long* ctr, unsigned long long target, long long limit,
                                                const volatile int* abort_flag) {
  // arrive: release-add without waiting for the old value (the writes of the whole CTA, made visible to this
  // thread by the bar.sync in front, are ordered before it); then poll with acquire loads
  asm volatile("red.release.gpu.global.add.u64 [%0], %1;" ::"l"(ctr), "l"(1ULL) : "memory");
  const long long t0 = clock64();
  for (;;) {
    const int aborted = abort_flag ? *abort_flag : 0;     // beside the poll: no latency of its own
    const bool there = ld_acquire_u64(ctr) >= target;
    if (aborted) return false;
    if (there) return true;
    if (clock64() - t0 > limit) return false;
  }
}

// Workers only.  Returns false if the CTA aborted, in all of them or in none: any role may raise the flag at any time, so one
// thread looks at it between the two barriers and the others take what it found.
// `wrote_operand`: this CTA wrote activations that other CTAs read with TMA after the barrier, so its global writes are
// ordered before the async proxy's reads.
// The barrier after a projection publishes only fp32 partials, which are read with ordinary loads: there the
// proxy fence is left out (with bulk copies of the weight ring in flight it took about 2 us per barrier).
__device__ __forceinline__ bool grid_barrier(const MegaArgs& a, MegaSmem* sm, unsigned long long& epoch, int wtid,
                                             bool wrote_operand) {
  if (wrote_operand) fence_proxy_async_global();
  named_bar_workers();
  ++epoch;
  if (wtid == 0) {
    const unsigned long long target = a.grid_base + epoch * gridDim.x;
    if (!arrive_and_poll(a.grid_ctr, target, a.wait_limit, &sm->abort)) {
      if (!sm->abort) atomicCAS(a.status, 0u, (uint32_t)kStatusGridBarrierTimeout);
      sm->abort = sm->leave = 1;
    }
  }
  named_bar_workers();
  return sm->leave == 0;
}

// The stages between projections are chains of dependent L2 round trips (~0.7 us each), not bandwidth: the
// helpers below put independent loads in flight together and keep only true dependencies serial.

// An L2 load that the compiler may not move (a plain __ldcg can sink to its first use, which puts its
// round trip back in series with the loads issued in between).
__device__ __forceinline__ float ldcg_now(const float* p) {
  float v;
  asm volatile("ld.global.cg.f32 %0, [%1];" : "=f"(v) : "l"(p));
  return v;
}

// Partial sums, read past L1.  FLAG: words that one SM writes while another looks at them are read (and written, st_partial)
// with relaxed accesses at gpu scope: a plain load need neither see a store ever nor read a word whole.  Nothing is ordered by
// them and nothing has to be, since only the words themselves are used; so they clobber no memory either (with a clobber and a
// predicate on every load 16 rows of the 7B shape, 32 layers, took 25340 us a call of 8 steps, without 25220, weak accesses 25190).
template <bool FLAG, int N>
__device__ __forceinline__ void ldcg_vec(const float* p, float (&x)[N]) {
  static_assert(N == 2 || N == 4, "N");
  if constexpr (FLAG && N == 2) asm volatile("ld.relaxed.gpu.global.v2.f32 {%0, %1}, [%2];" : "=f"(x[0]), "=f"(x[1]) : "l"(p));
  else if constexpr (FLAG) asm volatile("ld.relaxed.gpu.global.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(x[0]), "=f"(x[1]), "=f"(x[2]), "=f"(x[3]) : "l"(p));
  else if constexpr (N == 2) asm volatile("ld.global.cg.v2.f32 {%0, %1}, [%2];" : "=f"(x[0]), "=f"(x[1]) : "l"(p));
  else asm volatile("ld.global.cg.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(x[0]), "=f"(x[1]), "=f"(x[2]), "=f"(x[3]) : "l"(p));
}

// Into the same registers where `on`.
template <int N>
__device__ __forceinline__ void ld_partial_if(const float* p, bool on, float (&x)[N]) {
  static_assert(N == 2 || N == 4, "N");
  if constexpr (N == 2)
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %3, 0;\n\t@p ld.relaxed.gpu.global.v2.f32 {%0, %1}, [%2];\n\t}"
                 : "+f"(x[0]), "+f"(x[1]) : "l"(p), "r"((int)on));
  else
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %5, 0;\n\t@p ld.relaxed.gpu.global.v4.f32 {%0, %1, %2, %3}, [%4];\n\t}"
                 : "+f"(x[0]), "+f"(x[1]), "+f"(x[2]), "+f"(x[3]) : "l"(p), "r"((int)on));
}

// Where `on`, zeros elsewhere: no branch, so that the loads of a sum stay together, and no traffic.  (With the last
// segment read again in the place of those that a tile has not: 7B shape, 4 layers, 1 / 16 / 256 rows 400 / 462 / 1066 us a
// step, now 396.5 / 458 / 1030; residual stages of 256 rows on pairs, whose tiles have half of the segments, 8.5 -> 5.2 us.)
template <bool FLAG, int N>
__device__ __forceinline__ void ldcg_vec_if(const float* p, bool on, float (&x)[N]) {
  static_assert(N == 2 || N == 4, "N");
#pragma unroll
  for (int i = 0; i < N; ++i) x[i] = 0.f;
  if constexpr (FLAG) ld_partial_if<N>(p, on, x);
  else if constexpr (N == 2)
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %3, 0;\n\t@p ld.global.cg.v2.f32 {%0, %1}, [%2];\n\t}"
                 : "+f"(x[0]), "+f"(x[1]) : "l"(p), "r"((int)on));
  else
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %5, 0;\n\t@p ld.global.cg.v4.f32 {%0, %1, %2, %3}, [%4];\n\t}"
                 : "+f"(x[0]), "+f"(x[1]), "+f"(x[2]), "+f"(x[3]) : "l"(p), "r"((int)on));
}

// ---- partial sums that announce themselves (FLAG: the kernel of up to 16 rows).  Between two uses a slot holds kNoPartial in
// every word, and a drain never writes that pattern, so a consumer reads the words themselves until none of them is it:
// no barrier behind the projection, and a sum waits for its own segments only.  The CTA that wrote a slot clears it behind
// the barrier that follows the consuming stage, long before the slot's next use (every projection of a layer has slots of
// its own).  A store's way to the reader is then one hop; with a barrier it was drained stores -> release fence -> add ->
// poll -> loads.  7B shape, 4 layers, 1 / 8 / 16 rows 395 / 424 / 452 -> 390 / 413 / 446 us a step; 32 x 64 heads, 1 row 211 ->
// 202; the small configuration 75 -> 71.  With more rows the polls take the L2 from the CTAs that still stream: 24 / 32 / 45 /
// 64 rows 483 / 536 / 603 / 616 with a barrier, 487 / 534 / 608 / 650 without.  Fewer polls are no way out: one missing segment
// at a time 399 / 423 / 460 at 1 / 8 / 16 rows, a sleep of 64 or 100 ns between looks 427 / 446 / 490 and more.
constexpr uint32_t kNoPartial = 0xffffffffu;        // a NaN that no instruction produces (results are 0x7fffffff)
__device__ __forceinline__ void st_partial(float* p, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
  asm volatile("st.relaxed.gpu.global.v4.b32 [%0], {%1, %2, %3, %4};" ::"l"(p), "r"(a), "r"(b), "r"(c), "r"(d));
}
template <int N>
__device__ __forceinline__ bool no_partial(const float (&x)[N]) {
  bool m = false;
#pragma unroll
  for (int i = 0; i < N; ++i) m |= __float_as_uint(x[i]) == kNoPartial;
  return m;
}
// One more look is over: false if the wait has lasted too long or the CTA has aborted.
__device__ __forceinline__ bool partial_wait_on(const MegaArgs& a, MegaSmem* sm, long long t0) {
  if (sm->abort) return false;
  if (clock64() - t0 > a.wait_limit) {
    atomicCAS(a.status, 0u, (uint32_t)kStatusFlagTimeout);
    sm->abort = 1;
    return false;
  }
  return true;
}

// Partial sums of the N consecutive outputs n0.. (inside one tile) for token tok, read past L1: the tile's
// first segment, then segment 0 of CTAs c_next..c_last (additions in CTA order, so the sum does not depend
// on timing).  Split in three so that a stage can put the loads of several sums in flight before it waits:
//   tile_seg()       the tile's table entry (one load);
//   partials_issue() the first segment and the next BATCH segments (loads only, without branches);
//   partials_sum()   the additions, and any segments beyond the first batch.
__device__ __forceinline__ int4 tile_seg(const MegaSmem* sm, const MegaGemmShape& s, int n0) {
  const int tile = n0 / kTileN;
  if (s.smem_off >= 0) return sm->seg_tab[s.smem_off + tile];
  return __ldg(reinterpret_cast<const int4*>(s.tiles) + tile);
}
template <int N, int BATCH>
struct PartialLoads {
  float x[N];
  float u[BATCH][N];
};
template <bool FLAG, int N, int BATCH>
__device__ __forceinline__ void partials_issue(const MegaArgs& a, const MegaGemmShape& s, const int4 t, int n0, int tok, PartialLoads<N, BATCH>& q) {
  const size_t slot_stride = (size_t)a.NT * kTileN, cta_stride = slot_stride * s.max_seg;
  const size_t off = (size_t)tok * kTileN + (n0 % kTileN);
  ldcg_vec<FLAG, N>(s.partial + (size_t)t.x * slot_stride + off, q.x);
#pragma unroll
  for (int j = 0; j < BATCH; ++j) ldcg_vec_if<FLAG, N>(s.partial + (size_t)(t.y + j) * cta_stride + off, t.y + j <= t.z, q.u[j]);
}
template <bool FLAG, int N, int BATCH>
__device__ __forceinline__ void partials_sum(const MegaArgs& a, MegaSmem* sm, const MegaGemmShape& s, const int4 t, int n0, int tok,
                                             PartialLoads<N, BATCH>& q, float (&x)[N]) {
  const size_t slot_stride = (size_t)a.NT * kTileN, cta_stride = slot_stride * s.max_seg;
  const size_t off = (size_t)tok * kTileN + (n0 % kTileN);
  if constexpr (FLAG) {
    bool more = no_partial<N>(q.x);
#pragma unroll
    for (int j = 0; j < BATCH; ++j) more |= no_partial<N>(q.u[j]);
    if (more) {
      const long long t0 = clock64();
      do {
        ld_partial_if<N>(s.partial + (size_t)t.x * slot_stride + off, no_partial<N>(q.x), q.x);
#pragma unroll
        for (int j = 0; j < BATCH; ++j) ld_partial_if<N>(s.partial + (size_t)(t.y + j) * cta_stride + off, no_partial<N>(q.u[j]), q.u[j]);
        more = no_partial<N>(q.x);
#pragma unroll
        for (int j = 0; j < BATCH; ++j) more |= no_partial<N>(q.u[j]);
      } while (more && partial_wait_on(a, sm, t0));
    }
  }
#pragma unroll
  for (int i = 0; i < N; ++i) x[i] = q.x[i];
#pragma unroll
  for (int j = 0; j < BATCH; ++j)
#pragma unroll
    for (int i = 0; i < N; ++i) x[i] += q.u[j][i];
  for (int c = t.y + BATCH; c <= t.z; c += BATCH) {
    float u[BATCH][N];
#pragma unroll
    for (int j = 0; j < BATCH; ++j) ldcg_vec_if<FLAG, N>(s.partial + (size_t)(c + j) * cta_stride + off, c + j <= t.z, u[j]);
    if constexpr (FLAG) {
      const long long t0 = clock64();
      for (;;) {
        bool more = false;
#pragma unroll
        for (int j = 0; j < BATCH; ++j) more |= no_partial<N>(u[j]);
        if (!more || !partial_wait_on(a, sm, t0)) break;
#pragma unroll
        for (int j = 0; j < BATCH; ++j) ld_partial_if<N>(s.partial + (size_t)(c + j) * cta_stride + off, no_partial<N>(u[j]), u[j]);
      }
    }
#pragma unroll
    for (int j = 0; j < BATCH; ++j)
#pragma unroll
      for (int i = 0; i < N; ++i) x[i] += u[j][i];
  }
}
// One sum on its own.
template <bool FLAG, int N, int BATCH>
__device__ __forceinline__ void sum_partials_cg(const MegaArgs& a, MegaSmem* sm, const MegaGemmShape& s, int n0, int tok, float (&x)[N]) {
  const int4 t = tile_seg(sm, s, n0);
  PartialLoads<N, BATCH> q;
  partials_issue<FLAG, N, BATCH>(a, s, t, n0, tok, q);
  partials_sum<FLAG, N, BATCH>(a, sm, s, t, n0, tok, q, x);
}
// The slots that this CTA wrote for a projection, empty again.
__device__ __forceinline__ void clear_partials(const MegaArgs& a, const MegaGemmShape& gs, int part, int wtid) {
  long long it0, it1;
  mega_range(gs, part, it0, it1);
  if (it0 == it1) return;
  const int n = ((int)((it1 - 1) / gs.kb) - (int)(it0 / gs.kb) + 1) * a.NT * kTileN;
  float* p = gs.partial + (size_t)part * gs.max_seg * a.NT * kTileN;
  for (int i = wtid * 4; i < n; i += 4 * kMegaWorkers)
    *reinterpret_cast<uint4*>(p + i) = make_uint4(kNoPartial, kNoPartial, kNoPartial, kNoPartial);
}

// 1/rms of row r; warp-collective (every lane returns it).  Lane i reads slices i, i+32; issue and finish are apart so
// that a stage can put its own loads in between.
__device__ __forceinline__ float row_ss_issue(const MegaArgs& a, int r, int lane) {
  const int ns = (a.d + kRowSlice - 1) / kRowSlice;        // <= 64
  const float* p = a.rowss + (size_t)r * kMaxSlices;
  const float v0 = lane < ns ? ldcg_now(p + lane) : 0.f;
  const float v1 = lane + 32 < ns ? ldcg_now(p + lane + 32) : 0.f;
  return v0 + v1;
}
__device__ __forceinline__ float row_ss_inv_rms(const MegaArgs& a, float ss) { return rsqrtf(warp_sum(ss) / a.d + a.eps); }
__device__ __forceinline__ float warp_row_inv_rms(const MegaArgs& a, int r, int lane) { return row_ss_inv_rms(a, row_ss_issue(a, r, lane)); }

// ---- stage: embedding (or residual add) + lazy RMSNorm operand -------------------------------------
// Work unit = (row, slice of 128 columns) per warp, 4 columns per lane; units are dealt round-robin over
// the CTAs first, so the whole stage is one pass with a few warps busy in every CTA.
// mode 0: h = E[cur_tok]; mode 1: h += projection (partials of shape `gs`).  BATCH: segments of a sum asked for together.
// (Two or three units in flight per warp at 256 rows: 3 to 7 % slower, the registers for it spill or crowd the stages.)
template <bool FLAG, int BATCH>
__device__ void stage_residual(const MegaArgs& a, MegaSmem* sm, int wtid, int mode, const MegaGemmShape* gs,
                               const bf16* __restrict__ gain, bool dump) {
  const int ns = (a.d + kRowSlice - 1) / kRowSlice;
  const int n_units = a.B * ns;
  const int lane = wtid & 31, wid = wtid >> 5;
  for (int u = wid * gridDim.x + blockIdx.x; u < n_units; u += 8 * gridDim.x) {
    const int r = u / ns, sl = u - r * ns;
    if (!sm->active_s[r]) continue;
    const int c = sl * kRowSlice + lane * 4;
    float ss = 0.f;
    if (c < a.d) {
      float v[4];
      if (mode == 0) {
        int tok = a.st.cur_tok[r];
        if (tok < 0 || tok >= a.V) tok = 0;
        const uint2 e = __ldg(reinterpret_cast<const uint2*>(a.embed + (size_t)tok * a.d + c));
        const float2 e0 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&e.x));
        const float2 e1 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&e.y));
        v[0] = e0.x; v[1] = e0.y; v[2] = e1.x; v[3] = e1.y;
      } else {
        const float4 h4 = __ldcg(reinterpret_cast<const float4*>(a.h + (size_t)r * a.d + c));
        sum_partials_cg<FLAG, 4, BATCH>(a, sm, *gs, c, r, v);
        v[0] += h4.x; v[1] += h4.y; v[2] += h4.z; v[3] += h4.w;
      }
      const uint2 gb = __ldg(reinterpret_cast<const uint2*>(gain + c));
      const float2 g0 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&gb.x));
      const float2 g1 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&gb.y));
      *reinterpret_cast<float4*>(a.h + (size_t)r * a.d + c) = make_float4(v[0], v[1], v[2], v[3]);
      if (dump && a.dump_hidden) {                     // the caller's buffer: no alignment beyond a float's
        float* o = a.dump_hidden + (size_t)r * a.d + c;
        o[0] = v[0]; o[1] = v[1]; o[2] = v[2]; o[3] = v[3];
      }
      __align__(8) bf16 xb[4];
      xb[0] = __float2bfloat16_rn(v[0] * g0.x); xb[1] = __float2bfloat16_rn(v[1] * g0.y);
      xb[2] = __float2bfloat16_rn(v[2] * g1.x); xb[3] = __float2bfloat16_rn(v[3] * g1.y);
      *reinterpret_cast<uint2*>(a.x + (size_t)r * a.d + c) = *reinterpret_cast<const uint2*>(xb);
      ss = v[0] * v[0] + v[1] * v[1] + v[2] * v[2] + v[3] * v[3];
    }
    ss = warp_sum(ss);
    if (lane == 0) a.rowss[(size_t)r * kMaxSlices + sl] = ss;
  }
}

// ---- stage: q,k,v from partials + RoPE + cache append + paged attention ----------------------------------
// Work is counted in units of (row, head, 8 KiB of cache): 16 cached tokens at head size 128, 32 at 64; their keys and
// their values are contiguous 4 KiB each.  All units of the step, in (row, head, token) order, are cut into one
// contiguous range per CTA and that into one slice per worker warp, once per step.
//
// A warp streams its slice through its own few pieces of shared memory with bulk copies (keys and values of a unit are
// one piece each): a piece is asked for as soon as the one before it in the same place has been read, across pairs and
// -- the cache does not depend on this step's projections -- across layers, so a warp has its next pieces in flight
// while it computes, sits in a barrier or builds a query.  Before, a warp held one unit's loads in registers and worked
// on them before it asked for the next: the scan moved 4.2 to 4.7 TB/s (24 rows of 1700 cached tokens, 13B shape).
//
// A warp builds the query of every pair its slice touches (the warp with the pair's first unit also appends the new
// token's key and value and starts from its score), so warps do not wait for one another; only pairs that are cut
// between warps are merged at the end, through shared memory.  Ranges end between pairs unless some row is long
// (kAttnCutUnits): then a pair may be cut between CTAs too, and the CTA that has its start collects the others'
// partials from global memory, each announced by a flag.
//
// Scan layout: keys -- lane (g, gl) takes key g of a load step and a quarter (half at Dh 64) of its chunks, ordered so
// that the eight lanes of a shared-memory phase hit different banks; values -- a lane owns four dimensions of every key
// (every second key at Dh 64), so the running sum is four registers and needs no exchange at the end.
// Units of the longest row from which pairs are cut between CTAs: a cut costs a flag and a merge behind the scan (about 2.5 us),
// a pair that is not cut leaves its CTA up to its whole length over the others.  7B shape, 8 layers, cut from 8 / 20 / 40
// units on: 16 rows of 100-380 tokens 852 / 851 / 844 us a step, 4 rows of 300-600 792 / 792 / 775, one row of 173 tokens
// 779 / 731 / 731, one of 1500 822 / 822 / 821.
constexpr int kAttnCutUnits = 40;
constexpr int kAttnPairCost = 2;           // what a pair costs beside its units, in units (0 / 2 / 4: 200 rows 2502 / 2419 / 2431 us a step)

template <int DH> struct AttnLayout {
  static constexpr int GROUP = DH / 32;           // lanes per key
  static constexpr int KPW = 32 / GROUP;          // keys per warp-wide load step
  static constexpr int UT = 2 * KPW;              // cached tokens per unit
  static constexpr int UPP = kPageTokens / UT;    // units per page (2 at Dh 128, 1 at Dh 64)
  static constexpr int VK = 128 / DH;             // keys per value step (16 steps per unit)
  static constexpr int EPL = DH / 32;             // cooperative layout: consecutive dimensions per lane
};

// Packed pairs of fp32: two fused multiply-adds per instruction.
__device__ __forceinline__ uint64_t pack_f32x2(float lo, float hi) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ void unpack_f32x2(uint64_t v, float& lo, float& hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ uint64_t fma_f32x2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ uint64_t mul_f32x2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
// Two bf16 in a word -> two fp32 (element 0 in the low half).
__device__ __forceinline__ uint64_t bf16x2_to_f32x2(uint32_t u) {
  return pack_f32x2(__uint_as_float(u << 16), __uint_as_float(u & 0xffff0000u));
}

__device__ __forceinline__ uint4 lds128(uint32_t addr) {
  uint4 v;
  asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ uint2 lds64(uint32_t addr) {
  uint2 v;
  asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(addr) : "memory");
  return v;
}

// A warp's stream of cache pieces: where the next copy comes from, and the place of the next piece to be read.  The
// pieces of a pair of t units follow in the order K0, K1, V0, K2, V1, .., V(t-1), the order in which they are read.
// Lane i holds source and size of piece i of the current 32 and issues it: the search for a piece's pair, page and
// position is done for 32 pieces at a time (and once per step where a slice has no more).
struct KvStream {
  uint32_t base;           // shared-memory address of the warp's pieces
  uint64_t hint;
  const bf16* src;         // this lane's piece: its place in layer 0, its bytes
  uint32_t bytes;
  int next, total, layer;  // piece of the slice to ask for next, pieces of the slice, layer
  int in_slot, out_slot;   // place of the next copy / of the next piece to be read
  uint32_t out_phase;
  int flight;              // copies not read yet
};

// This lane's piece of the 32 from `first` on.
template <int DH>
__device__ __forceinline__ void kv_stream_locate(const MegaArgs& a, MegaSmem* sm, KvStream& k, int first, int wid, int lane) {
  using L = AttnLayout<DH>;
  const int i = first + lane;
  k.src = a.kv.pool;
  k.bytes = 0;
  if (i >= k.total) return;
  const int H = a.H, s0 = sm->sl_begin[wid], n = sm->sl_n[wid];
  // row of the unit s0 + i / 2, by bisection of the rows' first units
  const int x = s0 + (i >> 1);
  int r = 0;
#pragma unroll
  for (int step = kMaxBatch / 2; step > 0; step >>= 1)
    if (sm->prefix[r + step] * H <= x) r += step;
  // (rows without units share their successor's first unit: the last of them is the row that has it)
  const int row0 = sm->prefix[r] * H, npr = sm->prefix[r + 1] - sm->prefix[r];
  const int hd = (x - row0) / npr;
  const int p0 = row0 + hd * npr;                         // the pair's first unit
  const int f = max(p0, s0), t = min(p0 + npr, s0 + n) - f, j = i - 2 * (f - s0);
  const int part = j == 0 ? 0 : (j == 2 * t - 1 ? 1 : (j & 1) ^ 1);
  const int u = j == 0 ? 0 : (j == 2 * t - 1 ? t - 1 : (j & 1) ? (j + 1) >> 1 : (j >> 1) - 1);
  const int ui = f - p0 + u;                              // unit of the pair
  const int at = sm->prefix[r] - sm->prefix[sm->att_row0] + ui;
  int pg;
  if (at < kPgTab) {
    pg = sm->pg_tab[at];
  } else {
    pg = a.st.block_table[(size_t)r * a.st.max_pages + ui / L::UPP];
    if (pg < 0 || pg >= a.kv.n_pages) { atomicCAS(a.status, 0u, (uint32_t)kStatusBadPage); pg = 0; }
  }
  const int tok = ui * L::UT;
  k.src = a.kv.pool + (size_t)pg * a.kv.page_elems + ((size_t)(part * H + hd) * kPageTokens + tok % kPageTokens) * DH;
  k.bytes = (uint32_t)min(L::UT, sm->ctx_s[r] - tok) * (DH * 2);          // cached tokens only
}

// Asks for the next piece; nothing after the last layer's slice.
template <int DH>
__device__ __forceinline__ void kv_stream_next(const MegaArgs& a, MegaSmem* sm, KvStream& k, int wid, int lane) {
  if (k.layer >= a.n_layers || k.total == 0) return;
  if (lane == (k.next & 31)) {
    const uint32_t bar = smem_u32(&sm->kv_full[wid][k.in_slot]);
    mbar_expect_tx(bar, k.bytes);
    bulk_load(k.base + (uint32_t)k.in_slot * kKvPieceBytes, k.src + (size_t)k.layer * a.kv.layer_stride, k.bytes, bar, k.hint);
  }
  ++k.flight;
  if (++k.in_slot == a.kv_pieces) k.in_slot = 0;
  if (++k.next == k.total) { k.next = 0; ++k.layer; }
  if ((k.next & 31) == 0 && k.total > 32) kv_stream_locate<DH>(a, sm, k, k.next, wid, lane);
}

template <int DH>
__device__ __forceinline__ void kv_stream_start(const MegaArgs& a, MegaSmem* sm, KvStream& k, uint32_t kv0, int wid, int lane) {
  k.base = kv0 + (uint32_t)(wid * a.kv_pieces) * kKvPieceBytes;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(k.hint));
  k.layer = k.next = k.in_slot = k.out_slot = k.flight = 0;
  k.out_phase = 0;
  k.total = 2 * sm->sl_n[wid];
  kv_stream_locate<DH>(a, sm, k, 0, wid, lane);
  for (int i = 0; i < a.kv_pieces; ++i) kv_stream_next<DH>(a, sm, k, wid, lane);
}

// Waits for the next piece; returns false (in every lane) if the CTA aborted.
__device__ __forceinline__ bool kv_stream_wait(const MegaArgs& a, MegaSmem* sm, const KvStream& k, int wid) {
  const bool ok = mega_wait(smem_u32(&sm->kv_full[wid][k.out_slot]), k.out_phase, sm, a.status, kStatusProducerTimeout, a.wait_limit);
  return __all_sync(0xffffffffu, ok);
}
// The piece has been read by every lane: its place is free and the next copy may go there.
template <int DH>
__device__ __forceinline__ void kv_stream_done(const MegaArgs& a, MegaSmem* sm, KvStream& k, int wid, int lane) {
  --k.flight;
  kv_stream_next<DH>(a, sm, k, wid, lane);
}
__device__ __forceinline__ uint32_t kv_stream_advance(const MegaArgs& a, KvStream& k) {
  const uint32_t at = k.base + (uint32_t)k.out_slot * kKvPieceBytes;
  if (++k.out_slot == a.kv_pieces) { k.out_slot = 0; k.out_phase ^= 1u; }
  return at;
}
// An abandoned step leaves copies in flight: they get a bounded time to land before the shared memory is given up.
__device__ __forceinline__ void kv_stream_end(const MegaArgs& a, MegaSmem* sm, KvStream& k, int wid, int lane) {
  for (; k.flight > 0; --k.flight) {
    const long long t0 = clock64();
    while (!mbar_try_wait(smem_u32(&sm->kv_full[wid][k.out_slot]), k.out_phase) && clock64() - t0 < 2000000LL) __nanosleep(100);
    if (++k.out_slot == a.kv_pieces) { k.out_slot = 0; k.out_phase ^= 1u; }
  }
}

// Row, head and unit of the pair at position x of the step's units (x below their number); warp-collective.
__device__ __forceinline__ void locate_unit(const MegaSmem* sm, int H, int x, int lane, int& r, int& hd, int& ui) {
  int n = 0;
#pragma unroll
  for (int j = 0; j < kMaxBatch / 32; ++j) n += sm->prefix[lane * (kMaxBatch / 32) + j + 1] * H <= x ? 1 : 0;
  r = __reduce_add_sync(0xffffffffu, n);                  // rows that end before x
  const int off = x - sm->prefix[r] * H, npr = sm->prefix[r + 1] - sm->prefix[r];
  hd = off / npr;
  ui = off - hd * npr;
}

// The step's work, a pair counting as its units and kAttnPairCost more, has positions of its own: row r begins at
// cost[r] * H.  locate_work gives the pair at position x (below the total), the position inside it and its units.
__device__ __forceinline__ void locate_work(const MegaSmem* sm, int H, int x, int lane, int& r, int& hd, int& in, int& npr) {
  int n = 0;
#pragma unroll
  for (int j = 0; j < kMaxBatch / 32; ++j) n += sm->cost[lane * (kMaxBatch / 32) + j + 1] * H <= x ? 1 : 0;
  r = __reduce_add_sync(0xffffffffu, n);
  npr = sm->prefix[r + 1] - sm->prefix[r];
  const int off = x - sm->cost[r] * H;
  hd = off / (npr + kAttnPairCost);
  in = off - hd * (npr + kAttnPairCost);
}
// Where CTA c's range begins, as a position of work: between pairs unless the step has long rows.
__device__ __forceinline__ int range_begin(const MegaSmem* sm, int H, int c, int n_cta, int lane) {
  const int total = sm->cost[kMaxBatch] * H;
  const int x = (int)((long long)c * total / n_cta);
  if (x >= total || sm->max_units >= kAttnCutUnits) return x;
  int r, hd, in, npr;
  locate_work(sm, H, x, lane, r, hd, in, npr);
  return in ? x + npr + kAttnPairCost - in : x;
}
// The unit at a position of work (a pair's first unit for all of its extra cost).
__device__ __forceinline__ int unit_at(const MegaSmem* sm, int H, int x, int lane) {
  if (x >= sm->cost[kMaxBatch] * H) return sm->prefix[kMaxBatch] * H;
  int r, hd, in, npr;
  locate_work(sm, H, x, lane, r, hd, in, npr);
  return sm->prefix[r] * H + hd * npr + max(0, in - kAttnPairCost);
}

// Once per step (the lengths do not change between layers): units per row, every warp's slice, page ids.
template <int DH>
__device__ void attention_setup(const MegaArgs& a, MegaSmem* sm, int wtid) {
  using L = AttnLayout<DH>;
  const int lane = wtid & 31, wid = wtid >> 5;
  const int H = a.H, B = a.B;
  // ---- per-step copies in shared memory: row state, and the per-layer tile tables
  for (int r = wtid; r < kMaxBatch; r += kMegaWorkers) {
    sm->active_s[r] = (r < B && a.st.active[r]) ? 1 : 0;
    sm->ctx_s[r] = r < B ? a.st.ctx_len[r] : 0;
  }
  for (int t = 0; t < 4; ++t) {
    const MegaGemmShape& gs = a.shape[t];
    if (gs.smem_off < 0) continue;
    for (int i = wtid; i < gs.n_tiles; i += kMegaWorkers)
      sm->seg_tab[gs.smem_off + i] = __ldg(reinterpret_cast<const int4*>(gs.tiles) + i);
  }
  // ---- units per row (exclusive prefix, active rows only)
  if (wid == 0) {
    int cnt[8], loc = 0, most = 0;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int r = lane * 8 + j;
      int c = 0;
      if (r < B && a.st.active[r]) c = (a.st.ctx_len[r] + L::UT - 1) / L::UT;
      cnt[j] = c;
      loc += c;
      most = max(most, c);
    }
    int inc = loc;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int t = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += t;
    }
    most = __reduce_max_sync(0xffffffffu, most);
    int here = 0;                                         // active rows among this lane's eight, and before them
#pragma unroll
    for (int j = 0; j < 8; ++j) here += cnt[j] > 0 ? 1 : 0;
    int rows = here;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int t = __shfl_up_sync(0xffffffffu, rows, o);
      if (lane >= o) rows += t;
    }
    int run = inc - loc, n_rows = rows - here;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      sm->prefix[lane * 8 + j] = run;
      sm->cost[lane * 8 + j] = run + n_rows * kAttnPairCost;
      run += cnt[j];
      n_rows += cnt[j] > 0 ? 1 : 0;
    }
    if (lane == 31) {
      sm->prefix[kMaxBatch] = run;
      sm->cost[kMaxBatch] = run + n_rows * kAttnPairCost;
    }
    if (lane == 0) { sm->att_cut = 0; sm->max_units = most; }
  }
  named_bar_workers();
  // ---- this CTA's range, and the slice of every warp
  const int w_lo = range_begin(sm, H, blockIdx.x, gridDim.x, lane), w_hi = range_begin(sm, H, blockIdx.x + 1, gridDim.x, lane);
  const int lo = unit_at(sm, H, w_lo, lane), hi = unit_at(sm, H, w_hi, lane);
  const int s0 = unit_at(sm, H, w_lo + (int)((long long)(w_hi - w_lo) * wid / 8), lane);
  const int s1 = unit_at(sm, H, w_lo + (int)((long long)(w_hi - w_lo) * (wid + 1) / 8), lane);
  int r0 = 0, r1 = 0, cta_head = -1;                      // rows the CTA's range touches; pair it starts inside of
  if (hi > lo) {
    int hd, ui;
    locate_unit(sm, H, hi - 1, lane, r1, hd, ui);
    locate_unit(sm, H, lo, lane, r0, hd, ui);
    if (ui > 0) cta_head = r0 * H + hd;
  }
  {
    int r = 0, hd = 0, ui = 0, head = -1, tail = -1;
    if (s1 > s0) {
      int re, hde, uie;
      locate_unit(sm, H, s1 - 1, lane, re, hde, uie);
      if (uie + 1 < sm->prefix[re + 1] - sm->prefix[re] && s1 - 1 - uie >= s0) tail = re * H + hde;
      locate_unit(sm, H, s0, lane, r, hd, ui);
      if (ui > 0) head = r * H + hd;
    }
    if (lane == 0) {
      sm->sl_r[wid] = r; sm->sl_hd[wid] = hd; sm->sl_u0[wid] = ui; sm->sl_n[wid] = s1 - s0;
      sm->sl_begin[wid] = s0; sm->sl_head[wid] = head; sm->sl_tail[wid] = tail;
      if (head >= 0 || tail >= 0) sm->att_cut = 1;
      if (wid == 0) { sm->att_row0 = r0; sm->att_head = cta_head; }
    }
  }
  // ---- page of every unit of these rows, as far as the table goes
  const int first = sm->prefix[r0], n_tab = hi > lo ? min(kPgTab, sm->prefix[r1 + 1] - first) : 0;
  for (int r = r0; r <= r1; ++r) {
    const int at = sm->prefix[r] - first, npr = sm->prefix[r + 1] - sm->prefix[r];
    for (int u = wtid; u < npr && at + u < n_tab; u += kMegaWorkers) {
      int pg = a.st.block_table[(size_t)r * a.st.max_pages + u / L::UPP];
      if (pg < 0 || pg >= a.kv.n_pages) { atomicCAS(a.status, 0u, (uint32_t)kStatusBadPage); pg = 0; }
      sm->pg_tab[at + u] = pg;
    }
  }
  named_bar_workers();
}

// One running partial of a pair in the value layout: lane's four dimensions, the maximum and the sum of the weights.
struct AttnPartial {
  float acc[4], m, l;
};
__device__ __forceinline__ void attn_merge(AttnPartial& p, const float4 acc, float m, float l) {
  const float mn = fmaxf(p.m, m);
  const float w0 = exp2f(p.m - mn), w1 = exp2f(m - mn);
  p.acc[0] = p.acc[0] * w0 + acc.x * w1;
  p.acc[1] = p.acc[1] * w0 + acc.y * w1;
  p.acc[2] = p.acc[2] * w0 + acc.z * w1;
  p.acc[3] = p.acc[3] * w0 + acc.w * w1;
  p.l = p.l * w0 + l * w1;
  p.m = mn;
}
// The pair's bf16 output (lanes of the first VK-th part hold the DH dimensions).
template <int DH>
__device__ __forceinline__ void attn_store(const MegaArgs& a, const AttnPartial& p, int r, int hd, int lane) {
  if (lane * 4 >= DH) return;
  const float il = 1.f / p.l;
  __align__(8) bf16 ob[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) ob[j] = __float2bfloat16_rn(p.acc[j] * il);
  *reinterpret_cast<uint2*>(a.o + (size_t)r * a.d + hd * DH + lane * 4) = *reinterpret_cast<const uint2*>(ob);
}

template <int DH, bool FLAG>
__device__ void stage_attention(const MegaArgs& a, MegaSmem* sm, AttnScratch* sc, KvStream& kvs, int wtid, int layer,
                                unsigned long long ticket) {
  using L = AttnLayout<DH>;
  constexpr int GROUP = L::GROUP, KPW = L::KPW, UT = L::UT, VK = L::VK, EPL = L::EPL;
  const int lane = wtid & 31, wid = wtid >> 5;
  const int gl = lane % GROUP, g = lane / GROUP;
  const int sw = g & (4 / GROUP * 2 - 1) & 3;             // bank swizzle of the key chunks: g & 1 at Dh 128, g & 3 at Dh 64
  const int dl = (lane * 4) % DH, vk = lane * 4 / DH;     // value layout: first of the lane's dimensions, key of a step
  const int H = a.H, d = a.d;
  const MegaGemmShape& gs = a.shape[0];
  const float qscale = rsqrtf((float)DH) * 1.4426950408889634f;
  const size_t v_off = (size_t)H * kPageTokens * DH;

  int r = sm->sl_r[wid], hd = sm->sl_hd[wid], ui = sm->sl_u0[wid], left = sm->sl_n[wid];
  bool aborted = false;                                   // a wait ran out: this warp only keeps the barriers from here on
  while (left > 0 && !aborted) {
    const int npr = sm->prefix[r + 1] - sm->prefix[r], pos = sm->ctx_s[r];
    const int take = min(npr - ui, left);
    const bool own = ui == 0;                             // this warp has the pair's first unit: the new token is its
    const bool whole = own && take == npr;
    AttnPartial p;
    uint64_t q2[16];
    // ---- the rotated, scaled query; the new token's key and value
    {
      const int e0 = lane * EPL, nq = hd * DH + e0, nk = d + nq, nv = 2 * d + nq;
      const int4 tq = tile_seg(sm, gs, nq), tk = tile_seg(sm, gs, nk), tv = tile_seg(sm, gs, nv);
      PartialLoads<EPL, 4> lq, lk, lv;
      partials_issue<FLAG, EPL, 4>(a, gs, tq, nq, r, lq);
      partials_issue<FLAG, EPL, 4>(a, gs, tk, nk, r, lk);
      partials_issue<FLAG, EPL, 4>(a, gs, tv, nv, r, lv);
      // the two dimensions of a rotation are neighbours (in the weights, so here and in the cache)
      const float2* rp = a.rope + (size_t)pos * (DH / 2) + lane * (EPL / 2);
      float2 cs[EPL / 2];
#pragma unroll
      for (int j = 0; j < EPL / 2; ++j) cs[j] = __ldg(rp + j);
      int pg = own ? a.st.block_table[(size_t)r * a.st.max_pages + pos / kPageTokens] : 0;
      const float inv = warp_row_inv_rms(a, r, lane);
      float qx[EPL], kx[EPL], vx[EPL];
      partials_sum<FLAG, EPL, 4>(a, sm, gs, tq, nq, r, lq, qx);
      partials_sum<FLAG, EPL, 4>(a, sm, gs, tk, nk, r, lk, kx);
      partials_sum<FLAG, EPL, 4>(a, sm, gs, tv, nv, r, lv, vx);
      if (pg < 0 || pg >= a.kv.n_pages) { atomicCAS(a.status, 0u, (uint32_t)kStatusBadPage); pg = -1; }
      __align__(8) bf16 kb[EPL], vb[EPL];
      float qf[EPL], dot = 0.f;
#pragma unroll
      for (int j = 0; j < EPL; j += 2) {
        const float2 c = cs[j / 2];
        const float q0 = qx[j] * inv, q1 = qx[j + 1] * inv, k0 = kx[j] * inv, k1 = kx[j + 1] * inv;
        qf[j] = (q0 * c.x - q1 * c.y) * qscale;           // the query is only ever an ALU operand: it stays fp32
        qf[j + 1] = (q1 * c.x + q0 * c.y) * qscale;
        kb[j] = __float2bfloat16_rn(k0 * c.x - k1 * c.y);
        kb[j + 1] = __float2bfloat16_rn(k1 * c.x + k0 * c.y);
        vb[j] = __float2bfloat16_rn(vx[j] * inv);
        vb[j + 1] = __float2bfloat16_rn(vx[j + 1] * inv);
        dot += qf[j] * __bfloat162float(kb[j]) + qf[j + 1] * __bfloat162float(kb[j + 1]);
      }
      float* qs = sc->q_s[wid];
      __syncwarp();                                       // the warp has read the query before this one
      if constexpr (EPL == 4) *reinterpret_cast<float4*>(qs + e0) = make_float4(qf[0], qf[1], qf[2], qf[3]);
      else *reinterpret_cast<float2*>(qs + e0) = make_float2(qf[0], qf[1]);
      dot = warp_sum(dot);
      if (own) {
        if (pg >= 0) {
          bf16* kdst = a.kv.pool + (size_t)layer * a.kv.layer_stride + (size_t)pg * a.kv.page_elems +
                       ((size_t)hd * kPageTokens + (pos % kPageTokens)) * DH + e0;
          if constexpr (EPL == 4) {
            *reinterpret_cast<uint2*>(kdst) = *reinterpret_cast<const uint2*>(kb);
            *reinterpret_cast<uint2*>(kdst + v_off) = *reinterpret_cast<const uint2*>(vb);
          } else {
            *reinterpret_cast<uint32_t*>(kdst) = *reinterpret_cast<const uint32_t*>(kb);
            *reinterpret_cast<uint32_t*>(kdst + v_off) = *reinterpret_cast<const uint32_t*>(vb);
          }
        }
        p.m = dot;
        p.l = g == 0 ? 1.f : 0.f;                         // summed over the key slots at the end
        if constexpr (EPL == 4) {
#pragma unroll
          for (int j = 0; j < 4; ++j) p.acc[j] = __bfloat162float(vb[j]);
        } else {
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const float t = __shfl_sync(0xffffffffu, __bfloat162float(vb[j & 1]), (dl + j) >> 1);
            p.acc[j] = vk == 0 ? t : 0.f;
          }
        }
      } else {
        p.m = -CUDART_INF_F;
        p.l = 0.f;
#pragma unroll
        for (int j = 0; j < 4; ++j) p.acc[j] = 0.f;
      }
      __syncwarp();
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const float4* qc = reinterpret_cast<const float4*>(qs + ((c ^ sw) * GROUP + gl) * 8);
        const float4 q0 = qc[0], q1 = qc[1];
        q2[c * 4 + 0] = pack_f32x2(q0.x, q0.y); q2[c * 4 + 1] = pack_f32x2(q0.z, q0.w);
        q2[c * 4 + 2] = pack_f32x2(q1.x, q1.y); q2[c * 4 + 3] = pack_f32x2(q1.z, q1.w);
      }
    }
    uint64_t acc0 = pack_f32x2(p.acc[0], p.acc[1]), acc1 = pack_f32x2(p.acc[2], p.acc[3]);
    // ---- the units of this pair in the slice: the values of one are summed beside the scores of the next
    float s_[2];
    uint4 kk[2][4];
    uint2 vv[16];
    auto load_keys = [&]() {
      const uint32_t at = kv_stream_advance(a, kvs);
#pragma unroll
      for (int uu = 0; uu < 2; ++uu)
#pragma unroll
        for (int c = 0; c < 4; ++c) kk[uu][c] = lds128(at + (uint32_t)((uu * KPW + g) * DH * 2 + ((c ^ sw) * GROUP + gl) * 16));
    };
    auto load_values = [&]() {
      const uint32_t at = kv_stream_advance(a, kvs) + (uint32_t)lane * 8;
#pragma unroll
      for (int s = 0; s < 16; ++s) vv[s] = lds64(at + (uint32_t)s * 256);
    };
    auto scores = [&](int cnt) {                          // of the unit in kk; -inf behind its last token
#pragma unroll
      for (int uu = 0; uu < 2; ++uu) {
        uint64_t d0 = 0, d1 = 0;
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          d0 = fma_f32x2(bf16x2_to_f32x2(kk[uu][c].x), q2[c * 4 + 0], d0);
          d1 = fma_f32x2(bf16x2_to_f32x2(kk[uu][c].y), q2[c * 4 + 1], d1);
          d0 = fma_f32x2(bf16x2_to_f32x2(kk[uu][c].z), q2[c * 4 + 2], d0);
          d1 = fma_f32x2(bf16x2_to_f32x2(kk[uu][c].w), q2[c * 4 + 3], d1);
        }
        float x0, x1, x2, x3;
        unpack_f32x2(d0, x0, x1);
        unpack_f32x2(d1, x2, x3);
        float dot = (x0 + x1) + (x2 + x3);
#pragma unroll
        for (int o = GROUP / 2; o > 0; o >>= 1) dot += __shfl_xor_sync(0xffffffffu, dot, o);
        s_[uu] = uu * KPW + g < cnt ? dot : -CUDART_INF_F;
      }
    };
    float p0, p1;
    auto weights = [&]() {                                // of the unit whose scores are in s_
      float mn = fmaxf(s_[0], s_[1]);
#pragma unroll
      for (int o = GROUP; o < 32; o <<= 1) mn = fmaxf(mn, __shfl_xor_sync(0xffffffffu, mn, o));
      if (mn > p.m) {                                     // warp-uniform
        const float w = exp2f(p.m - mn);
        const uint64_t w2 = pack_f32x2(w, w);
        p.l *= w;
        acc0 = mul_f32x2(acc0, w2);
        acc1 = mul_f32x2(acc1, w2);
        p.m = mn;
      }
      const float mr = p.m == -CUDART_INF_F ? 0.f : p.m;  // no score above -inf so far: weights of 0, not NaN
      p0 = exp2f(s_[0] - mr);
      p1 = exp2f(s_[1] - mr);
      p.l += p0 + p1;
    };
    auto add_value = [&](int s) {
      const float pw = __shfl_sync(0xffffffffu, s < 8 ? p0 : p1, ((s * VK + vk) % KPW) * GROUP);
      const uint64_t w2 = pack_f32x2(pw, pw);
      acc0 = fma_f32x2(bf16x2_to_f32x2(vv[s].x), w2, acc0);
      acc1 = fma_f32x2(bf16x2_to_f32x2(vv[s].y), w2, acc1);
    };
    if (!kv_stream_wait(a, sm, kvs, wid)) { aborted = true; break; }
    load_keys();
    __syncwarp();
    kv_stream_done<DH>(a, sm, kvs, wid, lane);
    scores(pos - ui * UT);
    for (int k = 1; k < take; ++k) {
      ++ui;
      weights();
      if (!kv_stream_wait(a, sm, kvs, wid)) { aborted = true; break; }
      load_keys();
      if (!kv_stream_wait(a, sm, kvs, wid)) { aborted = true; break; }
      load_values();
      __syncwarp();
      kv_stream_done<DH>(a, sm, kvs, wid, lane);
      kv_stream_done<DH>(a, sm, kvs, wid, lane);
#pragma unroll
      for (int s = 0; s < 16; ++s) add_value(s);          // every unit but a pair's last is full
      scores(pos - ui * UT);
    }
    if (aborted) break;
    {
      const int cnt = min(UT, pos - ui * UT);
      weights();
      if (!kv_stream_wait(a, sm, kvs, wid)) { aborted = true; break; }
      load_values();
      __syncwarp();
      kv_stream_done<DH>(a, sm, kvs, wid, lane);
#pragma unroll
      for (int s = 0; s < 16; ++s) {
        if (s * VK < cnt) {                               // warp-uniform; what lies behind the last token is not a number to use
          if (VK == 2 && s * VK + vk >= cnt) vv[s] = make_uint2(0, 0);
          add_value(s);
        }
      }
      ++ui;
    }
    left -= take;
    // ---- the slice's partial of the pair
#pragma unroll
    for (int o = GROUP; o < 32; o <<= 1) p.l += __shfl_xor_sync(0xffffffffu, p.l, o);
    unpack_f32x2(acc0, p.acc[0], p.acc[1]);
    unpack_f32x2(acc1, p.acc[2], p.acc[3]);
    if constexpr (VK == 2) {
#pragma unroll
      for (int j = 0; j < 4; ++j) p.acc[j] += __shfl_xor_sync(0xffffffffu, p.acc[j], 16);
    }
    if (whole) {
      attn_store<DH>(a, p, r, hd, lane);
    } else {
      float* slot = sc->slot[wid][own ? 1 : 0];
      if (vk == 0) *reinterpret_cast<float4*>(slot + dl) = make_float4(p.acc[0], p.acc[1], p.acc[2], p.acc[3]);
      if (lane == 0) { slot[128] = p.m; slot[129] = p.l; }
    }
    if (left > 0) {
      ui = 0;
      if (++hd == H) {
        hd = 0;
        do ++r; while (sm->prefix[r + 1] == sm->prefix[r]);
      }
    }
  }
  if (!sm->att_cut) return;

  // ---- pairs cut between warps or CTAs
  named_bar_workers();
  if (sm->abort) return;
  auto add_slot = [&](AttnPartial& p, int w, int which) {
    const float* slot = sc->slot[w][which];
    attn_merge(p, *reinterpret_cast<const float4*>(slot + dl), slot[128], slot[129]);
  };
  AttnPartial zero;
  zero.m = -CUDART_INF_F;
  zero.l = 0.f;
#pragma unroll
  for (int j = 0; j < 4; ++j) zero.acc[j] = 0.f;
  // the pair this CTA's range starts inside of: its owner is an earlier CTA
  if (wid == 0 && sm->att_head >= 0) {
    AttnPartial p = zero;
    p.m = -3.0e38f;                                       // finite: an empty start leaves exp2f(m - max) at 0 and not at NaN
    for (int w = 0; w < 8; ++w)
      if (sm->sl_head[w] == sm->att_head) add_slot(p, w, 0);
    float* out = a.att_part + (size_t)blockIdx.x * (DH + 4);
    if (vk == 0) __stcg(reinterpret_cast<float4*>(out + dl), make_float4(p.acc[0], p.acc[1], p.acc[2], p.acc[3]));
    if (lane == 0) { __stcg(out + DH, p.m); __stcg(out + DH + 1, p.l); }
    __syncwarp();
    if (lane == 0) asm volatile("st.release.gpu.global.u64 [%0], %1;" ::"l"(a.att_flag + blockIdx.x), "l"(ticket) : "memory");
  }
  const int pair = sm->sl_tail[wid];
  if (pair >= 0) {
    AttnPartial p = zero;
    p.m = -3.0e38f;
    add_slot(p, wid, 1);
    for (int w = wid + 1; w < 8; ++w)
      if (sm->sl_head[w] == pair) add_slot(p, w, 0);
    const int pr = pair / H, ph = pair - pr * H;
    const int end = sm->prefix[pr] * H + (ph + 1) * (sm->prefix[pr + 1] - sm->prefix[pr]);
    bool ok = true;
    // (ranges end between pairs in a step without long rows: then no other CTA starts before this pair's end)
    if (sm->max_units >= kAttnCutUnits) {
      for (int c = blockIdx.x + 1; c < (int)gridDim.x && ok; ++c) {
        const int b0 = unit_at(sm, H, range_begin(sm, H, c, gridDim.x, lane), lane);
        const int b1 = unit_at(sm, H, range_begin(sm, H, c + 1, gridDim.x, lane), lane);
        if (b0 >= end) break;
        if (b0 == b1) continue;                           // fewer units than CTAs
        if (lane == 0) {
          const long long t0 = clock64();
          while (ld_acquire_u64(a.att_flag + c) != ticket) {
            if (sm->abort) { ok = false; break; }
            if (clock64() - t0 > a.wait_limit) {
              atomicCAS(a.status, 0u, (uint32_t)kStatusFlagTimeout);
              sm->abort = 1;
              ok = false;
              break;
            }
          }
        }
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
        __syncwarp();                                     // lane 0's acquire holds for every lane's reads (a vote orders no memory)
        const float* in = a.att_part + (size_t)c * (DH + 4);
        attn_merge(p, __ldcg(reinterpret_cast<const float4*>(in + dl)), __ldcg(in + DH), __ldcg(in + DH + 1));
      }
    }
    if (!ok) return;
    attn_store<DH>(a, p, pr, ph, lane);
  }
}

// ---- stage: SwiGLU ----------------------------------------------------------------------------------
// Work unit = (row, 256 features) per warp: gate and up rows alternate in the weights, so a lane's four loads of four
// consecutive outputs are two features each (and a warp-wide load covers 512 contiguous bytes of a partial segment); units
// are dealt round-robin over the CTAs.  The row is the warp's own, so its 1/rms is two more loads beside the partials
// instead of a pass over all rows with a barrier behind it (200 rows: 19.3 -> 10.2 us).
template <bool FLAG>
__device__ void stage_swiglu(const MegaArgs& a, MegaSmem* sm, int wtid) {
  const MegaGemmShape& gs = a.shape[2];
  const int lane = wtid & 31, wid = wtid >> 5;
  const int nc = (a.F + 255) >> 8, n_units = a.B * nc;
  for (int u = wid * gridDim.x + blockIdx.x; u < n_units; u += 8 * gridDim.x) {
    const int r = u / nc, n0 = (u - r * nc) * 512 + lane * 4;        // outputs: gate, up, gate, up of two features
    if (!sm->active_s[r]) continue;
    PartialLoads<4, 2> q[4];
    int4 ts[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int n = n0 + 128 * k < 2 * a.F ? n0 + 128 * k : 0;       // lanes beyond the last feature read the first ones, store nothing
      ts[k] = tile_seg(sm, gs, n);
      partials_issue<FLAG, 4, 2>(a, gs, ts[k], n, r, q[k]);
    }
    const float inv = warp_row_inv_rms(a, r, lane);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int n = n0 + 128 * k;
      if (n >= 2 * a.F) continue;
      float x[4];
      partials_sum<FLAG, 4, 2>(a, sm, gs, ts[k], n, r, q[k], x);
      const float g0 = x[0] * inv, g1 = x[2] * inv;
      const __nv_bfloat162 o = __floats2bfloat162_rn(__fdividef(g0, 1.f + __expf(-g0)) * (x[1] * inv),
                                                     __fdividef(g1, 1.f + __expf(-g1)) * (x[3] * inv));
      *reinterpret_cast<__nv_bfloat162*>(a.act + (size_t)r * a.F + (n >> 1)) = o;
    }
  }
}

// ---- stage: per-tile arg-max of the logits --------------------------------------------------------------
// A warp has one 256-row vocabulary tile (so its table entry is looked up once) and takes batch rows two at a time, in
// turn with the other warps of the tile; 2 x 4 consecutive ids per lane: the decision among a lane's ids needs no
// exchange, so a (tile, row) costs one warp reduction, and many rows spread over every warp of the chip.  At first a
// tile's 128 ids sat on 128 threads that walked through all rows one after the other, a reduction each, on half of the
// CTAs (16 / 96 / 200 rows: 17.8 / 56.8 / 108 us); units of (tile, two rows) with a look-up each: 8.8 / 25.1 / 43.7;
// now 4.7 / 11.9 / 24.8.
template <bool FLAG>
__device__ void stage_tile_argmax(const MegaArgs& a, MegaSmem* sm, int wtid) {
  const MegaGemmShape& gs = a.shape[4];
  const int lane = wtid & 31, wid = wtid >> 5;
  const int n_warps = 8 * gridDim.x, n_pairs = (a.B + 1) >> 1;
  const int n_groups = max(1, min(n_pairs, n_warps / gs.n_tiles));       // warps that share a tile
  const bool sampled = a.sample.inv_temp != 0.f;
  for (int u = wid * gridDim.x + blockIdx.x; u < gs.n_tiles * n_groups; u += n_warps) {
    const int group = u / gs.n_tiles, tile = u - group * gs.n_tiles;
    const int v0 = tile * kTileN + lane * 4;              // and 128 further: a warp-wide load covers 512 contiguous bytes
    const int4 ts = tile_seg(sm, gs, v0);
    for (int rg = group; rg < n_pairs; rg += n_groups) {
      // everything the two rows need is asked for before the first use
      float ss[2];
      int gen[2], row_key[2], skip[2];
      PartialLoads<4, 2> q[2][2];
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const int r = min(2 * rg + k, a.B - 1);
        ss[k] = row_ss_issue(a, r, lane);
#pragma unroll
        for (int h = 0; h < 2; ++h) partials_issue<FLAG, 4, 2>(a, gs, ts, v0 + 128 * h, r, q[k][h]);
        gen[k] = a.st.gen[r] + 1;
        row_key[k] = a.st.row_key[r];
        skip[k] = a.st.eos_at[r] > 0 ? a.eos_id : -1;
      }
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const int r = 2 * rg + k;
        if (r >= a.B || !sm->active_s[r]) continue;       // warp-uniform
        const float inv = row_ss_inv_rms(a, ss[k]);
        uint32_t bk = 0;                                  // below every real key
        int bi = 0x7fffffff;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          float lg[4];
          partials_sum<FLAG, 4, 2>(a, sm, gs, ts, v0 + 128 * h, r, q[k][h], lg);
#pragma unroll
          for (int j = 0; j < 4; ++j) lg[j] *= inv;
          if (a.dump_logits) {
#pragma unroll
            for (int j = 0; j < 4; ++j)
              if (v0 + 128 * h + j < a.V) a.dump_logits[(size_t)r * a.V + v0 + 128 * h + j] = lg[j];
          }
          if (sampled) {                                  // four draws side by side: each is a chain of ten rounds
#pragma unroll
            for (int j = 0; j < 4; ++j) lg[j] = sampled_value(lg[j], a.sample, v0 + 128 * h + j, gen[k], row_key[k]);
          }
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const int v = v0 + 128 * h + j;
            const uint32_t key = v < a.V && v != skip[k] ? float_order_key(lg[j]) : 0u;
            if (key > bk) { bk = key; bi = v; }           // ids ascend: '>' keeps the lowest
          }
        }
        const uint32_t best = __reduce_max_sync(0xffffffffu, bk);
        bi = (int)__reduce_min_sync(0xffffffffu, bk == best ? (unsigned int)bi : 0x7fffffffu);
        if (lane == 0) {
          a.tile_val[(size_t)r * a.n_tiles_lm + tile] = __uint_as_float(best);
          a.tile_idx[(size_t)r * a.n_tiles_lm + tile] = bi;
        }
      }
    }
  }
}

// ---- stage: final arg-max over tiles + row bookkeeping (one warp per row) -------------------------------
static __device__ void stage_final(const MegaArgs& a, int wtid) {
  const int lane = wtid & 31, wid = wtid >> 5;
  for (int r = blockIdx.x * 8 + wid; r < a.B; r += gridDim.x * 8) {
    int tok = a.eos_id;
    if (a.st.active[r]) {
      uint32_t bk = 0;
      int bi = 0x7fffffff;
      for (int t = lane; t < a.shape[4].n_tiles; t += 32) {
        const uint32_t k = __float_as_uint(__ldcg(a.tile_val + (size_t)r * a.n_tiles_lm + t));
        const int id = __ldcg(a.tile_idx + (size_t)r * a.n_tiles_lm + t);
        if (k > bk || (k == bk && id < bi)) { bk = k; bi = id; }
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const uint32_t ok = __shfl_xor_sync(0xffffffffu, bk, o);
        const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
        if (ok > bk || (ok == bk && oi < bi)) { bk = ok; bi = oi; }
      }
      if (lane == 0) {
        a.st.ctx_len[r] += 1;
        const int cap = a.st.scalars[0];
        const int gidx = a.st.gen[r] + 1;
        tok = (bi == 0x7fffffff) ? 0 : bi;
        if (a.dump_choice) a.dump_choice[r] = tok;
        if (a.st.eos_at[r] > 0 && gidx == a.st.eos_at[r]) tok = a.eos_id;
        if (a.forced) tok = a.forced[r];
        a.st.out_tokens[(size_t)r * a.st.max_new + (gidx - 1)] = tok;
        a.st.gen[r] = gidx;
        a.st.cur_tok[r] = tok;
        if (tok == a.eos_id) { a.st.finished[r] = 1; a.st.active[r] = 0; }
        else if (gidx >= cap) { a.st.active[r] = 0; }
        else atomicAdd(a.st.scalars + 1, 1);
      }
    }
    if (lane == 0 && a.next_tokens) a.next_tokens[r] = tok;
  }
}

// ------------------------------------------------------------------------------------ the kernel
// ROWS: batches of up to 16, 64 (64 token lanes per instruction) or 128 rows, or up to 256, on pairs of CTAs (a
// cluster of two, 128 lanes in each).  At first 256 rows were two instructions of 128 lanes on one CTA: both halves of the
// tensor memory in one accumulator, so that every segment's drain held up the MMAs, and 148 ranges to write partials for
// instead of 74.  7B shape, 4 layers, 136 / 160 / 200 / 256 rows: 957 / 1088 / 1280 / 1200 -> 860 / 960 / 1145 / 1035 us a
// step; 32 x 64 heads, 160 / 256 rows: 650 / 831 -> 515 / 646.
// TRACE: with the stage-boundary time stamps of CTA 0 (ss_set_trace); the timed paths run the variant without them.
template <int DH, int ROWS, bool TRACE>
__global__ void __launch_bounds__(kMegaThreads, 1)
decode_step_mega_kernel(const __grid_constant__ CUtensorMap map_x, const __grid_constant__ CUtensorMap map_o,
                        const __grid_constant__ CUtensorMap map_act, const __grid_constant__ CUtensorMap map_w,
                        const __grid_constant__ MegaArgs a) {
  constexpr bool WIDE = ROWS > 64, PAIR = ROWS > 128, FLAG = ROWS == 16;
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  MegaSmem* sm = reinterpret_cast<MegaSmem*>(smem_raw);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int cta = blockIdx.x;
  float* scratch = reinterpret_cast<float*>(smem_raw + sizeof(MegaSmem));
  const uint32_t stage0 = (smem_u32(smem_raw) + (uint32_t)(sizeof(MegaSmem) + mega_scratch_bytes(WIDE)) + 1023u) & ~1023u;
  // ring: S activation blocks first, then S weight blocks.  A token tile shorter than the instruction's lanes is read
  // by the tensor core as that many rows anyway; the surplus rows fall on the blocks that follow.
  const uint32_t rank = PAIR ? cluster_cta_rank() : 0u;    // in the pair: 0 issues the MMAs
  const int part = PAIR ? cta >> 1 : cta;                  // whose range of a projection this CTA works on
  const uint32_t x_bytes = (uint32_t)a.x_rows * kTileK * 2;
  constexpr uint32_t w_bytes = PAIR ? kBlockBytes / 2 : kBlockBytes;
  // what lands in a stage; on pairs in both CTAs together, counted by the first one's barrier
  const uint32_t stage_tx = (PAIR ? 2u : 1u) * (w_bytes + x_bytes);
  const int S = a.stages;
  const uint32_t x0 = stage0, w0 = stage0 + (uint32_t)S * x_bytes;
  const uint32_t kv0 = w0 + (uint32_t)S * w_bytes;         // the worker warps' pieces of the cache scan
  constexpr uint32_t kTmemCols = 512;
  const int n_gemm = 4 * a.n_layers + 1;

  if (threadIdx.x == 0) {
    for (int s = 0; s < S; ++s) {
      mbar_init(smem_u32(&sm->full[s]), 1);
      mbar_init(smem_u32(&sm->empty[s]), 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(smem_u32(&sm->acc_full[b]), 1);
      mbar_init(smem_u32(&sm->acc_empty[b]), PAIR ? 16 : 8);   // every worker warp (pairs: of both CTAs, used in the first)
    }
    for (int b = 0; b < 8 * kKvMaxPieces; ++b) mbar_init(smem_u32(&sm->kv_full[0][0] + b), 1);
    mbar_init(smem_u32(&sm->mma_done), 1);
    sm->w_issued = 0;
    sm->act_epoch = 0;
    sm->abort = 0;
    sm->leave = 0;
    fence_barrier_init();
    tma_prefetch_desc(&map_x);
    tma_prefetch_desc(&map_o);
    tma_prefetch_desc(&map_act);
    if (PAIR) tma_prefetch_desc(&map_w);
  }
  if (warp == 1) {
    if constexpr (PAIR) {
      tmem_alloc_pair(smem_u32(&sm->tmem_base), kTmemCols);
      tmem_relinquish_pair();
    } else {
      tmem_alloc(smem_u32(&sm->tmem_base), kTmemCols);
      tmem_relinquish();
    }
  }
  tc_fence_before();
  __syncthreads();
  if (PAIR) cluster_sync_all();                      // both CTAs' barriers exist before either signals the other's
  tc_fence_after();
  const uint32_t tmem_base = sm->tmem_base;

  if (warp == 0) {
    // ===================== weight producer =====================
    if (lane == 0) {
      uint64_t hint_w;
      asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(hint_w));
      int gi = 0;
      bool ok = true;
      for (int gm = 0; gm < n_gemm && ok; ++gm) {
        const MegaGemmShape& gs = a.shape[gm == n_gemm - 1 ? 4 : (gm & 3)];
        const uint8_t* w = a.wptr[gm];
        // the weights seen as lines of 128 bytes: this CTA's half of a block is 128 of its 256
        const int line0 = PAIR ? (int)((w - a.wbase) >> 7) + (int)rank * kTileM : 0;
        long long it0, it1;
        mega_range(gs, part, it0, it1);
        for (long long it = it0; it < it1; ++it, ++gi) {
          const int stage = gi % S;
          if (gi >= S) {
            ok = mega_wait(smem_u32(&sm->empty[stage]), (uint32_t)(((gi / S) & 1) ^ 1), sm, a.status, kStatusProducerTimeout, a.wait_limit);
            if (!ok) break;
          }
          const uint32_t full = smem_u32(&sm->full[stage]);
          if (rank == 0) mbar_expect_tx(full, stage_tx);
          if constexpr (PAIR)
            tma_load_2d_pair(w0 + (uint32_t)stage * w_bytes, &map_w, full, 0, line0 + (int)it * kTileN, hint_w);
          else
            bulk_load(w0 + (uint32_t)stage * w_bytes, w + (size_t)it * kBlockBytes, kBlockBytes, full, hint_w);
          __threadfence_block();
          sm->w_issued = gi + 1;
        }
      }
      if (!ok || sm->abort) {
        // The step was abandoned.  Before this CTA gives its shared memory up, the bulk copies it still has in
        // flight (at most the last S ring stages) are given time to land: a bounded look at each stage's barrier,
        // which flips once the stage's bytes are in (a stage whose activation block was never requested does not
        // flip; its weight block has landed long before the limit, a thousand times a copy's latency, runs out).
        // (On pairs the second CTA has no barrier of its own to look at: both wait the limit once.)
        for (int j = !PAIR && gi > S ? gi - S : 0; j < (PAIR ? 1 : gi); ++j) {
          const long long t0 = clock64();
          while ((PAIR || !mbar_try_wait(smem_u32(&sm->full[j % S]), (uint32_t)((j / S) & 1))) && clock64() - t0 < 2000000LL) __nanosleep(100);
        }
      }
    }
  } else if (warp == 2) {
    // ===================== activation loader =====================
    if (lane == 0) {
      uint64_t hint_x;
      asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(hint_x));
      int gi = 0;
      bool ok = true;
      for (int gm = 0; gm < n_gemm && ok; ++gm) {
        const int type = gm == n_gemm - 1 ? 4 : (gm & 3);
        const MegaGemmShape& gs = a.shape[type];
        const CUtensorMap* mp = (type == 1) ? &map_o : (type == 3) ? &map_act : &map_x;
        long long it0, it1;
        mega_range(gs, part, it0, it1);
        if (it0 == it1) continue;
        // the operand is complete once the workers have passed the grid barrier before this projection
        {
          const long long t0 = clock64();
          while (sm->act_epoch <= gm) {
            __nanosleep(20);
            if (sm->abort) { ok = false; break; }
            if (clock64() - t0 > a.wait_limit) {
              atomicCAS(a.status, 0u, (uint32_t)kStatusFlagTimeout);
              sm->abort = 1;
              ok = false;
              break;
            }
          }
          if (!ok) break;
          // the worker that set the flag had acquired the grid barrier at gpu scope and released the flag at CTA
          // scope; a CTA-scope fence here completes the chain (a gpu-scope fence costs a round trip to L2)
          __threadfence_block();
          fence_proxy_async_global();          // global only: the full fence stalls ~2 us while ring copies are in flight
        }
        int k = (int)(it0 % gs.kb);
        for (long long it = it0; it < it1; ++it, ++gi) {
          const long long t0 = clock64();
          while (sm->w_issued <= gi) {
            __nanosleep(40);
            if (sm->abort) { ok = false; break; }
            if (clock64() - t0 > a.wait_limit) {
              atomicCAS(a.status, 0u, (uint32_t)kStatusFlagTimeout);
              sm->abort = 1;
              ok = false;
              break;
            }
          }
          if (!ok) break;
          const int stage = gi % S;
          if constexpr (PAIR)
            tma_load_2d_pair(x0 + (uint32_t)stage * x_bytes, mp, smem_u32(&sm->full[stage]), k * kTileK, (int)rank * a.x_rows, hint_x);
          else
            tma_load_2d(x0 + (uint32_t)stage * x_bytes, mp, smem_u32(&sm->full[stage]), k * kTileK, 0, hint_x);
          if (++k == gs.kb) k = 0;
        }
      }
    }
  } else if (warp == 1) {
    // ===================== MMA issuer (pairs: in the first CTA) =====================
    if (lane == 0 && rank == 0) {
      // M = token lanes (64 up to 64 rows: half the tensor-core work on unused lanes), N = 256 weight rows
      const uint32_t idesc = umma_idesc_bf16(kTileN, ROWS < 64 ? 64 : ROWS);
      int gi = 0, seg = 0;
      bool ok = true;
      for (int gm = 0; gm < n_gemm && ok; ++gm) {
        const MegaGemmShape& gs = a.shape[gm == n_gemm - 1 ? 4 : (gm & 3)];
        long long it0, it1;
        mega_range(gs, part, it0, it1);
        long long it = it0;
        while (it < it1 && ok) {
          const int tile = (int)(it / gs.kb);
          long long seg_end = (long long)(tile + 1) * gs.kb;
          if (seg_end > it1) seg_end = it1;
          const int buf = seg & 1;
          ok = mega_wait(smem_u32(&sm->acc_empty[buf]), (uint32_t)(((seg >> 1) & 1) ^ 1), sm, a.status, kStatusMmaTimeout, a.wait_limit);
          if (!ok) break;
          tc_fence_after();
          const uint32_t d_tmem = tmem_base + (uint32_t)(buf * kTileN);
          bool first = true;
          for (; it < seg_end; ++it, ++gi) {
            const int stage = gi % S;
            ok = mega_wait(smem_u32(&sm->full[stage]), (uint32_t)((gi / S) & 1), sm, a.status, kStatusMmaTimeout, a.wait_limit);
            if (!ok) break;
            tc_fence_after();
            const uint64_t dw = smem_desc_sw128(w0 + (uint32_t)stage * w_bytes);
            const uint64_t dx = smem_desc_sw128(x0 + (uint32_t)stage * x_bytes);
#pragma unroll
            for (int k = 0; k < kTileK / 16; ++k) {
              const uint32_t add = (first && k == 0) ? 0u : 1u;
              if constexpr (PAIR) umma_bf16_pair(d_tmem, dx + (uint64_t)(k * 2), dw + (uint64_t)(k * 2), idesc, add);
              else umma_bf16(d_tmem, dx + (uint64_t)(k * 2), dw + (uint64_t)(k * 2), idesc, add);
            }
            first = false;
            if constexpr (PAIR) umma_commit_pair(smem_u32(&sm->empty[stage]));
            else umma_commit(smem_u32(&sm->empty[stage]));
          }
          if (!ok) break;
          if constexpr (PAIR) umma_commit_pair(smem_u32(&sm->acc_full[buf]));
          else umma_commit(smem_u32(&sm->acc_full[buf]));
          ++seg;
        }
      }
      if (!ok) {
        // The step was abandoned, perhaps by another role right behind an issue: the MMAs in flight read the ring and write
        // the accumulators, and get a bounded time to end before either is given up.
        if constexpr (PAIR) umma_commit_pair(smem_u32(&sm->mma_done));
        else umma_commit(smem_u32(&sm->mma_done));
        const long long t0 = clock64();
        while (!mbar_try_wait(smem_u32(&sm->mma_done), 0) && clock64() - t0 < 2000000LL) __nanosleep(100);
      }
    }
  } else if (warp >= 3) {
    // ===================== workers =====================
    const int wtid = threadIdx.x - 96;
    const int wid = wtid >> 5;
    const int quarter = warp & 3;                   // tensor-memory lane quarter this warp may read
    const int colhalf = wid >> 2;                   // warps 3-6 take the first 128 weight rows of a tile
    unsigned long long epoch = 0;
    int seg = 0;
    bool ok = true;

    const bool tracer = TRACE && cta == 0 && wtid == 0 && a.trace != nullptr;
    int tr = 0;
    if (tracer) a.trace[tr++] = global_timer_ns();
    if (cta == 0 && wtid == 0) a.st.scalars[1] = 0;   // rows still active after this step (counted in the last stage)
    attention_setup<DH>(a, sm, wtid);
    KvStream kvs;
    kv_stream_start<DH>(a, sm, kvs, kv0, wid, lane);
    stage_residual<FLAG, PAIR ? 6 : 12>(a, sm, wtid, 0, nullptr, a.norm_ptr[0], a.n_layers == 0);
    ok = grid_barrier(a, sm, epoch, wtid, true);
    if (ok && wtid == 0) { __threadfence_block(); sm->act_epoch = 1; }
    if (tracer) a.trace[tr++] = global_timer_ns();

    for (int gm = 0; gm < n_gemm && ok; ++gm) {
      const int type = gm == n_gemm - 1 ? 4 : (gm & 3);
      const int layer = gm >> 2;
      const MegaGemmShape& gs = a.shape[type];
      float* const partial = gs.partial;
      // ---- drain this CTA's segments of projection gm into fp32 partials
      long long it0, it1;
      mega_range(gs, part, it0, it1);
      long long it = it0;
      int seg_local = 0;
      while (it < it1) {
        const int tile = (int)(it / gs.kb);
        long long seg_end = (long long)(tile + 1) * gs.kb;
        if (seg_end > it1) seg_end = it1;
        const int buf = seg & 1;
        const bool full = mega_wait(smem_u32(&sm->acc_full[buf]), (uint32_t)((seg >> 1) & 1), sm, a.status, kStatusEpilogueTimeout, a.wait_limit);
        if (!__all_sync(0xffffffffu, full)) break;             // aborted: this warp goes on to the next grid barrier, where all leave
        tc_fence_after();
        const size_t slot = (size_t)part * gs.max_seg + seg_local;
        // batch rows held by this warp's lanes: 32 per lane quarter (16 with the 64-row instruction), on pairs as far as the
        // CTA's half of the batch goes
        constexpr int cap_q = WIDE ? 32 : 16;
        const int per_q = PAIR ? min(32, a.x_rows - quarter * 32) : cap_q;
        const int tok0 = (int)rank * a.x_rows + quarter * cap_q;
        if (per_q > 0 && tok0 < a.B) {                         // else no batch row in this warp's lanes (warp-uniform)
          const int tok = lane < per_q ? tok0 + lane : a.B;
          const uint32_t taddr = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(buf * kTileN + colhalf * 128);
          float* dst = partial + (slot * a.NT + tok) * kTileN + colhalf * 128;
          // 64 columns per TMEM load: the last segment's drain is the serial tail of every projection
#pragma unroll 1
          for (int c = 0; c < 128; c += 64) {
            uint32_t v[64];
            tmem_ld64(taddr + c, v);
            if constexpr (FLAG) {
#pragma unroll
              for (int j = 0; j < 64; ++j) v[j] = min(v[j], kNoPartial - 1u);      // (a NaN stays one)
            }
            if constexpr (FLAG) {
              // one MMA's worth of rows or fewer: the tail is a chain of latencies, direct stores are the shortest one
              if (tok < a.B) {
#pragma unroll
                for (int j = 0; j < 64; j += 4)
                  st_partial(dst + c + j, v[j], v[j + 1], v[j + 2], v[j + 3]);
              }
            } else {
              // many rows: a lane holds one token's outputs, so direct 128-bit stores put every lane's 16 bytes
              // into a sector of its own, 1 KiB apart, and the drain is bound by the sectors it writes.  The
              // warp turns 16 outputs at a time through shared memory and stores 64-byte runs, eight tokens per
              // instruction.  (Direct 256-bit stores, a whole sector each: up to 5 % slower at 160 to 256 rows.)
              float* tr = scratch + wid * (cap_q * kDrainPad);
              const int t_hi = lane >> 2, cg = lane & 3;
#pragma unroll
              for (int sub = 0; sub < 4; ++sub) {
                if (lane < per_q) {
#pragma unroll
                  for (int j = 0; j < 16; j += 4)
                    *reinterpret_cast<uint4*>(tr + lane * kDrainPad + j) =
                        make_uint4(v[sub * 16 + j], v[sub * 16 + j + 1], v[sub * 16 + j + 2], v[sub * 16 + j + 3]);
                }
                __syncwarp();
#pragma unroll
                for (int i = 0; i < cap_q / 8; ++i) {
                  const int tl = 8 * i + t_hi;
                  if (tl < per_q && tok0 + tl < a.B)
                    *reinterpret_cast<uint4*>(partial + (slot * a.NT + tok0 + tl) * kTileN + colhalf * 128 + c + sub * 16 + 4 * cg) =
                        *reinterpret_cast<const uint4*>(tr + tl * kDrainPad + 4 * cg);
                }
                __syncwarp();
              }
            }
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) {
          if (rank == 0) mbar_arrive(smem_u32(&sm->acc_empty[buf]));
          else mbar_arrive_leader(smem_u32(&sm->acc_empty[buf]));
        }
        it = seg_end;
        ++seg;
        ++seg_local;
      }
      if (tracer) a.trace[tr++] = global_timer_ns();       // this CTA's accumulators drained
      if constexpr (!FLAG) {
        ok = grid_barrier(a, sm, epoch, wtid, false);
        if (!ok) break;
      }
      if (tracer) a.trace[tr++] = global_timer_ns();       // every CTA's partials visible (FLAG: the stage looks for them)
      // ---- the stage that consumes the projection
      if (type == 0) {
        stage_attention<DH, FLAG>(a, sm, reinterpret_cast<AttnScratch*>(scratch), kvs, wtid, layer, a.grid_base + epoch);
      } else if (type == 1) {
        stage_residual<FLAG, PAIR ? 6 : 12>(a, sm, wtid, 1, &a.shape[1], a.norm_ptr[2 * layer + 1], false);
      } else if (type == 2) {
        stage_swiglu<FLAG>(a, sm, wtid);
      } else if (type == 3) {
        stage_residual<FLAG, PAIR ? 6 : 12>(a, sm, wtid, 1, &a.shape[3], a.norm_ptr[2 * layer + 2], layer + 1 == a.n_layers);
      } else {
        stage_tile_argmax<FLAG>(a, sm, wtid);
      }
      if (tracer) a.trace[tr++] = global_timer_ns();       // this CTA's share of the stage done
      ok = grid_barrier(a, sm, epoch, wtid, true);
      if (!ok) break;
      if (tracer) a.trace[tr++] = global_timer_ns();       // stage complete everywhere
      if (type == 4) stage_final(a, wtid);
      else if (wtid == 0) { __threadfence_block(); sm->act_epoch = gm + 2; }
      if constexpr (FLAG) clear_partials(a, gs, part, wtid);
    }
    kv_stream_end(a, sm, kvs, wid, lane);
  }

  tc_fence_before();
  __syncthreads();
  // neither CTA of a pair may give up its shared or tensor memory while the other's MMAs or copies can still touch it
  if (PAIR) cluster_sync_all();
  if (warp == 1) {
    tc_fence_after();
    if constexpr (PAIR) tmem_dealloc_pair(tmem_base, kTmemCols);
    else tmem_dealloc(tmem_base, kTmemCols);
  }
}

// The instantiation for batches of up to 16 / 64 / 128 / 256 rows, without or with the stage trace.
template <int DH>
const void* mega_kernel_of(int rows, bool trace) {
  if (rows == 256) return trace ? (const void*)decode_step_mega_kernel<DH, 256, true> : (const void*)decode_step_mega_kernel<DH, 256, false>;
  if (rows == 128) return trace ? (const void*)decode_step_mega_kernel<DH, 128, true> : (const void*)decode_step_mega_kernel<DH, 128, false>;
  if (rows == 16) return trace ? (const void*)decode_step_mega_kernel<DH, 16, true> : (const void*)decode_step_mega_kernel<DH, 16, false>;
  return trace ? (const void*)decode_step_mega_kernel<DH, 64, true> : (const void*)decode_step_mega_kernel<DH, 64, false>;
}
const void* mega_kernel_64(int rows, bool trace);          // ss_mega_64.cu
const void* mega_kernel_128(int rows, bool trace);         // ss_mega_128.cu

// Self-test of the workers' way out: eight worker warps that come to one grid barrier after the other at different times,
// and a ninth warp that raises the abort flag in between, at another time in every CTA.  All eight must have passed the
// same number of barriers; *torn counts the CTAs where they have not.
constexpr int kLeaveSelftestThreads = kMegaWorkers + 32;
static __global__ void __launch_bounds__(kLeaveSelftestThreads, 1)
leave_selftest_kernel(const __grid_constant__ MegaArgs a, uint32_t* torn) {
  __shared__ MegaSmem smem;
  MegaSmem* sm = &smem;
  if (threadIdx.x == 0) sm->abort = sm->leave = 0;
  __syncthreads();
  const int wid = threadIdx.x >> 5;
  auto pause = [](long long cycles) {
    const long long t0 = clock64();
    while (clock64() - t0 < cycles) { }
  };
  if (wid < 8) {
    unsigned long long epoch = 0;
    bool ok = true;
    while (ok) {
      pause(((unsigned)(wid * 5 + blockIdx.x) * 7u + (unsigned)epoch * 3u) % 8u * 150u);
      ok = grid_barrier(a, sm, epoch, threadIdx.x, false);
    }
    if ((threadIdx.x & 31) == 0) sm->prefix[wid] = (int)epoch;
  } else if (threadIdx.x == kMegaWorkers) {
    pause(60000 + 37 * (long long)blockIdx.x);             // some dozens of barriers
    sm->abort = 1;
  }
  __syncthreads();
  if (threadIdx.x == 0)
    for (int w = 1; w < 8; ++w)
      if (sm->prefix[w] != sm->prefix[0]) { atomicAdd(torn, 1u); break; }
}

// Self-test of the bounded waits between SMs and on barriers, with nothing else in flight (no bulk copies, no tensor-core
// work).  Every CTA has one of them, for something that never comes: an arrival more than the grid can deliver; partial sums
// in an empty slot; the completion of a barrier that nobody arrives on; a flag that nobody sets.  Each must run out after
// a.wait_limit cycles, record its status and let the kernel end normally; *ran_out gets a bit for each that did.
constexpr uint32_t kWaitSelftests = 4;
static __global__ void __launch_bounds__(32)
wait_selftest_kernel(const __grid_constant__ MegaArgs a, const uint32_t* flag, uint32_t* ran_out) {
  __shared__ MegaSmem smem;
  MegaSmem* sm = &smem;
  const int lane = threadIdx.x;
  const uint32_t which = blockIdx.x % kWaitSelftests, bar = smem_u32(&sm->acc_full[0]);
  if (lane == 0) {
    sm->abort = 0;
    mbar_init(bar, 1);
    fence_barrier_init();
  }
  __syncwarp();
  bool ended = false;
  if (which == 1) {
    PartialLoads<4, 2> q;
    float x[4];
    const int4 only_slot0 = make_int4(0, 1, 0, 0);
    partials_issue<true, 4, 2>(a, a.shape[0], only_slot0, lane * 4, 0, q);
    partials_sum<true, 4, 2>(a, sm, a.shape[0], only_slot0, lane * 4, 0, q, x);
    ended = __all_sync(0xffffffffu, no_partial<4>(q.x));
  } else if (lane == 0) {
    if (which == 0) {
      ended = !arrive_and_poll(a.grid_ctr, a.grid_base + (unsigned long long)gridDim.x + 1ULL, a.wait_limit, nullptr);
      if (ended) atomicCAS(a.status, 0u, (uint32_t)kStatusGridBarrierTimeout);
    } else if (which == 2) {
      ended = !mega_wait(bar, 0, sm, a.status, kStatusMmaTimeout, a.wait_limit);
    } else {
      ended = !flag_wait(flag, a.status, a.wait_limit);
    }
  }
  if (lane == 0 && ended) atomicOr(ran_out, 1u << which);
}

}  // namespace ss
