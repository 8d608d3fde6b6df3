// Internal declarations shared by the host runtime and the kernel launchers.
#pragma once

#include <cstddef>
#include <cstdint>
#include <vector_types.h>
#include <vector>

#include "seqsched.h"

namespace ss {

// ---- scheduler (ss_sched.cpp) ------------------------------------------------------------
int validate_sched_cfg(const ss_sched_cfg* c);
int32_t length_bin(int32_t x, const ss_sched_cfg& c);
int32_t batch_allowance(int32_t L, const ss_sched_cfg& c);
int plan_first_pass(const ss_sched_cfg& c, const int32_t* prompt_len, const int32_t* pred_len,
                    const int32_t* perm, int32_t n, std::vector<int32_t>& order,
                    std::vector<ss_batch_desc>& out);

// ---- constants ---------------------------------------------------------------------------
constexpr int kPageTokens = 32;        // tokens per key/value page
constexpr int kTileM = 128;            // weight rows per GEMM tile (tcgen05 M)
constexpr int kTileK = 64;             // bf16 elements per 128-byte swizzled row
constexpr int kTileN = 256;            // weight rows per block of the tiled layout (tcgen05 N of the decode step)
constexpr int kBlockBytes = kTileN * kTileK * 2;   // one (256-row tile, k-block) block: 32 KiB
constexpr int kMaxBatch = 256;

// Device status codes (which bounded wait expired / which check failed).
enum : uint32_t {
  kStatusOk = 0,
  kStatusProducerTimeout = 1,
  kStatusMmaTimeout = 2,
  kStatusEpilogueTimeout = 3,
  kStatusBadPage = 4,
  kStatusGridBarrierTimeout = 5,
  kStatusFlagTimeout = 6,
};

// SM cycles (about 2 s) that any wait inside a kernel may last unless ss_set_wait_limit_ms() says otherwise.
constexpr long long kDefaultWaitLimit = 4000000000LL;

// ---- GEMM:  D[n_out, tok] = W[n_out, K] . X[tok, K]^T  -------------------------------------
// gemm_wx_kernel: the tile-iteration space (n_tiles x kb) is cut into `gridx` equal contiguous ranges, one per CTA (split
// along K where a range ends inside a tile); every (CTA, tile) segment is written as an fp32 partial and the consumer
// kernel adds the segments of a tile in CTA order, so the result does not depend on timing.
// gemm_wx_pair_kernel finishes a tile in its epilogue: added to the fp32 residual; rotated and written as bf16 q, k, v
// operand and cache entries; or gated (SwiGLU) and written as bf16 operand.
enum GemmMode : int { kGemmResidual = 1, kGemmQkv = 2, kGemmSwiglu = 3 };

struct GemmPlan {
  int n_out, K, n_tiles, kb;
  int NT;              // token tile (tcgen05 N), multiple of 16, <= 256
  int gridx;           // CTAs (pairs of CTAs in gemm_wx_pair_kernel)
  // gemm_wx_pair_kernel
  int tok_tiles, group;        // token tiles, and how many of them the pairs go through together
  int split_units, ranges;     // units (256 weight rows, token tile) that are cut along K, and ranges they are cut into
  int max_seg;         // partial slots per CTA
  int stages;
  int smem_bytes;
  int tmem_cols;
};

struct GemmArgs {
  GemmPlan p;
  const void* w_tiled; // weights repacked as contiguous 32 KiB (256-row tile, k-block) images, or null (row-major via TMA)
  int mode;            // gemm_wx_pair_kernel: GemmMode
  int n_tok;           // valid tokens
  float* partial;      // gemm_wx_kernel: [gridx*max_seg][NT][128]; gemm_wx_pair_kernel: [ranges][2][NT][128]
  uint32_t* pair_flag; // gemm_wx_pair_kernel: [ranges][2][8], set while a partial waits for its owner
  float* residual;     // kGemmResidual: [tok][n_out]
  void* out;           // kGemmQkv: bf16 [tok][3 d]; kGemmSwiglu: bf16 [tok][n_out / 2]
  // kGemmQkv
  int d, H, Dh;
  const float2* rope;          // [position][Dh / 2] (cos, sin)
  const int32_t* tok_pos;      // [tok] position in its row
  const int32_t* tok_slot;     // [tok] page * kPageTokens + place in the page
  void* kv_layer;              // the layer's pages
  size_t page_elems;
  uint32_t* status;
  long long wait_limit;        // SM cycles after which a wait inside the kernel gives up
};

// Where the partial sums of one 128-row tile live: the first segment in slot `slot0`, the others
// in segment 0 of CTAs c_next..c_last (a CTA that starts inside a tile has it as its first tile).
struct TileSeg {
  int32_t slot0, c_next, c_last, pad;
};

// Partial-slot bookkeeping shared by the GEMM and its consumers.
struct SplitInfo {
  int gridx, kb, max_seg, NT;
  long long total;          // n_tiles * kb
  const TileSeg* tiles;     // device table [n_tiles], or null (noalloc_reduce_kernel derives the segments itself)
};

}  // namespace ss
