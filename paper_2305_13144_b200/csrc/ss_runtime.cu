// Host runtime behind the C ABI: context, arena carve-up, weight repacking, key/value page
// allocator, kernel sequencing (prompt pass, decode steps) and the group loop of Sec. 4.1
// (micro-batches, caps, failure collection and recomputation).
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <new>
#include <string>
#include <vector>

#include "ss_decode_mega.cuh"

using namespace ss;

namespace {

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

constexpr size_t kAlign = 1024;
constexpr size_t kRowStateBytes = (size_t)kMaxBatch * 4 * 8;   // 7 row arrays and the scalars
inline size_t align_up(size_t x, size_t a = kAlign) { return (x + a - 1) / a * a; }
inline int ceil_div(int a, int b) { return (a + b - 1) / b; }
inline int round_up(int a, int b) { return ceil_div(a, b) * b; }

// Projection matrices live in the tiled streaming layout (see repack_weights_kernel).
struct LayerWeights {
  bf16 *attn_norm, *ffn_norm;
  uint8_t *wqkv, *wo, *wgu, *wdown;
};

inline size_t tiled_bytes(int64_t n_out, int64_t K) {
  return (size_t)ceil_div((int)n_out, kTileN) * ceil_div((int)K, kTileK) * (size_t)kBlockBytes;
}

// Split of a decode projection: 256-row tiles x k-blocks in equal contiguous ranges over the CTAs.
struct DecodeSplit {
  int n_tiles, kb, gsplit, max_seg;
  long long total;
};
DecodeSplit plan_decode(int n_out, int K, int n_sm) {
  DecodeSplit p{};
  p.n_tiles = ceil_div(n_out, kTileN);
  p.kb = ceil_div(K, kTileK);
  p.total = (long long)p.n_tiles * p.kb;
  p.gsplit = (int)std::min<long long>(n_sm, p.total);
  const int ipc = std::max(1, (int)((p.total + p.gsplit - 1) / p.gsplit));
  p.max_seg = (ipc + p.kb - 2) / p.kb + 1;
  return p;
}

// Split of a projection in 128-row tiles (gemm_wx_kernel) over the SMs, for one tile of NT tokens.
GemmPlan plan_gemm(int n_out, int K, int NT, int n_sm) {
  GemmPlan p{};
  p.n_out = n_out;
  p.K = K;
  p.n_tiles = ceil_div(n_out, kTileM);
  p.kb = ceil_div(K, kTileK);
  p.NT = NT;
  const long long total = (long long)p.n_tiles * p.kb;
  p.gridx = (int)std::min<long long>(n_sm, total);
  const int ipc = std::max(1, (int)((total + p.gridx - 1) / p.gridx));
  p.max_seg = (ipc + p.kb - 2) / p.kb + 1;
  const int stage_bytes = kTileM * kTileK * 2 + NT * kTileK * 2;
  const int budget = 227 * 1024 - 2048;                       // header + alignment slack
  p.stages = std::max(2, std::min(kGemmMaxStages, budget / stage_bytes));
  p.smem_bytes = 2048 + p.stages * stage_bytes;
  int cols = 32;
  while (cols < 2 * NT) cols <<= 1;
  p.tmem_cols = cols;
  return p;
}
// Activations of the token tiles that the pairs of the prompt-pass GEMM go through together.  At 16000 tokens (7B shape, 6
// layers) all 63 tiles in one group read every activation again in each round of pairs, 133 MB against an L2 of 126: 44.2 ms a
// pass, the SMs at 877 MHz under the power cap; groups of 24 / 40 / 64 MB: 35.5 / 34.9 / 36.8 ms, at 1190 MHz.
constexpr size_t kPairGroupBytes = (size_t)40 << 20;
// Token tile of a short prompt chunk.
int short_tile(int tokens) { return std::min(kShortTokens, round_up(tokens, 16)); }

SplitInfo split_of(const GemmPlan& p, const TileSeg* tiles) {
  SplitInfo s;
  s.gridx = p.gridx;
  s.kb = p.kb;
  s.max_seg = p.max_seg;
  s.NT = p.NT;
  s.total = (long long)p.n_tiles * p.kb;
  s.tiles = tiles;
  return s;
}

// Per tile: where its partial segments live (depends on the split only, not on the token tile).
std::vector<TileSeg> tile_table(const GemmPlan& p) {
  SplitInfo s = split_of(p, nullptr);
  std::vector<TileSeg> t(p.n_tiles);
  for (int tile = 0; tile < p.n_tiles; ++tile) {
    const long long x0 = (long long)tile * p.kb;
    const int c0 = split_owner(s, x0), c1 = split_owner(s, x0 + p.kb - 1);
    const int seg0 = tile - (int)(split_begin(s, c0) / p.kb);
    t[tile] = {c0 * p.max_seg + seg0, c0 + 1, c1, 0};
  }
  return t;
}

std::vector<TileSeg> decode_tile_table(const DecodeSplit& p) {
  SplitInfo s{};
  s.gridx = p.gsplit;
  s.kb = p.kb;
  s.max_seg = p.max_seg;
  s.total = p.total;
  std::vector<TileSeg> t(p.n_tiles);
  for (int tile = 0; tile < p.n_tiles; ++tile) {
    const long long x0 = (long long)tile * p.kb;
    const int c0 = split_owner(s, x0), c1 = split_owner(s, x0 + p.kb - 1);
    const int seg0 = tile - (int)(split_begin(s, c0) / p.kb);
    t[tile] = {c0 * p.max_seg + seg0, c0 + 1, c1, 0};
  }
  return t;
}

}  // namespace

struct ss_ctx {
  ss_model_cfg m;
  ss_runtime_cfg rt;
  cudaStream_t stream;
  int n_sm = 0;
  bool use_pdl = true;
  bool trace_on = false;
  long long wait_limit = kDefaultWaitLimit;   // SM cycles any wait inside a kernel may last
  int clock_khz = 1965000;
  int last_cuda = 0;
  int64_t launches = 0;
  EncodeTiledFn encode = nullptr;

  // ---- arena
  uint8_t* arena = nullptr;
  size_t arena_bytes = 0;
  // weights
  bf16 *embed = nullptr, *final_norm = nullptr;
  uint8_t* lm_head = nullptr;
  uint8_t* staging = nullptr;      // one row-major tensor on its way into the tiled layout
  size_t staging_bytes = 0;
  std::vector<LayerWeights> layers;
  std::vector<uint8_t> loaded;     // per tensor slot
  int n_loaded = 0, n_expected = 0;
  // misc device
  float* inv_freq = nullptr;
  float2* rope = nullptr;          // [max_ctx][Dh / 2] (cos, sin)
  uint32_t* status = nullptr;
  RowState st{};
  KvLayout kv{};
  int32_t* d_chunk = nullptr;      // a prompt chunk's arrays, packed: tokens, cache slots, positions, prefix sums, last tokens
  int32_t *d_tokens = nullptr, *d_tok_slot = nullptr, *d_tok_pos = nullptr, *d_cu = nullptr, *d_last = nullptr;
  // prompt-pass activations (R rows)
  int R = 0;
  float* h = nullptr;
  bf16 *x = nullptr, *qkv = nullptr, *attn_o = nullptr, *act = nullptr;
  // decode activations (kMaxBatch rows)
  float* h_dec = nullptr;
  bf16 *x_dec = nullptr, *o_dec = nullptr, *act_dec = nullptr;
  float* partial = nullptr;
  size_t partial_bytes = 0;
  // decode step of up to 16 rows: every projection's partial sums have slots of their own, all ones while nothing is in them
  float* part_dec[5] = {nullptr, nullptr, nullptr, nullptr, nullptr};
  size_t part_dec_bytes = 0;
  TileSeg* tbl[5] = {nullptr, nullptr, nullptr, nullptr, nullptr};   // decode step: qkv, o, gate/up, down, lm head
  TileSeg* tbl_pair[5] = {nullptr, nullptr, nullptr, nullptr, nullptr};   // the same split over pairs of CTAs
  TileSeg* tbl128[5] = {nullptr, nullptr, nullptr, nullptr, nullptr};   // the same projections in 128-row tiles: short prompts, first LM head
  float* rowss = nullptr;          // [kMaxBatch][kMaxSlices]
  unsigned long long* grid_ctr = nullptr;
  float* att_part = nullptr;       // decode attention: partial results that cross CTAs, and their flags
  unsigned long long* att_flag = nullptr;
  uint32_t* pair_flag = nullptr;   // prompt-pass projections: partials that wait for their owner
  unsigned long long* trace = nullptr;  // stage-boundary time stamps of the last decode step
  int trace_len = 0;
  unsigned long long grid_epochs = 0;   // grid barriers passed by all launches so far
  const uint8_t** wptr_dev = nullptr;
  const bf16** norm_dev = nullptr;
  float* tile_val = nullptr;       // [kMaxBatch][n_tiles of the vocabulary]
  int32_t* tile_idx = nullptr;
  int n_tiles_lm = 0;
  // tensor maps for activation operands, keyed by (buffer id, box rows)
  std::map<std::pair<int, int>, CUtensorMap> xmaps;
  // the tiled projection matrices seen as lines of 128 bytes (for the paired prompt-pass GEMM), [4 * layer + type]
  std::vector<CUtensorMap> wmaps;
  CUtensorMap wmap_all;            // all of them in one map, for the decode step on pairs of CTAs

  // ---- page allocator
  std::vector<int32_t> free_pages;
  std::vector<int32_t> batch_pages;      // pages that go back to the pool when the batch in flight is released
  // ---- kept prompts (App. C: the instruction's keys and values computed once, for the perception pass, and used
  // again by the generation): pages that outlive the batch that filled them, by caller-chosen id
  struct KeptPrompt {
    std::vector<int32_t> pages;          // covering positions [0, len)
    int32_t len;                         // tokens kept
    int32_t last_tok;                    // token at position len - 1 (fed again when a batch resumes from here)
  };
  std::map<int32_t, KeptPrompt> kept;
  std::vector<std::vector<int32_t>> row_pages;   // batch in flight: every row's pages in block-table order
  std::vector<int32_t> batch_tokens, batch_cu;   // its prompts (host copy), empty for a resumed batch
  int prompt_cache_mode = 0;                     // ss_run_group / ss_run_batches: 0 off, 1 keep, 2 resume
  std::vector<int32_t> cache_keep_len;           // mode 1: tokens to keep per query

  // ---- batch state (host mirror)
  int B = 0;
  int cap = 0;
  bool in_batch = false;
  std::vector<int32_t> prompt_len;
  int32_t* pinned = nullptr;     // [0] n_active, [1] status
  // Staging for what a batch sends and fetches: a copy costs the host 5 to 10 us each, and a batch needed 2 to 7 on its way
  // up and one per row on its way back (200 rows: 2.2 of 19.7 ms per batch of six steps).  Up: row state and block table
  // as one copy, a chunk's token arrays as another.  Down: row state, tokens.  Page-locked memory was no faster.  A copy
  // from ordinary memory may still be reading its source when the call returns, so `up` is filled again only behind
  // `up_sent`, which is recorded after every copy out of it.
  std::vector<uint8_t> up;
  std::vector<int32_t> down_rows, down_tokens;   // tokens: as many as a batch has brought back so far
  cudaEvent_t up_sent = nullptr;
  cudaEvent_t layers_done = nullptr;   // behind the last layer of a prompt pass
  size_t up_chunk = 0;           // where the chunk arrays start inside `up`
  size_t table_off = 0;          // where the block table starts behind the row state (device and staging alike)
  // ---- sampling (greedy while inv_temp == 0)
  SampleCfg sample{0.f, 0u, 0u};
  std::vector<int32_t> next_row_keys;   // keys of the next batch's rows; empty = 0, 1, 2, ...
};

namespace {

int cuda_fail(ss_ctx* c, cudaError_t e) {
  c->last_cuda = (int)e;
  return SS_ERR_CUDA;
}
#define SS_CUDA(c, expr)                                \
  do {                                                  \
    cudaError_t _e = (expr);                            \
    if (_e != cudaSuccess) return cuda_fail((c), _e);   \
  } while (0)

template <class... KArgs, class... Args>
cudaError_t launch(ss_ctx* c, void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem, Args... args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = c->stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = c->use_pdl ? 1 : 0;
  c->launches++;
  return cudaLaunchKernelEx(&cfg, kern, KArgs(args)...);
}

int make_map(ss_ctx* c, CUtensorMap* out, const void* base, int64_t rows, int64_t cols, int box_rows) {
  cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)cols * 2};
  cuuint32_t box[2] = {(cuuint32_t)kTileK, (cuuint32_t)box_rows};
  cuuint32_t estr[2] = {1, 1};
  CUresult r = c->encode(out, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr,
                         CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                         CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) {
    c->last_cuda = (int)r;
    return SS_ERR_CUDA;
  }
  return SS_OK;
}

// A tiled weight matrix as a 2-D tensor of 128-byte lines (64 bf16 each); box = 128 lines = one CTA's half of a block.
// The lines already hold the swizzled shared-memory image, so the copy itself does not swizzle.
int make_line_map(ss_ctx* c, CUtensorMap* out, const void* base, size_t bytes) {
  cuuint64_t dims[2] = {(cuuint64_t)kTileK, (cuuint64_t)(bytes / 128)};
  cuuint64_t strides[1] = {128};
  cuuint32_t box[2] = {(cuuint32_t)kTileK, (cuuint32_t)kTileM};
  cuuint32_t estr[2] = {1, 1};
  CUresult r = c->encode(out, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr,
                         CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                         CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) {
    c->last_cuda = (int)r;
    return SS_ERR_CUDA;
  }
  return SS_OK;
}

// activation operand map (cached): id 0 = x, 1 = attn_o, 2 = act, 6 = q,k,v (prompt pass); 3 = x_dec, 4 = o_dec, 5 = act_dec
int xmap(ss_ctx* c, int id, int box_rows, const CUtensorMap** out) {
  auto key = std::make_pair(id, box_rows);
  auto it = c->xmaps.find(key);
  if (it == c->xmaps.end()) {
    const int d = c->m.d_model, F = c->m.d_ffn;
    const void* base = nullptr;
    int64_t rows = 0, cols = 0;
    switch (id) {
      case 0: base = c->x; rows = c->R; cols = d; break;
      case 1: base = c->attn_o; rows = c->R; cols = d; break;
      case 2: base = c->act; rows = c->R; cols = F; break;
      case 3: base = c->x_dec; rows = kMaxBatch; cols = d; break;
      case 6: base = c->qkv; rows = c->R; cols = 3 * (int64_t)d; break;
      case 4: base = c->o_dec; rows = kMaxBatch; cols = d; break;
      default: base = c->act_dec; rows = kMaxBatch; cols = F; break;
    }
    CUtensorMap m;
    int rc = make_map(c, &m, base, rows, cols, box_rows);
    if (rc != SS_OK) return rc;
    it = c->xmaps.emplace(key, m).first;
  }
  *out = &it->second;
  return SS_OK;
}

// A projection split over all SMs, into fp32 partials.
int run_gemm(ss_ctx* c, const uint8_t* w_tiled, const CUtensorMap& mx, const GemmPlan& p, int n_tok) {
  GemmArgs a{};
  a.p = p;
  a.w_tiled = w_tiled;
  a.n_tok = n_tok;
  a.partial = c->partial;
  a.status = c->status;
  a.wait_limit = c->wait_limit;
  if ((size_t)p.gridx * p.max_seg * p.NT * 128 * sizeof(float) > c->partial_bytes) return SS_ERR_CAPACITY;
  // the weight tensor map is unused with tiled weights; the activation map stands in for it
  SS_CUDA(c, launch(c, gemm_wx_kernel, dim3(p.gridx), dim3(kGemmThreads), (size_t)p.smem_bytes, mx, mx, a));
  return SS_OK;
}

// The same product on pairs of CTAs (gemm_wx_pair_kernel): token tiles of up to 256, finished in the epilogue that `a` asks for.
GemmPlan plan_pair(int n_out, int K, int n_tok, int n_sm, size_t partial_bytes) {
  GemmPlan p{};
  p.n_out = n_out;
  p.K = K;
  p.n_tiles = 2 * ceil_div(n_out, kTileN);
  p.kb = ceil_div(K, kTileK);
  // equal token tiles in steps of the epilogue's 32
  p.tok_tiles = ceil_div(n_tok, kPairTokens);
  p.NT = round_up(ceil_div(n_tok, p.tok_tiles), 32);
  const int stage_bytes = kTileM * kTileK * 2 + p.NT * kTileK;
  p.stages = std::min(kGemmMaxStages, (227 * 1024 - 2048) / stage_bytes);
  p.smem_bytes = 2048 + p.stages * stage_bytes;
  // token tiles whose activations stay in L2 together
  const size_t tile_bytes = (size_t)p.NT * K * 2;
  const int fit = (int)std::max<size_t>(1, kPairGroupBytes / tile_bytes);
  p.group = ceil_div(p.tok_tiles, ceil_div(p.tok_tiles, fit));
  const int n_units = (p.n_tiles / 2) * p.tok_tiles, n_pairs = n_sm / 2;
  // Up to two token tiles the last round of pairs (all of o's and down's units at the 7B shape) is cut along K where that
  // shortens it.  It would last kb k-blocks and lasts kb * rest / n_pairs; a unit's owner then adds the n_pairs / rest - 1
  // parts that others have of it, about ten k-blocks' time each, and as much is lost on the way.  Whole calls of 258 and 510
  // tokens, always cut / never / by this line: d 1024, 4 layers, 508 / 408 / 408 and 629 / 449 / 449 us (eight units in nine
  // parts each); 32 x 64 heads 605 / 564 / 540 and 717 / 604 / 596; 7B shape 864 / 1004 / 864 and 1002 / 1070 / 998; 13B
  // shape, 2 layers, 1094 / 1205 / 1092 and 1308 / 1322 / 1308.  With more tiles the cut gains nothing (768 and 1024 tokens,
  // 1850 and 2400 us either way: the power cap gives what idle pairs leave to the others), and cutting one full round more
  // besides costs 5 to 13 % from 768 to 3200 tokens: pairs that are not at the same k-block share no weights.
  const int rest = n_units % n_pairs;
  p.split_units = p.tok_tiles <= 2 && (long long)p.kb * (n_pairs - rest) * rest > 10LL * n_pairs * n_pairs ? rest : 0;
  // (each of the ranges then has more than ten k-blocks)
  p.ranges = p.split_units ? (int)std::min<size_t>(n_pairs, partial_bytes / ((size_t)p.NT * 1024)) : 0;
  if (p.ranges < 1) p.split_units = 0;
  p.gridx = std::min(n_pairs, std::max(p.ranges, n_units - p.split_units));
  return p;
}
int run_gemm_pair(ss_ctx* c, const CUtensorMap& mw, const CUtensorMap& mx, const GemmPlan& p, GemmArgs a) {
  a.p = p;
  a.partial = c->partial;
  a.pair_flag = c->pair_flag;
  a.status = c->status;
  a.wait_limit = c->wait_limit;
  SS_CUDA(c, launch(c, gemm_wx_pair_kernel, dim3(2 * a.p.gridx), dim3(kPairThreads), (size_t)a.p.smem_bytes, mw, mx, a));
  return SS_OK;
}

struct ArenaPlan {
  size_t total = 0;
  size_t take(size_t bytes) {
    size_t off = total;
    total = align_up(total + bytes);
    return off;
  }
};

struct Offsets {
  size_t embed, lm_head, final_norm, staging, staging_bytes, weights_end;
  std::vector<size_t> attn_norm, wqkv, wo, ffn_norm, wgu, wdown;
  size_t inv_freq, rope, att_part, att_flag, pair_flag, status, rows, block_table, out_tokens, tok, h, x, qkv, attn_o, act;
  size_t h_dec, x_dec, o_dec, act_dec, partial, kv;
  size_t tbl[5], tbl_pair[5], tbl128[5], tile_val, tile_idx, rowss, grid_ctr, wptr, norm_ptr, trace;
  size_t partial_bytes, part_dec_base, part_dec_bytes, part_dec[5];
  int R, max_pages, n_pages;
  size_t total;
};

int validate_model(const ss_model_cfg* m, const ss_runtime_cfg* rt) {
  if (!m || !rt) return SS_ERR_ARG;
  if (m->n_layers < 0 || m->d_model <= 0 || m->n_heads <= 0 || m->d_ffn <= 0 || m->vocab <= 0) return SS_ERR_ARG;
  if (m->eos_id < 0 || m->eos_id >= m->vocab) return SS_ERR_ARG;
  if (m->n_heads * m->head_dim != m->d_model) return SS_ERR_ARG;
  if (m->head_dim != 64 && m->head_dim != 128) return SS_ERR_UNSUPPORTED;
  if (m->d_model % 64 || m->d_model > 8192 || m->d_ffn % 8) return SS_ERR_UNSUPPORTED;
  if (rt->max_batch < 1 || rt->max_batch > kMaxBatch) return SS_ERR_ARG;
  if (rt->max_ctx < 2 || rt->max_prefill_tokens < 1 || rt->max_new_tokens < 1 || rt->kv_pool_tokens < 1) return SS_ERR_ARG;
  return SS_OK;
}

void layout(const ss_model_cfg& m, const ss_runtime_cfg& rt, int n_sm, Offsets& o) {
  ArenaPlan a;
  const size_t d = m.d_model, F = m.d_ffn, V = m.vocab;
  o.embed = a.take(V * d * 2);
  o.attn_norm.resize(m.n_layers); o.wqkv.resize(m.n_layers); o.wo.resize(m.n_layers);
  o.ffn_norm.resize(m.n_layers); o.wgu.resize(m.n_layers); o.wdown.resize(m.n_layers);
  for (int l = 0; l < m.n_layers; ++l) {
    o.attn_norm[l] = a.take(d * 2);
    o.wqkv[l] = a.take(tiled_bytes(3 * d, d));
    o.wo[l] = a.take(tiled_bytes(d, d));
    o.ffn_norm[l] = a.take(d * 2);
    o.wgu[l] = a.take(tiled_bytes(2 * F, d));
    o.wdown[l] = a.take(tiled_bytes(d, F));
  }
  o.final_norm = a.take(d * 2);
  o.lm_head = a.take(tiled_bytes(V, d));
  o.weights_end = a.total;
  o.staging_bytes = std::max(std::max(V * d, F * d), d * d) * 2;
  o.staging = a.take(o.staging_bytes);
  o.inv_freq = a.take(m.head_dim / 2 * sizeof(float));
  o.rope = a.take((size_t)rt.max_ctx * (m.head_dim / 2) * sizeof(float2));
  o.att_part = a.take((size_t)n_sm * (m.head_dim + 4) * sizeof(float));
  o.att_flag = a.take((size_t)n_sm * 8);
  o.pair_flag = a.take((size_t)n_sm * 8 * sizeof(uint32_t));
  o.status = a.take(64);
  o.rows = a.take(kRowStateBytes + 64);
  o.max_pages = ceil_div(rt.max_ctx, kPageTokens);
  o.block_table = a.take((size_t)kMaxBatch * o.max_pages * 4);
  o.out_tokens = a.take((size_t)kMaxBatch * rt.max_new_tokens * 4);
  o.R = round_up(std::max(rt.max_prefill_tokens, kMaxBatch), 256);
  o.tok = a.take(((size_t)o.R * 3 + 2 * kMaxBatch + 8) * 4);
  o.h = a.take((size_t)o.R * d * 4);
  o.x = a.take((size_t)o.R * d * 2);
  o.qkv = a.take((size_t)o.R * 3 * d * 2);
  o.attn_o = a.take((size_t)o.R * d * 2);
  o.act = a.take((size_t)o.R * F * 2);
  o.h_dec = a.take((size_t)kMaxBatch * d * 4);
  o.x_dec = a.take((size_t)kMaxBatch * d * 2);
  o.o_dec = a.take((size_t)kMaxBatch * d * 2);
  o.act_dec = a.take((size_t)kMaxBatch * F * 2);
  // partial work space: the largest split projection at its widest token tile
  const int NTmax = round_up(rt.max_batch, 16);
  size_t pb = 0;
  const int shapes[5][2] = {{(int)(3 * d), (int)d}, {(int)d, (int)d}, {(int)(2 * F), (int)d}, {(int)d, (int)F}, {(int)V, (int)d}};
  for (int i = 0; i < 5; ++i) {
    for (int parts : {n_sm, n_sm / 2}) {
      const DecodeSplit p = plan_decode(shapes[i][0], shapes[i][1], parts);
      pb = std::max(pb, (size_t)p.gsplit * p.max_seg * NTmax * kTileN * sizeof(float));
    }
    // split prompt pass: the layers' projections over a short chunk, the LM head over the batch's rows
    const GemmPlan q = plan_gemm(shapes[i][0], shapes[i][1], i < 4 ? short_tile(rt.max_prefill_tokens) : NTmax, n_sm);
    pb = std::max(pb, (size_t)q.gridx * q.max_seg * q.NT * 128 * sizeof(float));
  }
  size_t pd = 0;
  for (int i = 0; i < 5; ++i) {
    const DecodeSplit p = plan_decode(shapes[i][0], shapes[i][1], n_sm);
    o.part_dec[i] = pd;
    pd += align_up((size_t)p.gsplit * p.max_seg * 16 * kTileN * sizeof(float));
  }
  o.part_dec_bytes = pd;
  o.part_dec_base = a.take(pd);
  o.partial_bytes = pb;
  o.partial = a.take(pb);
  o.rowss = a.take((size_t)kMaxBatch * kMaxSlices * 4);
  o.grid_ctr = a.take(64);
  o.wptr = a.take((size_t)(4 * m.n_layers + 1) * sizeof(void*));
  o.norm_ptr = a.take((size_t)(2 * m.n_layers + 1) * sizeof(void*));
  o.trace = a.take((size_t)(2 + 4 * (4 * m.n_layers + 1)) * 8);
  for (int i = 0; i < 5; ++i) o.tbl[i] = a.take((size_t)ceil_div(shapes[i][0], kTileN) * sizeof(TileSeg));
  for (int i = 0; i < 5; ++i) o.tbl_pair[i] = a.take((size_t)ceil_div(shapes[i][0], kTileN) * sizeof(TileSeg));
  for (int i = 0; i < 5; ++i) o.tbl128[i] = a.take((size_t)ceil_div(shapes[i][0], kTileM) * sizeof(TileSeg));
  o.tile_val = a.take((size_t)kMaxBatch * ceil_div((int)V, kTileM) * 4);
  o.tile_idx = a.take((size_t)kMaxBatch * ceil_div((int)V, kTileM) * 4);
  o.n_pages = (int)((rt.kv_pool_tokens + kPageTokens - 1) / kPageTokens) + rt.max_batch;
  const size_t page_bytes = (size_t)2 * m.n_heads * kPageTokens * m.head_dim * 2;
  o.kv = a.take((size_t)std::max(1, m.n_layers) * o.n_pages * page_bytes);
  o.total = a.total;
}

// SMs of the current device; 148 (a B200) when no device can be asked, e.g. when sizing an arena on a host
// without a GPU.
int query_sms() {
  int dev = 0, n = 148;
  if (cudaGetDevice(&dev) == cudaSuccess) {
    int v = 0;
    if (cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess && v > 0) n = v;
  }
  return n;
}

struct WeightSlot {
  void* dst;          // plain tensors: destination; tiled: base of the tiled matrix
  int64_t rows, cols; // expected shape of the source
  int slot;
  bool tiled;
  int row_off;        // tiled: row offset inside the stacked matrix
  int half, step;     // tiled: placement of the rows (repack_weights_kernel)
};

int weight_slot(const ss_ctx* c, const std::string& name, WeightSlot* out) {
  const int64_t d = c->m.d_model, F = c->m.d_ffn, V = c->m.vocab;
  auto plain = [&](void* p, int64_t r, int64_t cc, int s) { *out = {p, r, cc, s, false, 0, 0, 1}; return SS_OK; };
  auto tiled = [&](void* p, int64_t r, int64_t cc, int s, int64_t off, int half = 0, int step = 1) {
    *out = {p, r, cc, s, true, (int)off, half, step};
    return SS_OK;
  };
  const int rot = c->m.head_dim / 2;      // the two dimensions of a rotation become neighbouring rows
  if (name == "embed") return plain(c->embed, V, d, 0);
  if (name == "lm_head") return tiled(c->lm_head, V, d, 1, 0);
  if (name == "final_norm") return plain(c->final_norm, 1, d, 2);
  if (name.size() > 2 && name[0] == 'l') {
    size_t dot = name.find('.');
    if (dot == std::string::npos) return SS_ERR_ARG;
    int l = atoi(name.substr(1, dot - 1).c_str());
    if (l < 0 || l >= c->m.n_layers) return SS_ERR_ARG;
    const std::string k = name.substr(dot + 1);
    const LayerWeights& w = c->layers[l];
    const int base = 3 + l * 9;
    if (k == "attn_norm") return plain(w.attn_norm, 1, d, base + 0);
    if (k == "wq") return tiled(w.wqkv, d, d, base + 1, 0, rot);
    if (k == "wk") return tiled(w.wqkv, d, d, base + 2, d, rot);
    if (k == "wv") return tiled(w.wqkv, d, d, base + 3, 2 * d);
    if (k == "wo") return tiled(w.wo, d, d, base + 4, 0);
    if (k == "ffn_norm") return plain(w.ffn_norm, 1, d, base + 5);
    if (k == "w_gate") return tiled(w.wgu, F, d, base + 6, 0, 0, 2);
    if (k == "w_up") return tiled(w.wgu, F, d, base + 7, 1, 0, 2);
    if (k == "w_down") return tiled(w.wdown, d, F, base + 8, 0);
  }
  return SS_ERR_ARG;
}

// Grid-barrier counter, attention flags (which hold barrier numbers) and flags of waiting partials back to zero, and no
// partial sum in any slot of the decode step.
void reset_grid(ss_ctx* c) {
  cudaMemsetAsync(c->part_dec[0], 0xff, c->part_dec_bytes, c->stream);
  cudaMemsetAsync(c->pair_flag, 0, (size_t)c->n_sm * 8 * sizeof(uint32_t), c->stream);
  cudaMemsetAsync(c->grid_ctr, 0, 8, c->stream);
  cudaMemsetAsync(c->att_flag, 0, (size_t)c->n_sm * 8, c->stream);
  cudaStreamSynchronize(c->stream);
  c->grid_epochs = 0;
}

// A non-zero status word: the step that set it was abandoned half way.  The error is reported once; the word
// and the grid-barrier counter (left in an unknown state by the abort) are cleared so that the context can
// start a new batch.
int report_device_status(ss_ctx* c, uint32_t word) {
  cudaMemsetAsync(c->status, 0, 4, c->stream);
  reset_grid(c);
  return word == (uint32_t)kStatusBadPage ? SS_ERR_STATE : SS_ERR_DEVICE_TIMEOUT;
}

double weight_bytes_per_step(const ss_model_cfg& m) {
  const double d = m.d_model, F = m.d_ffn, V = m.vocab;
  return m.n_layers * (4 * d * d + 3 * d * F + 2 * d) * 2.0 + V * d * 2.0 + d * 2.0;
}
double kv_bytes_per_token(const ss_model_cfg& m) { return 2.0 * m.d_model * 2.0 * m.n_layers; }

// The decode kernel's instantiations: head size 64 / 128, batches up to 16 / 64 / 128 / 256 rows, without / with the stage trace.
const void* mega_kernel_fn(int head_dim, int rows, bool trace) {
  return head_dim == 128 ? mega_kernel_128(rows, trace) : mega_kernel_64(rows, trace);
}
// Loads the instantiations that a context can launch: those of its head size, and the ones with the trace when a trace is
// asked for.
cudaError_t prepare_mega_kernels(int head_dim, bool trace) {
  cudaError_t e = cudaSuccess;
  for (int rows : {16, 64, 128, 256})
    if (e == cudaSuccess) e = cudaFuncSetAttribute(mega_kernel_fn(head_dim, rows, trace), cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
  return e;
}

// ------------------------------------------------------------------------------------ decode step
// One cooperative launch of the persistent kernel (see ss_decode_mega.cuh).
int enqueue_decode_step(ss_ctx* c, const ss_step_opts* opts, int32_t* next_tokens) {
  const ss_model_cfg& m = c->m;
  const int B = c->B, d = m.d_model, F = m.d_ffn, V = m.vocab;
  const int NT = round_up(B, 16);
  const CUtensorMap *mx, *mo, *ma;
  int rc;
  // 65 to 128 rows fit the lanes of one CTA.  Where a CTA streams many blocks per layer that is the better form, since a
  // pair's MMAs (two CTAs, 32 KiB of weights) pace the stream; where it streams few, the drains weigh more and pairs have
  // half of the segments.  72 / 112 / 128 rows, one CTA and pairs, us a step of 4 layers: 7B shape (83 blocks) 570 / - / 792
  // and 650 / - / 830; d 3072 (47) 416 / 578 / 562 and 432 / 570 / 548; d 2560 (33) 383 / 513 / 522 and 371 / 470 / 456; 32 x
  // 64 heads (21) 331 / 450 / 456 and 316 / 400 / 398.  (The line goes by the blocks alone: between 40 and 50 of them pairs are
  // 1 to 3 % ahead from 112 rows on and 4 % behind at 72.)  Up to 64 rows one CTA: 48 rows of 32 x 64 heads 290 and 306.
  const double layer_blocks = (4.0 * d * d + 3.0 * d * F) * 2 / kBlockBytes / c->n_sm;
  const int kernel_rows = NT <= 16 ? 16 : NT <= 64 ? 64 : (NT <= 128 && layer_blocks > 40) ? 128 : 256;
  const bool pair = kernel_rows == 256, flagged = kernel_rows == 16;
  const int xr = pair ? round_up(ceil_div(B, 2), 8) : NT;      // activation rows per TMA load (in steps of the swizzle's 8)
  if ((rc = xmap(c, 3, xr, &mx)) || (rc = xmap(c, 4, xr, &mo)) || (rc = xmap(c, 5, xr, &ma))) return rc;
  MegaArgs a{};
  a.n_layers = m.n_layers; a.d = d; a.H = m.n_heads; a.Dh = m.head_dim; a.F = F; a.V = V; a.eos_id = m.eos_id;
  a.eps = m.rms_eps;
  a.wptr = c->wptr_dev;
  a.norm_ptr = c->norm_dev;
  a.embed = c->embed;
  a.rope = c->rope;
  const int shp[5][2] = {{3 * d, d}, {d, d}, {2 * F, d}, {d, F}, {V, d}};
  size_t need_partial = 0;
  int tab_entries = 0;
  for (int i = 0; i < 4; ++i) tab_entries += ceil_div(shp[i][0], kTileN);
  int tab_off = 0;
  for (int i = 0; i < 5; ++i) {
    const DecodeSplit p = plan_decode(shp[i][0], shp[i][1], pair ? c->n_sm / 2 : c->n_sm);
    const int off = (i < 4 && tab_entries <= kSegTabEntries) ? tab_off : -1;   // the per-layer tables, if they fit
    tab_off += p.n_tiles;
    a.shape[i] = {p.n_tiles, p.kb, p.max_seg, p.gsplit, p.total, pair ? c->tbl_pair[i] : c->tbl[i], flagged ? c->part_dec[i] : c->partial, off};
    need_partial = std::max(need_partial, (size_t)p.gsplit * p.max_seg * NT * kTileN * sizeof(float));
  }
  if (!flagged && need_partial > c->partial_bytes) return SS_ERR_CAPACITY;
  a.B = B; a.NT = NT;
  a.x_rows = xr;
  a.wbase = c->arena;
  const int stage_bytes = (pair ? kBlockBytes / 2 : kBlockBytes) + xr * kTileK * 2;
  // shared memory left behind the header is shared out between the weight ring and the pieces of the cache scan
  const int header = (int)sizeof(MegaSmem) + mega_scratch_bytes(kernel_rows > 64) + 1024, piece_set = 8 * kKvPieceBytes;
  const int room = 227 * 1024 - header;
  a.stages = std::max(2, std::min(kMegaMaxStages, (room - 2 * piece_set) / stage_bytes));
  a.kv_pieces = std::min(kKvMaxPieces, (room - a.stages * stage_bytes) / piece_set);
  const size_t smem = (size_t)header + (size_t)a.stages * stage_bytes + (size_t)a.kv_pieces * piece_set;
  a.att_part = c->att_part;
  a.att_flag = c->att_flag;
  a.st = c->st; a.kv = c->kv;
  a.h = c->h_dec; a.x = c->x_dec; a.o = c->o_dec; a.act = c->act_dec;
  a.rowss = c->rowss;
  a.tile_val = c->tile_val; a.tile_idx = c->tile_idx; a.n_tiles_lm = c->n_tiles_lm;
  a.forced = opts ? opts->forced_tokens : nullptr;
  a.next_tokens = next_tokens;
  a.dump_logits = opts ? opts->dump_logits : nullptr;
  a.dump_hidden = opts ? opts->dump_hidden : nullptr;
  a.dump_choice = opts ? opts->dump_choice : nullptr;
  a.sample = c->sample;
  a.grid_ctr = c->grid_ctr;
  a.grid_base = c->grid_epochs * (unsigned long long)c->n_sm;
  a.status = c->status;
  a.trace = c->trace_on ? c->trace : nullptr;
  a.wait_limit = c->wait_limit;
  void* args[5] = {(void*)mx, (void*)mo, (void*)ma, (void*)&c->wmap_all, (void*)&a};
  const void* fn = mega_kernel_fn(m.head_dim, kernel_rows, a.trace != nullptr);
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(c->n_sm);
  cfg.blockDim = dim3(kMegaThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = c->stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = 2;
  attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pair ? 2 : 1;
  SS_CUDA(c, cudaLaunchKernelExC(&cfg, fn, args));
  c->grid_epochs += 1 + (flagged ? 1 : 2) * (unsigned long long)(4 * m.n_layers + 1);
  c->launches++;
  return SS_OK;
}

// ------------------------------------------------------------------------------------ prompt pass (one chunk of whole sequences)
int enqueue_prefill_chunk(ss_ctx* c, int s0, int s1, const int32_t* cu, int T) {
  const ss_model_cfg& m = c->m;
  const int d = m.d_model, F = m.d_ffn, H = m.n_heads, Dh = m.head_dim, V = m.vocab;
  const int nseq = s1 - s0;
  int max_len = 0;
  for (int s = s0; s < s1; ++s) max_len = std::max(max_len, cu[s + 1] - cu[s]);
  const CUtensorMap *mx, *mo, *ma, *mq;
  int rc;
  if ((rc = xmap(c, 6, kAttnTile, &mq))) return rc;
  // what the q,k,v projection does behind the sum, whichever kernel does it
  GemmArgs qkv{};
  qkv.mode = kGemmQkv;
  qkv.n_tok = T;
  qkv.out = c->qkv;
  qkv.d = d; qkv.H = H; qkv.Dh = Dh;
  qkv.rope = c->rope;
  qkv.tok_pos = c->d_tok_pos;
  qkv.tok_slot = c->d_tok_slot;
  qkv.page_elems = c->kv.page_elems;
  GemmArgs res{}, glu{};
  res.mode = kGemmResidual;
  res.n_tok = T;
  res.residual = c->h;
  glu.mode = kGemmSwiglu;
  glu.n_tok = T;
  glu.out = c->act;
  // more than one token tile of a pair: the paired kernel; up to it, the projections are split over the SMs along K too
  const bool pair = T > kShortTokens;
  const int shp[4][2] = {{3 * d, d}, {d, d}, {2 * F, d}, {d, F}};
  GemmPlan plan[4];
  SplitInfo split[4];
  for (int i = 0; i < 4; ++i) {
    if (pair) { plan[i] = plan_pair(shp[i][0], shp[i][1], T, c->n_sm, c->partial_bytes); continue; }
    plan[i] = plan_gemm(shp[i][0], shp[i][1], short_tile(T), c->n_sm);
    split[i] = split_of(plan[i], c->tbl128[i]);
  }
  const int NT = pair ? plan[0].NT / 2 : plan[0].NT;
  if ((rc = xmap(c, 0, NT, &mx)) || (rc = xmap(c, 1, NT, &mo)) || (rc = xmap(c, 2, NT, &ma))) return rc;
  auto attend = [&]() -> int {
    const dim3 ag(ceil_div(max_len, kAttnTile), H, nseq);
    if (Dh == 128)
      SS_CUDA(c, launch(c, attn_prefill_kernel<128>, ag, dim3(128), (size_t)attn_prefill_smem<128>(), *mq, (const int32_t*)c->d_cu, c->attn_o, d, c->status, c->wait_limit));
    else
      SS_CUDA(c, launch(c, attn_prefill_kernel<64>, ag, dim3(128), (size_t)attn_prefill_smem<64>(), *mq, (const int32_t*)c->d_cu, c->attn_o, d, c->status, c->wait_limit));
    return SS_OK;
  };
  const bf16* first_norm = m.n_layers ? c->layers[0].attn_norm : c->final_norm;
  SS_CUDA(c, launch(c, embed_rmsnorm_kernel, dim3(T), dim3(256), 0, (const int32_t*)c->d_tokens,
                    (const bf16*)c->embed, first_norm, c->h, c->x, d, m.rms_eps, V));
  for (int l = 0; l < m.n_layers; ++l) {
    const LayerWeights& w = c->layers[l];
    const bf16* next_norm = l + 1 < m.n_layers ? c->layers[l + 1].attn_norm : c->final_norm;
    qkv.kv_layer = c->kv.pool + (size_t)l * c->kv.layer_stride;
    if (pair) {
      if ((rc = run_gemm_pair(c, c->wmaps[4 * l + 0], *mx, plan[0], qkv)) || (rc = attend()) ||
          (rc = run_gemm_pair(c, c->wmaps[4 * l + 1], *mo, plan[1], res))) return rc;
      SS_CUDA(c, launch(c, rmsnorm_kernel, dim3(T), dim3(256), 0, (const float*)c->h, (const bf16*)w.ffn_norm, c->x, d, m.rms_eps));
      if ((rc = run_gemm_pair(c, c->wmaps[4 * l + 2], *mx, plan[2], glu)) ||
          (rc = run_gemm_pair(c, c->wmaps[4 * l + 3], *ma, plan[3], res))) return rc;
      if (l + 1 < m.n_layers)
        SS_CUDA(c, launch(c, rmsnorm_kernel, dim3(T), dim3(256), 0, (const float*)c->h, next_norm, c->x, d, m.rms_eps));
    } else {
      const float* part = c->partial;
      if ((rc = run_gemm(c, w.wqkv, *mx, plan[0], T))) return rc;
      SS_CUDA(c, launch(c, short_qkv_kernel, dim3(T, ceil_div(3 * d, 1024)), dim3(256), 0, part, split[0], qkv));
      if ((rc = attend()) || (rc = run_gemm(c, w.wo, *mo, plan[1], T))) return rc;
      SS_CUDA(c, launch(c, short_residual_kernel, dim3(T), dim3(1024), 0, part, split[1], c->h, (const bf16*)w.ffn_norm, c->x, d, m.rms_eps));
      if ((rc = run_gemm(c, w.wgu, *mx, plan[2], T))) return rc;
      SS_CUDA(c, launch(c, short_swiglu_kernel, dim3(T, ceil_div(2 * F, 1024)), dim3(256), 0, part, split[2], c->act, F));
      if ((rc = run_gemm(c, w.wdown, *ma, plan[3], T))) return rc;
      SS_CUDA(c, launch(c, short_residual_kernel, dim3(T), dim3(1024), 0, part, split[3], c->h, next_norm, c->x, d, m.rms_eps));
    }
  }
  return SS_OK;
}

// ------------------------------------------------------------------------------------ staging
// Copies n bytes out of the staging area.
cudaError_t send_up(ss_ctx* c, void* dst, const void* src, size_t n) {
  const cudaError_t e = cudaMemcpyAsync(dst, src, n, cudaMemcpyHostToDevice, c->stream);
  const cudaError_t r = cudaEventRecord(c->up_sent, c->stream);
  if (r != cudaSuccess) cudaStreamSynchronize(c->stream);
  return e != cudaSuccess ? e : r;
}
// The staging area may be filled again: every copy out of it has run.
cudaError_t wait_up(ss_ctx* c) { return cudaEventSynchronize(c->up_sent); }

// Sends the row state and the block tables of B rows, filled in at c->up (row arrays first, tables at table_off).
cudaError_t send_rows(ss_ctx* c, int B) {
  return send_up(c, c->st.ctx_len, c->up.data(), c->table_off + (size_t)B * c->st.max_pages * 4);
}

// Row state and block table of a new batch of B rows in the staging area: everything zero, no pages.
void clear_rows(ss_ctx* c, int B, int cap, int32_t** rows, int32_t** bt) {
  *rows = (int32_t*)c->up.data();
  *bt = (int32_t*)(c->up.data() + c->table_off);
  std::memset(*rows, 0, kRowStateBytes);
  std::fill(*bt, *bt + (size_t)B * c->st.max_pages, -1);
  (*rows)[7 * kMaxBatch + 0] = cap;
  (*rows)[7 * kMaxBatch + 1] = B;
}

}  // namespace

// ======================================================================================= C ABI
extern "C" {

const char* ss_strerror(int code) {
  switch (code) {
    case SS_OK: return "ok";
    case SS_ERR_ARG: return "bad argument";
    case SS_ERR_CAPACITY: return "buffer or arena too small";
    case SS_ERR_KV_BUDGET: return "batch does not fit the key/value pool";
    case SS_ERR_STATE: return "call out of order";
    case SS_ERR_CUDA: return "CUDA call failed";
    case SS_ERR_DEVICE_TIMEOUT: return "a bounded wait inside a kernel expired";
    case SS_ERR_UNSUPPORTED: return "shape not supported by the kernels";
    default: return "unknown error";
  }
}

int ss_arena_bytes(const ss_model_cfg* model, const ss_runtime_cfg* rt, size_t* out_bytes) {
  int rc = validate_model(model, rt);
  if (rc) return rc;
  if (!out_bytes) return SS_ERR_ARG;
  Offsets o;
  layout(*model, *rt, query_sms(), o);  // the split tables and partial sums are sized by the SM count
  *out_bytes = o.total;
  return SS_OK;
}

int ss_create(const ss_model_cfg* model, const ss_runtime_cfg* rt, void* dev_arena, size_t arena_bytes, void* stream,
              ss_ctx** out) {
  int rc = validate_model(model, rt);
  if (rc) return rc;
  if (!dev_arena || !out || ((uintptr_t)dev_arena % kAlign)) return SS_ERR_ARG;
  int ndev = 0;
  if (cudaGetDeviceCount(&ndev) != cudaSuccess || ndev == 0) return SS_ERR_CUDA;
  Offsets o;
  const int n_sm = query_sms();
  layout(*model, *rt, n_sm, o);
  if (arena_bytes < o.total) return SS_ERR_CAPACITY;
  ss_ctx* c = new ss_ctx();
  c->m = *model;
  c->rt = *rt;
  c->stream = (cudaStream_t)stream;
  c->n_sm = n_sm;
  {
    int dev = 0, khz = 0;
    if (cudaGetDevice(&dev) == cudaSuccess && cudaDeviceGetAttribute(&khz, cudaDevAttrClockRate, dev) == cudaSuccess && khz > 0)
      c->clock_khz = khz;
  }
  void* fn = nullptr;
  cudaDriverEntryPointQueryResult qr;
  if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &qr) != cudaSuccess || !fn) {
    delete c;
    return SS_ERR_CUDA;
  }
  c->encode = (EncodeTiledFn)fn;
  uint8_t* A = (uint8_t*)dev_arena;
  c->arena = A;
  c->arena_bytes = arena_bytes;
  const int64_t d = model->d_model, F = model->d_ffn, V = model->vocab;
  c->embed = (bf16*)(A + o.embed);
  c->lm_head = A + o.lm_head;
  c->staging = A + o.staging;
  c->staging_bytes = o.staging_bytes;
  c->final_norm = (bf16*)(A + o.final_norm);
  c->layers.resize(model->n_layers);
  auto fail = [&](int code) { delete c; return code; };
  for (int l = 0; l < model->n_layers; ++l) {
    LayerWeights& w = c->layers[l];
    w.attn_norm = (bf16*)(A + o.attn_norm[l]);
    w.wqkv = A + o.wqkv[l];
    w.wo = A + o.wo[l];
    w.ffn_norm = (bf16*)(A + o.ffn_norm[l]);
    w.wgu = A + o.wgu[l];
    w.wdown = A + o.wdown[l];
  }
  // tiles that reach beyond a matrix's rows or columns must read as zero
  if (cudaMemsetAsync(A + o.embed, 0, o.weights_end - o.embed, c->stream) != cudaSuccess) return fail(SS_ERR_CUDA);
  c->n_expected = 3 + 9 * model->n_layers;
  c->loaded.assign(c->n_expected, 0);
  c->inv_freq = (float*)(A + o.inv_freq);
  c->rope = (float2*)(A + o.rope);
  c->att_part = (float*)(A + o.att_part);
  c->att_flag = (unsigned long long*)(A + o.att_flag);
  c->pair_flag = (uint32_t*)(A + o.pair_flag);
  c->status = (uint32_t*)(A + o.status);
  int32_t* rows = (int32_t*)(A + o.rows);
  c->st.ctx_len = rows + 0 * kMaxBatch;
  c->st.cur_tok = rows + 1 * kMaxBatch;
  c->st.gen = rows + 2 * kMaxBatch;
  c->st.active = rows + 3 * kMaxBatch;
  c->st.finished = rows + 4 * kMaxBatch;
  c->st.eos_at = rows + 5 * kMaxBatch;
  c->st.row_key = rows + 6 * kMaxBatch;
  c->st.scalars = rows + 7 * kMaxBatch;
  c->st.block_table = (int32_t*)(A + o.block_table);
  c->st.out_tokens = (int32_t*)(A + o.out_tokens);
  c->st.max_pages = o.max_pages;
  c->st.max_new = rt->max_new_tokens;
  c->R = o.R;
  c->d_chunk = (int32_t*)(A + o.tok);
  c->table_off = o.block_table - o.rows;
  c->h = (float*)(A + o.h);
  c->x = (bf16*)(A + o.x);
  c->qkv = (bf16*)(A + o.qkv);
  c->attn_o = (bf16*)(A + o.attn_o);
  c->act = (bf16*)(A + o.act);
  c->h_dec = (float*)(A + o.h_dec);
  c->x_dec = (bf16*)(A + o.x_dec);
  c->o_dec = (bf16*)(A + o.o_dec);
  c->act_dec = (bf16*)(A + o.act_dec);
  c->partial = (float*)(A + o.partial);
  c->partial_bytes = o.partial_bytes;
  for (int i = 0; i < 5; ++i) c->part_dec[i] = (float*)(A + o.part_dec_base + o.part_dec[i]);
  c->part_dec_bytes = o.part_dec_bytes;
  c->rowss = (float*)(A + o.rowss);
  c->grid_ctr = (unsigned long long*)(A + o.grid_ctr);
  c->wptr_dev = (const uint8_t**)(A + o.wptr);
  c->trace = (unsigned long long*)(A + o.trace);
  c->trace_len = 2 + 4 * (4 * model->n_layers + 1);
  c->norm_dev = (const bf16**)(A + o.norm_ptr);
  {
    std::vector<const uint8_t*> wp;
    std::vector<const bf16*> np;
    for (int l = 0; l < model->n_layers; ++l) {
      const LayerWeights& w = c->layers[l];
      wp.push_back(w.wqkv); wp.push_back(w.wo); wp.push_back(w.wgu); wp.push_back(w.wdown);
      np.push_back(w.attn_norm); np.push_back(w.ffn_norm);
    }
    wp.push_back(c->lm_head);
    np.push_back(c->final_norm);
    if (cudaMemcpy(c->wptr_dev, wp.data(), wp.size() * sizeof(void*), cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemcpy(c->norm_dev, np.data(), np.size() * sizeof(void*), cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemset(A + o.rowss, 0, o.wptr - o.rowss) != cudaSuccess)
      return fail(SS_ERR_CUDA);
  }
  c->wmaps.resize((size_t)4 * model->n_layers);
  for (int l = 0; l < model->n_layers; ++l) {
    const LayerWeights& w = c->layers[l];
    const uint8_t* base[4] = {w.wqkv, w.wo, w.wgu, w.wdown};
    const size_t bytes[4] = {tiled_bytes(3 * d, d), tiled_bytes(d, d), tiled_bytes(2 * F, d), tiled_bytes(d, F)};
    for (int t = 0; t < 4; ++t)
      if (int rc2 = make_line_map(c, &c->wmaps[4 * l + t], base[t], bytes[t])) return fail(rc2);
  }
  if (int rc2 = make_line_map(c, &c->wmap_all, A, o.weights_end)) return fail(rc2);
  c->tile_val = (float*)(A + o.tile_val);
  c->tile_idx = (int32_t*)(A + o.tile_idx);
  c->n_tiles_lm = ceil_div((int)V, kTileM);
  {
    const int shp[5][2] = {{(int)(3 * d), (int)d}, {(int)d, (int)d}, {(int)(2 * F), (int)d}, {(int)d, (int)F}, {(int)V, (int)d}};
    for (int i = 0; i < 5; ++i) {
      c->tbl[i] = (TileSeg*)(A + o.tbl[i]);
      c->tbl_pair[i] = (TileSeg*)(A + o.tbl_pair[i]);
      for (int pairs = 0; pairs < 2; ++pairs) {
        const std::vector<TileSeg> t = decode_tile_table(plan_decode(shp[i][0], shp[i][1], pairs ? c->n_sm / 2 : c->n_sm));
        if (cudaMemcpy(pairs ? c->tbl_pair[i] : c->tbl[i], t.data(), t.size() * sizeof(TileSeg), cudaMemcpyHostToDevice) != cudaSuccess)
          return fail(SS_ERR_CUDA);
      }
    }
    for (int i = 0; i < 5; ++i) {
      c->tbl128[i] = (TileSeg*)(A + o.tbl128[i]);
      const std::vector<TileSeg> t = tile_table(plan_gemm(shp[i][0], shp[i][1], 16, c->n_sm));
      if (cudaMemcpy(c->tbl128[i], t.data(), t.size() * sizeof(TileSeg), cudaMemcpyHostToDevice) != cudaSuccess)
        return fail(SS_ERR_CUDA);
    }
  }
  c->kv.pool = (bf16*)(A + o.kv);
  c->kv.page_elems = (size_t)2 * model->n_heads * kPageTokens * model->head_dim;
  c->kv.layer_stride = (size_t)o.n_pages * c->kv.page_elems;
  c->kv.n_pages = o.n_pages;
  c->kv.H = model->n_heads;
  c->kv.Dh = model->head_dim;
  c->free_pages.resize(o.n_pages);
  for (int i = 0; i < o.n_pages; ++i) c->free_pages[i] = o.n_pages - 1 - i;

  // rotary inverse frequencies, exact in double then rounded once
  std::vector<float> inv(model->head_dim / 2);
  for (int i = 0; i < model->head_dim / 2; ++i)
    inv[i] = (float)std::pow((double)model->rope_theta, -2.0 * i / model->head_dim);
  cudaError_t e = cudaMemcpyAsync(c->inv_freq, inv.data(), inv.size() * 4, cudaMemcpyHostToDevice, c->stream);
  if (e == cudaSuccess) {
    rope_table_kernel<<<(unsigned)rt->max_ctx, model->head_dim / 2, 0, c->stream>>>(c->inv_freq, c->rope);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaMemsetAsync(c->att_flag, 0, (size_t)n_sm * 8, c->stream);
  if (e == cudaSuccess) e = cudaMemsetAsync(c->pair_flag, 0, (size_t)n_sm * 8 * sizeof(uint32_t), c->stream);
  if (e == cudaSuccess) e = cudaMemsetAsync(c->status, 0, 64, c->stream);
  if (e == cudaSuccess) e = cudaMemsetAsync(rows, 0, kRowStateBytes + 64, c->stream);
  // activation operands must be finite wherever a TMA box may reach beyond the valid rows
  if (e == cudaSuccess) e = cudaMemsetAsync(A + o.h, 0, o.partial - o.h, c->stream);
  if (e == cudaSuccess) e = cudaMemsetAsync(c->part_dec[0], 0xff, c->part_dec_bytes, c->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(c->stream);
  if (e == cudaSuccess) e = cudaHostAlloc((void**)&c->pinned, 64, cudaHostAllocDefault);
  if (e == cudaSuccess) e = cudaEventCreateWithFlags(&c->up_sent, cudaEventDisableTiming);
  if (e == cudaSuccess) e = cudaEventCreateWithFlags(&c->layers_done, cudaEventDisableTiming);
  c->up_chunk = align_up(c->table_off + (size_t)rt->max_batch * o.max_pages * 4);
  try {
    c->up.resize(c->up_chunk + ((size_t)o.R * 3 + 2 * kMaxBatch + 8) * 4);
    c->down_rows.resize(kRowStateBytes / 4);
  } catch (const std::bad_alloc&) {
    e = cudaErrorMemoryAllocation;
  }
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(gemm_wx_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(gemm_wx_pair_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(attn_prefill_kernel<128>, cudaFuncAttributeMaxDynamicSharedMemorySize, attn_prefill_smem<128>());
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(attn_prefill_kernel<64>, cudaFuncAttributeMaxDynamicSharedMemorySize, attn_prefill_smem<64>());
  if (e == cudaSuccess) e = prepare_mega_kernels(model->head_dim, false);
  if (e != cudaSuccess) {
    if (c->pinned) cudaFreeHost(c->pinned);
    if (c->up_sent) cudaEventDestroy(c->up_sent);
    if (c->layers_done) cudaEventDestroy(c->layers_done);
    delete c;
    return SS_ERR_CUDA;
  }
  *out = c;
  return SS_OK;
}

int ss_destroy(ss_ctx* c) {
  if (!c) return SS_ERR_ARG;
  cudaStreamSynchronize(c->stream);
  if (c->pinned) cudaFreeHost(c->pinned);
  cudaEventDestroy(c->up_sent);
  cudaEventDestroy(c->layers_done);
  delete c;
  return SS_OK;
}

int ss_load_weights(ss_ctx* c, const ss_tensor_desc* t, int32_t n) {
  if (!c || (n > 0 && !t) || n < 0) return SS_ERR_ARG;
  for (int i = 0; i < n; ++i) {
    if (!t[i].name || !t[i].data) return SS_ERR_ARG;
    WeightSlot ws;
    int rc = weight_slot(c, t[i].name, &ws);
    if (rc) return rc;
    if (t[i].rows * t[i].cols != ws.rows * ws.cols || (ws.rows > 1 && (t[i].rows != ws.rows || t[i].cols != ws.cols)))
      return SS_ERR_ARG;
    const size_t bytes = (size_t)ws.rows * ws.cols * 2;
    if (!ws.tiled) {
      SS_CUDA(c, cudaMemcpyAsync(ws.dst, t[i].data, bytes,
                                 t[i].is_device ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice, c->stream));
    } else {
      const void* src = t[i].data;
      if (!t[i].is_device || ((uintptr_t)src & 15)) {
        if (bytes > c->staging_bytes) return SS_ERR_CAPACITY;
        SS_CUDA(c, cudaMemcpyAsync(c->staging, src, bytes,
                                   t[i].is_device ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice, c->stream));
        src = c->staging;
      }
      const long long chunks = (long long)ws.rows * (ws.cols / 8);
      repack_weights_kernel<<<(unsigned)((chunks + 255) / 256), 256, 0, c->stream>>>(
          (const uint4*)src, ws.rows, (int)ws.cols, (uint8_t*)ws.dst, ws.row_off, ceil_div((int)ws.cols, kTileK), ws.half, ws.step);
      SS_CUDA(c, cudaGetLastError());
      c->launches++;
      // the staging buffer (or the caller's tensor) is free again once the repack has run
      SS_CUDA(c, cudaStreamSynchronize(c->stream));
    }
    if (!c->loaded[ws.slot]) { c->loaded[ws.slot] = 1; c->n_loaded++; }
  }
  SS_CUDA(c, cudaStreamSynchronize(c->stream));
  return SS_OK;
}

int ss_release_batch(ss_ctx* c) {
  if (!c) return SS_ERR_ARG;
  for (int32_t p : c->batch_pages) c->free_pages.push_back(p);
  c->batch_pages.clear();
  c->row_pages.clear();
  c->in_batch = false;
  c->B = 0;
  return SS_OK;
}

}  // extern "C"

// ss_prefill() without the wait at its end.
static int start_batch(ss_ctx* c, const int32_t* tokens, const int32_t* cu, int32_t B, const int32_t* eos_at, int32_t cap,
                       const ss_step_opts* opts, int32_t* first_tokens) {
  if (!c || !tokens || !cu || B < 1 || cap < 1) return SS_ERR_ARG;
  if (c->n_loaded != c->n_expected || c->in_batch) return SS_ERR_STATE;
  if (B > c->rt.max_batch || cap > c->rt.max_new_tokens) return SS_ERR_CAPACITY;
  if (cu[0] != 0) return SS_ERR_ARG;
  const ss_model_cfg& m = c->m;
  // admission: pages for the worst case of every row
  size_t need_pages = 0;
  for (int r = 0; r < B; ++r) {
    const int len = cu[r + 1] - cu[r];
    if (len < 1) return SS_ERR_ARG;
    if (len > c->rt.max_prefill_tokens || len + cap > c->rt.max_ctx) return SS_ERR_CAPACITY;
    need_pages += ceil_div(len + cap, kPageTokens);
    if (eos_at && eos_at[r] < 1) return SS_ERR_ARG;
  }
  if (need_pages > c->free_pages.size()) return SS_ERR_KV_BUDGET;
  const int Ttot = cu[B];
  for (int i = 0; i < Ttot; ++i)
    if (tokens[i] < 0 || tokens[i] >= m.vocab) return SS_ERR_ARG;

  // host-side batch state
  int32_t *rows, *bt;
  SS_CUDA(c, wait_up(c));
  clear_rows(c, B, cap, &rows, &bt);
  c->batch_pages.clear();
  c->prompt_len.assign(B, 0);
  c->row_pages.assign(B, {});
  c->batch_tokens.assign(tokens, tokens + Ttot);
  c->batch_cu.assign(cu, cu + B + 1);
  for (int r = 0; r < B; ++r) {
    const int len = cu[r + 1] - cu[r];
    c->prompt_len[r] = len;
    const int np = ceil_div(len + cap, kPageTokens);
    for (int p = 0; p < np; ++p) {
      const int32_t pg = c->free_pages.back();
      c->free_pages.pop_back();
      c->batch_pages.push_back(pg);
      c->row_pages[r].push_back(pg);
      bt[(size_t)r * c->st.max_pages + p] = pg;
    }
  }
  c->in_batch = true;
  c->B = B;
  c->cap = cap;
  for (int r = 0; r < B; ++r) {
    rows[0 * kMaxBatch + r] = c->prompt_len[r];   // ctx_len after the prompt pass
    rows[3 * kMaxBatch + r] = 1;                  // active
    rows[5 * kMaxBatch + r] = eos_at ? eos_at[r] : 0;
    rows[6 * kMaxBatch + r] = r < (int)c->next_row_keys.size() ? c->next_row_keys[r] : r;
  }
  c->next_row_keys.clear();
  int rc = SS_OK;
  auto bail = [&](int code) { ss_release_batch(c); return code; };
#define SS_CUDA_B(expr)                                              \
  do {                                                               \
    cudaError_t _e = (expr);                                         \
    if (_e != cudaSuccess) { c->last_cuda = (int)_e; return bail(SS_ERR_CUDA); } \
  } while (0)
  SS_CUDA_B(send_rows(c, B));

  // chunks of whole sequences
  int s0 = 0;
  while (s0 < B) {
    int s1 = s0, T = 0;
    while (s1 < B && T + (cu[s1 + 1] - cu[s1]) <= c->rt.max_prefill_tokens) { T += cu[s1 + 1] - cu[s1]; ++s1; }
    // the chunk's arrays, packed into one copy (filled while the chunk before runs)
    if (s0 > 0) SS_CUDA_B(wait_up(c));
    const int n_seq = s1 - s0;
    int32_t* tok = (int32_t*)(c->up.data() + c->up_chunk);
    int32_t *tok_slot = tok + T, *tok_pos = tok + 2 * (size_t)T, *cu_loc = tok + 3 * (size_t)T, *last = cu_loc + n_seq + 1;
    std::copy(tokens + cu[s0], tokens + cu[s1], tok);
    for (int s = s0, t = 0; s < s1; ++s) {
      cu_loc[s - s0] = t;
      for (int p = 0; p < cu[s + 1] - cu[s]; ++p, ++t) {
        tok_slot[t] = c->row_pages[s][p / kPageTokens] * kPageTokens + p % kPageTokens;
        tok_pos[t] = p;
      }
      cu_loc[s - s0 + 1] = t;
      last[s - s0] = t - 1;
    }
    SS_CUDA_B(send_up(c, c->d_chunk, tok, (3 * (size_t)T + 2 * n_seq + 1) * 4));
    c->d_tokens = c->d_chunk;
    c->d_tok_slot = c->d_chunk + T;
    c->d_tok_pos = c->d_chunk + 2 * (size_t)T;
    c->d_cu = c->d_chunk + 3 * (size_t)T;
    c->d_last = c->d_cu + n_seq + 1;
    if ((rc = enqueue_prefill_chunk(c, s0, s1, cu, T))) return bail(rc);
    SS_CUDA_B(launch(c, gather_last_rmsnorm_kernel, dim3(s1 - s0), dim3(256), 0, (const float*)c->h,
                     (const int32_t*)c->d_last, c->h_dec + (size_t)s0 * m.d_model, (const bf16*)c->final_norm,
                     c->x_dec + (size_t)s0 * m.d_model,
                     (opts && opts->dump_hidden) ? opts->dump_hidden + (size_t)s0 * m.d_model : (float*)nullptr,
                     m.d_model, m.rms_eps));
    s0 = s1;
  }
  SS_CUDA_B(cudaEventRecord(c->layers_done, c->stream));
  // LM head on the last tokens, first generated token, bookkeeping
  const int NT = round_up(B, 16);
  const CUtensorMap* mx;
  if ((rc = xmap(c, 3, NT, &mx))) return bail(rc);
  const GemmPlan p_lm = plan_gemm(m.vocab, m.d_model, NT, c->n_sm);
  if ((rc = run_gemm(c, c->lm_head, *mx, p_lm, B))) return bail(rc);
  SS_CUDA_B(launch(c, lmhead_tile_argmax_kernel, dim3(c->n_tiles_lm, ceil_div(B, kArgmaxRows)), dim3(128), 0, (const float*)c->partial,
                   split_of(p_lm, c->tbl128[4]), c->st, opts ? opts->dump_logits : (float*)nullptr, c->tile_val,
                   c->tile_idx, B, m.vocab, c->n_tiles_lm, m.eos_id, c->sample));
  SS_CUDA_B(launch(c, bookkeeping_kernel, dim3(1), dim3(1024), 0, c->st, (const float*)c->tile_val,
                   (const int32_t*)c->tile_idx, c->n_tiles_lm, opts ? opts->forced_tokens : (const int32_t*)nullptr,
                   first_tokens, opts ? opts->dump_choice : (int32_t*)nullptr, B, m.eos_id, 1));
#undef SS_CUDA_B
  return SS_OK;
}

extern "C" {

int ss_prefill(ss_ctx* c, const int32_t* tokens, const int32_t* cu, int32_t B, const int32_t* eos_at, int32_t cap,
               const ss_step_opts* opts, int32_t* first_tokens) {
  if (int rc = start_batch(c, tokens, cu, B, eos_at, cap, opts, first_tokens)) return rc;
  // the caller may read dump_hidden and reuse its inputs; the LM head, queued already, keeps the GPU busy meanwhile
  const cudaError_t e = cudaEventSynchronize(c->layers_done);
  if (e != cudaSuccess) { ss_release_batch(c); return cuda_fail(c, e); }
  return SS_OK;
}

int ss_keep_prompts(ss_ctx* c, const int32_t* ids, const int32_t* keep_len) {
  if (!c || !ids || !keep_len) return SS_ERR_ARG;
  if (!c->in_batch || c->batch_cu.empty()) return SS_ERR_STATE;      // no batch, or one that was itself resumed
  const int B = c->B;
  for (int r = 0; r < B; ++r) {
    if (keep_len[r] < 2 || keep_len[r] > c->prompt_len[r]) return SS_ERR_ARG;
    for (int q = 0; q < r; ++q)
      if (ids[q] == ids[r]) return SS_ERR_ARG;
  }
  for (int r = 0; r < B; ++r) {
    auto old = c->kept.find(ids[r]);
    if (old != c->kept.end()) {
      for (int32_t p : old->second.pages) c->free_pages.push_back(p);
      c->kept.erase(old);
    }
    const int n_keep = ceil_div(keep_len[r], kPageTokens);
    ss_ctx::KeptPrompt k;
    k.pages.assign(c->row_pages[r].begin(), c->row_pages[r].begin() + n_keep);
    k.len = keep_len[r];
    k.last_tok = c->batch_tokens[c->batch_cu[r] + keep_len[r] - 1];
    // these pages no longer go back to the pool with the batch
    for (int32_t p : k.pages) {
      auto it = std::find(c->batch_pages.begin(), c->batch_pages.end(), p);
      if (it != c->batch_pages.end()) { *it = c->batch_pages.back(); c->batch_pages.pop_back(); }
    }
    c->kept.emplace(ids[r], std::move(k));
  }
  return SS_OK;
}

int ss_drop_prompts(ss_ctx* c, const int32_t* ids, int32_t n) {
  if (!c || n < -1 || (n > 0 && !ids)) return SS_ERR_ARG;
  if (c->in_batch) return SS_ERR_STATE;
  if (n == -1) {
    for (auto& kv : c->kept)
      for (int32_t p : kv.second.pages) c->free_pages.push_back(p);
    c->kept.clear();
    return SS_OK;
  }
  for (int i = 0; i < n; ++i) {
    auto it = c->kept.find(ids[i]);
    if (it == c->kept.end()) continue;
    for (int32_t p : it->second.pages) c->free_pages.push_back(p);
    c->kept.erase(it);
  }
  return SS_OK;
}

int ss_resume(ss_ctx* c, const int32_t* ids, int32_t B, const int32_t* eos_at, int32_t cap, const ss_step_opts* opts,
              int32_t* first_tokens) {
  if (!c || !ids || B < 1 || cap < 1) return SS_ERR_ARG;
  if (c->n_loaded != c->n_expected || c->in_batch) return SS_ERR_STATE;
  if (B > c->rt.max_batch || cap > c->rt.max_new_tokens) return SS_ERR_CAPACITY;
  size_t need_pages = 0;
  for (int r = 0; r < B; ++r) {
    auto it = c->kept.find(ids[r]);
    if (it == c->kept.end()) return SS_ERR_STATE;
    for (int q = 0; q < r; ++q)
      if (ids[q] == ids[r]) return SS_ERR_ARG;
    const int len = it->second.len;
    if (len + cap > c->rt.max_ctx) return SS_ERR_CAPACITY;
    if (eos_at && eos_at[r] < 1) return SS_ERR_ARG;
    need_pages += (size_t)ceil_div(len + cap, kPageTokens) - it->second.pages.size();
  }
  if (need_pages > c->free_pages.size()) return SS_ERR_KV_BUDGET;
  int32_t *rows, *bt;
  SS_CUDA(c, wait_up(c));
  clear_rows(c, B, cap, &rows, &bt);
  c->batch_pages.clear();
  c->batch_tokens.clear();
  c->batch_cu.clear();
  c->prompt_len.assign(B, 0);
  c->row_pages.assign(B, {});
  for (int r = 0; r < B; ++r) {
    const ss_ctx::KeptPrompt& k = c->kept[ids[r]];
    c->prompt_len[r] = k.len;
    c->row_pages[r] = k.pages;
    const int np = ceil_div(k.len + cap, kPageTokens);
    for (int p = (int)k.pages.size(); p < np; ++p) {
      const int32_t pg = c->free_pages.back();
      c->free_pages.pop_back();
      c->batch_pages.push_back(pg);
      c->row_pages[r].push_back(pg);
    }
    for (int p = 0; p < np; ++p) bt[(size_t)r * c->st.max_pages + p] = c->row_pages[r][p];
    // the row stands one token before the end of its kept prompt: that token is fed again by the first step
    rows[0 * kMaxBatch + r] = k.len - 1;
    rows[1 * kMaxBatch + r] = k.last_tok;
    rows[3 * kMaxBatch + r] = 1;
    rows[5 * kMaxBatch + r] = eos_at ? eos_at[r] : 0;
    rows[6 * kMaxBatch + r] = r < (int)c->next_row_keys.size() ? c->next_row_keys[r] : r;
  }
  c->next_row_keys.clear();
  c->in_batch = true;
  c->B = B;
  c->cap = cap;
  auto bail = [&](int code) { ss_release_batch(c); return code; };
  const cudaError_t e = send_rows(c, B);
  if (e != cudaSuccess) { c->last_cuda = (int)e; return bail(SS_ERR_CUDA); }
  int rc = enqueue_decode_step(c, opts, first_tokens);
  if (rc) return bail(rc);
  return SS_OK;
}

int ss_set_prompt_cache(ss_ctx* c, int32_t mode, const int32_t* keep_len, int32_t n) {
  if (!c || mode < 0 || mode > 2 || n < 0 || (mode == 1 && (!keep_len || n < 1))) return SS_ERR_ARG;
  c->prompt_cache_mode = mode;
  c->cache_keep_len.clear();
  if (mode == 1) c->cache_keep_len.assign(keep_len, keep_len + n);
  return SS_OK;
}

int ss_decode_step(ss_ctx* c, const ss_step_opts* opts, int32_t* next_tokens, int32_t* n_active_host) {
  if (!c) return SS_ERR_ARG;
  if (!c->in_batch) return SS_ERR_STATE;
  int rc = enqueue_decode_step(c, opts, next_tokens);
  if (rc) return rc;
  if (n_active_host)
    SS_CUDA(c, cudaMemcpyAsync(n_active_host, c->st.scalars + 1, 4, cudaMemcpyDeviceToHost, c->stream));
  return SS_OK;
}

int ss_decode_steps(ss_ctx* c, int32_t n_steps, int32_t* n_active_host) {
  if (!c || n_steps < 0) return SS_ERR_ARG;
  if (!c->in_batch) return SS_ERR_STATE;
  for (int s = 0; s < n_steps; ++s) {
    int rc = enqueue_decode_step(c, nullptr, nullptr);
    if (rc) return rc;
  }
  if (n_active_host)
    SS_CUDA(c, cudaMemcpyAsync(n_active_host, c->st.scalars + 1, 4, cudaMemcpyDeviceToHost, c->stream));
  return SS_OK;
}

int ss_read_batch(ss_ctx* c, int32_t* out_tokens, int32_t stride, int32_t* out_len, uint8_t* out_status) {
  if (!c || !out_len || !out_status || (out_tokens && stride < 1)) return SS_ERR_ARG;
  if (!c->in_batch) return SS_ERR_STATE;
  const int B = c->B;
  // row state and status come back together; the tokens (rows of the batch's cap) with them where that is little, else
  // once it is known how many there are
  int32_t* rows = c->down_rows.data();
  auto fetch_tokens = [&](int n) -> cudaError_t {
    try {
      if (c->down_tokens.size() < (size_t)B * n) c->down_tokens.resize((size_t)B * n);
    } catch (const std::bad_alloc&) {
      return cudaErrorMemoryAllocation;
    }
    return cudaMemcpy2DAsync(c->down_tokens.data(), (size_t)n * 4, c->st.out_tokens, (size_t)c->st.max_new * 4, (size_t)n * 4, B, cudaMemcpyDeviceToHost,
                             c->stream);
  };
  int n_tok = out_tokens && (size_t)B * c->cap <= 16384 ? c->cap : 0;
  SS_CUDA(c, cudaMemcpyAsync(rows, c->st.ctx_len, kRowStateBytes, cudaMemcpyDeviceToHost, c->stream));
  SS_CUDA(c, cudaMemcpyAsync(c->pinned + 1, c->status, 4, cudaMemcpyDeviceToHost, c->stream));
  if (n_tok) SS_CUDA(c, fetch_tokens(n_tok));
  SS_CUDA(c, cudaStreamSynchronize(c->stream));
  if (c->pinned[1] != 0) return report_device_status(c, (uint32_t)c->pinned[1]);
  const int32_t *gen = rows + 2 * kMaxBatch, *fin = rows + 4 * kMaxBatch;
  int longest = 0;
  for (int r = 0; r < B; ++r) {
    if (out_tokens && gen[r] > stride) return SS_ERR_CAPACITY;
    out_len[r] = gen[r];
    out_status[r] = fin[r] ? 1 : 0;
    longest = std::max(longest, gen[r]);
  }
  if (out_tokens && longest > 0) {
    if (!n_tok) {
      n_tok = longest;
      SS_CUDA(c, fetch_tokens(n_tok));
      SS_CUDA(c, cudaStreamSynchronize(c->stream));
    }
    const int32_t* tok = c->down_tokens.data();
    for (int r = 0; r < B; ++r) std::copy(tok + (size_t)r * n_tok, tok + (size_t)r * n_tok + gen[r], out_tokens + (size_t)r * stride);
  }
  return SS_OK;
}

int ss_step_model_bytes(const ss_ctx* c, const int32_t* ctx_len, const uint8_t* active, int32_t B, double* out) {
  if (!c || !ctx_len || !out || B < 0) return SS_ERR_ARG;
  double bytes = weight_bytes_per_step(c->m);
  const double kvt = kv_bytes_per_token(c->m);
  for (int r = 0; r < B; ++r)
    if (!active || active[r]) bytes += kvt * ((double)ctx_len[r] + 1.0) + (double)c->m.d_model * 2.0;
  *out = bytes;
  return SS_OK;
}

int ss_last_device_status(ss_ctx* c, uint32_t* out) {
  if (!c || !out) return SS_ERR_ARG;
  SS_CUDA(c, cudaMemcpyAsync(c->pinned + 1, c->status, 4, cudaMemcpyDeviceToHost, c->stream));
  SS_CUDA(c, cudaStreamSynchronize(c->stream));
  *out = (uint32_t)c->pinned[1];
  return SS_OK;
}

int ss_set_sampling(ss_ctx* c, float temperature, uint64_t seed) {
  if (!c || !(temperature >= 0.f) || !std::isfinite(temperature)) return SS_ERR_ARG;
  c->sample.inv_temp = temperature > 0.f ? 1.f / temperature : 0.f;
  c->sample.seed_lo = (uint32_t)(seed & 0xffffffffu);
  c->sample.seed_hi = (uint32_t)(seed >> 32);
  return SS_OK;
}

int ss_set_row_keys(ss_ctx* c, const int32_t* keys, int32_t n) {
  if (!c || n < 0 || n > kMaxBatch || (n > 0 && !keys)) return SS_ERR_ARG;
  c->next_row_keys.assign(keys, keys + n);
  return SS_OK;
}

int ss_set_wait_limit_ms(ss_ctx* c, int32_t ms) {
  if (!c || ms < 1 || ms > 60000) return SS_ERR_ARG;
  c->wait_limit = (long long)ms * c->clock_khz;
  return SS_OK;
}

int ss_selftest_wait_timeout(ss_ctx* c, int32_t limit_us) {
  if (!c || limit_us < 1 || limit_us > 1000000) return SS_ERR_ARG;
  if (c->in_batch) return SS_ERR_STATE;
  // the workers of an abandoned step leave together
  {
    MegaArgs a{};
    a.grid_ctr = c->grid_ctr;
    a.grid_base = c->grid_epochs * (unsigned long long)c->n_sm;
    a.status = c->status;
    a.wait_limit = c->wait_limit;
    uint32_t* torn = c->status + 1;
    SS_CUDA(c, cudaMemsetAsync(torn, 0, 4, c->stream));
    void* args[2] = {(void*)&a, (void*)&torn};
    SS_CUDA(c, cudaLaunchCooperativeKernel((const void*)leave_selftest_kernel, dim3(c->n_sm), dim3(kLeaveSelftestThreads), args, 0, c->stream));
    c->launches++;
    SS_CUDA(c, cudaMemcpyAsync(c->pinned + 1, c->status, 8, cudaMemcpyDeviceToHost, c->stream));
    SS_CUDA(c, cudaStreamSynchronize(c->stream));
    const bool clean = c->pinned[1] == 0 && c->pinned[2] == 0;
    reset_grid(c);
    if (!clean) {
      SS_CUDA(c, cudaMemsetAsync(c->status, 0, 4, c->stream));
      return SS_OK;                    // an abort does not end as it should
    }
  }
  MegaArgs a{};
  a.NT = 16;
  a.shape[0].max_seg = 1;
  a.shape[0].partial = c->part_dec[0];
  a.grid_ctr = c->grid_ctr;
  a.grid_base = c->grid_epochs * (unsigned long long)c->n_sm;
  a.status = c->status;
  a.wait_limit = (long long)limit_us * c->clock_khz / 1000;
  const uint32_t* flag = c->pair_flag;
  uint32_t* ran_out = c->status + 1;
  SS_CUDA(c, cudaMemsetAsync(ran_out, 0, 4, c->stream));
  void* args[3] = {(void*)&a, (void*)&flag, (void*)&ran_out};
  SS_CUDA(c, cudaLaunchCooperativeKernel((const void*)wait_selftest_kernel, dim3(c->n_sm), dim3(32), args, 0, c->stream));
  c->launches++;
  SS_CUDA(c, cudaMemcpyAsync(c->pinned + 1, c->status, 8, cudaMemcpyDeviceToHost, c->stream));
  // what an abandoned step can leave behind: sums in the slots, flags up
  SS_CUDA(c, cudaMemsetAsync(c->part_dec[0], 0, c->part_dec_bytes, c->stream));
  SS_CUDA(c, cudaMemsetAsync(c->pair_flag, 1, (size_t)c->n_sm * 8 * sizeof(uint32_t), c->stream));
  SS_CUDA(c, cudaStreamSynchronize(c->stream));
  const int rc = report_device_status(c, (uint32_t)c->pinned[1]);          // clears all of it
  return c->pinned[1] != 0 && (uint32_t)c->pinned[2] == (1u << kWaitSelftests) - 1 ? rc : SS_OK;
}

int ss_set_trace(ss_ctx* c, int32_t on) {
  if (!c) return SS_ERR_ARG;
  if (on) SS_CUDA(c, prepare_mega_kernels(c->m.head_dim, true));
  c->trace_on = on != 0;
  return SS_OK;
}

int ss_step_trace(ss_ctx* c, uint64_t* out, int32_t cap, int32_t* n) {
  if (!c || !out || !n) return SS_ERR_ARG;
  if (!c->trace_on) return SS_ERR_STATE;
  *n = c->trace_len;
  if (cap < c->trace_len) return SS_ERR_CAPACITY;
  SS_CUDA(c, cudaMemcpyAsync(out, c->trace, (size_t)c->trace_len * 8, cudaMemcpyDeviceToHost, c->stream));
  SS_CUDA(c, cudaStreamSynchronize(c->stream));
  return SS_OK;
}

int ss_last_cuda_error(const ss_ctx* c) { return c ? c->last_cuda : 0; }
int64_t ss_kernel_launches(const ss_ctx* c) { return c ? c->launches : 0; }

}  // extern "C"

// Runs the micro-batches batches[0..n_batches) (rows: order[first_row .. first_row + n_rows)) one after the other:
// prompt pass, decode until every row has finished or the cap, read back.  Rows the cap cut (cap < max_new, no EOS)
// are appended to `fails`; the others get their final tokens, length and status.  Adds to `gs`, writes one log record
// per batch from log[*n_log] on.
static int run_batch_list(ss_ctx* c, const ss_sched_cfg* cfg, const int32_t* prompt_tokens, const int64_t* prompt_off,
                          const int32_t* eos_at, const int32_t* order, const ss_batch_desc* batches, int32_t n_batches,
                          int32_t* out_tokens, const int64_t* out_off, int32_t* out_len, uint8_t* out_status,
                          std::vector<int32_t>& fails, ss_batch_log* log, int32_t log_cap, int32_t* n_log,
                          ss_group_stats& gs) {
  cudaEvent_t ev[3] = {nullptr, nullptr, nullptr};       // batch start, prompt pass done, decode done
  auto cleanup = [&](int code) {
    for (auto& e : ev)
      if (e) cudaEventDestroy(e);
    if (c->in_batch) ss_release_batch(c);
    return code;
  };
  // every CUDA failure below leaves through cleanup(): events destroyed, pages of a batch in flight returned
#define SS_CUDA_G(expr)                                                          \
  do {                                                                           \
    cudaError_t _e = (expr);                                                     \
    if (_e != cudaSuccess) { c->last_cuda = (int)_e; return cleanup(SS_ERR_CUDA); } \
  } while (0)
  for (auto& e : ev) SS_CUDA_G(cudaEventCreate(&e));
  const double W = weight_bytes_per_step(c->m), kvt = kv_bytes_per_token(c->m);
  std::vector<int32_t> toks, cu, eos_b, len_b, tok_b;
  std::vector<uint8_t> st_b;
  int rc;
  for (int32_t bi = 0; bi < n_batches; ++bi) {
    const ss_batch_desc b = batches[bi];
    const int32_t* rows_src = order + b.first_row;
    const int B = b.n_rows;
    if (log && *n_log >= log_cap) return cleanup(SS_ERR_CAPACITY);
    toks.clear();
    cu.assign(1, 0);
    eos_b.clear();
    int max_target = 0;
    for (int r = 0; r < B; ++r) {
      const int q = rows_src[r];
      toks.insert(toks.end(), prompt_tokens + prompt_off[q], prompt_tokens + prompt_off[q + 1]);
      cu.push_back((int32_t)toks.size());
      if (eos_at) { eos_b.push_back(eos_at[q]); max_target = std::max(max_target, eos_at[q]); }
    }
    c->next_row_keys.assign(rows_src, rows_src + B);      // a row's sampling key is its query id, in every pass
    // prompt reuse (App. C): a batch whose queries all have kept prompts starts from them instead of a prompt pass
    bool resume = c->prompt_cache_mode == 2;
    for (int r = 0; r < B && resume; ++r) resume = c->kept.count(rows_src[r]) != 0;
    SS_CUDA_G(cudaEventRecord(ev[0], c->stream));
    if (resume) rc = ss_resume(c, rows_src, B, eos_at ? eos_b.data() : nullptr, b.cap, nullptr, nullptr);
    else rc = start_batch(c, toks.data(), cu.data(), B, eos_at ? eos_b.data() : nullptr, b.cap, nullptr, nullptr);
    if (rc) return cleanup(rc);
    if (c->prompt_cache_mode == 1 && !resume) {
      std::vector<int32_t> kl(B);
      for (int r = 0; r < B; ++r) {
        const int q = rows_src[r];
        if (q >= (int)c->cache_keep_len.size()) return cleanup(SS_ERR_ARG);
        kl[r] = c->cache_keep_len[q];
      }
      if ((rc = ss_keep_prompts(c, rows_src, kl.data()))) return cleanup(rc);
    }
    SS_CUDA_G(cudaEventRecord(ev[1], c->stream));
    if (eos_at) {
      // lengths are forced, so the number of steps is known: the longest target or the cap
      const int steps = std::min(b.cap, max_target);
      if ((rc = ss_decode_steps(c, steps - 1, nullptr))) return cleanup(rc);
    } else {
      int done = 1;
      while (done < b.cap) {
        const int chunk = std::min(8, b.cap - done);
        if ((rc = ss_decode_steps(c, chunk, c->pinned))) return cleanup(rc);
        SS_CUDA_G(cudaStreamSynchronize(c->stream));
        done += chunk;
        if (c->pinned[0] == 0) break;
      }
    }
    SS_CUDA_G(cudaEventRecord(ev[2], c->stream));
    len_b.assign(B, 0);
    st_b.assign(B, 0);
    tok_b.assign((size_t)B * cfg->max_new_tokens, 0);
    if ((rc = ss_read_batch(c, tok_b.data(), cfg->max_new_tokens, len_b.data(), st_b.data()))) return cleanup(rc);
    ss_release_batch(c);
    float pf = 0, dc = 0;
    cudaEventElapsedTime(&pf, ev[0], ev[1]);
    cudaEventElapsedTime(&dc, ev[1], ev[2]);
    int steps = 0, n_failed = 0;
    for (int r = 0; r < B; ++r) {
      const int q = rows_src[r];
      steps = std::max(steps, len_b[r]);
      const bool failed = !st_b[r] && b.cap < cfg->max_new_tokens;
      if (failed) {
        fails.push_back(q);
        ++n_failed;
      } else {
        out_len[q] = len_b[r];
        out_status[q] = st_b[r];
        std::copy(tok_b.begin() + (size_t)r * cfg->max_new_tokens,
                  tok_b.begin() + (size_t)r * cfg->max_new_tokens + len_b[r], out_tokens + out_off[q]);
        gs.useful_tokens += len_b[r];
      }
      const double nr = std::max(0, len_b[r] - 1);     // decode steps the row took part in
      gs.model_bytes += kvt * (nr * (cu[r + 1] - cu[r]) + nr * (nr + 1) / 2.0);
    }
    gs.model_bytes += W * std::max(0, steps - 1);
    if (log) log[*n_log] = {b.first_row, B, b.cap, b.is_recompute, steps, n_failed, pf, dc};
    ++*n_log;
    gs.n_batches += 1;
    gs.steps += steps;
    gs.row_steps += (int64_t)B * steps;
    gs.prefill_ms += pf;
    gs.decode_ms += dc;
    gs.n_failed += n_failed;
  }
#undef SS_CUDA_G
  return cleanup(SS_OK);
}

extern "C" {

int ss_run_batches(ss_ctx* c, const ss_sched_cfg* cfg, const int32_t* prompt_tokens, const int64_t* prompt_off,
                   const int32_t* eos_at, int32_t n, const int32_t* order, int32_t n_order, const ss_batch_desc* batches,
                   int32_t n_batches, int32_t* out_tokens, const int64_t* out_off, int32_t* out_len, uint8_t* out_status,
                   int32_t* fail_rows, int32_t* n_fail, ss_batch_log* log, int32_t log_cap, int32_t* n_log,
                   ss_group_stats* stats) {
  if (!c || !cfg || n < 0 || n_batches < 0 || n_order < 0 || !n_log || !n_fail) return SS_ERR_ARG;
  if (n_batches > 0 && (!prompt_tokens || !prompt_off || !order || !batches || !out_tokens || !out_off || !out_len ||
                        !out_status || !fail_rows))
    return SS_ERR_ARG;
  int rc = validate_sched_cfg(cfg);
  if (rc) return rc;
  if (c->in_batch) return SS_ERR_STATE;
  if (cfg->max_new_tokens > c->rt.max_new_tokens) return SS_ERR_CAPACITY;
  for (int32_t i = 0; i < n_batches; ++i) {
    const ss_batch_desc& b = batches[i];
    if (b.n_rows < 1 || b.first_row < 0 || (int64_t)b.first_row + b.n_rows > n_order || b.cap < 1 ||
        b.cap > cfg->max_new_tokens)
      return SS_ERR_ARG;
    for (int r = 0; r < b.n_rows; ++r) {
      const int32_t q = order[b.first_row + r];
      if (q < 0 || q >= n) return SS_ERR_ARG;
      if (out_off[q + 1] - out_off[q] < cfg->max_new_tokens) return SS_ERR_CAPACITY;
    }
  }
  cudaEvent_t g0 = nullptr, g1 = nullptr;
  if (cudaEventCreate(&g0) != cudaSuccess || cudaEventCreate(&g1) != cudaSuccess) {
    if (g0) cudaEventDestroy(g0);
    return SS_ERR_CUDA;
  }
  ss_group_stats gs{};
  const int64_t launches0 = c->launches;
  std::vector<int32_t> fails;
  *n_log = 0;
  cudaEventRecord(g0, c->stream);
  rc = run_batch_list(c, cfg, prompt_tokens, prompt_off, eos_at, order, batches, n_batches, out_tokens, out_off,
                      out_len, out_status, fails, log, log_cap, n_log, gs);
  if (rc == SS_OK) {
    cudaEventRecord(g1, c->stream);
    if (cudaEventSynchronize(g1) != cudaSuccess) rc = SS_ERR_CUDA;
    else cudaEventElapsedTime(&gs.total_ms, g0, g1);
  }
  cudaEventDestroy(g0);
  cudaEventDestroy(g1);
  if (rc) return rc;
  std::copy(fails.begin(), fails.end(), fail_rows);
  *n_fail = (int32_t)fails.size();
  gs.kernel_launches = c->launches - launches0;
  if (stats) *stats = gs;
  return SS_OK;
}

int ss_run_group(ss_ctx* c, const ss_sched_cfg* cfg, const int32_t* prompt_tokens, const int64_t* prompt_off,
                 const int32_t* pred_len, const int32_t* perm, const int32_t* eos_at, int32_t n, int32_t* out_tokens,
                 const int64_t* out_off, int32_t* out_len, uint8_t* out_status, int32_t* order, ss_batch_log* log,
                 int32_t log_cap, int32_t* n_log, ss_group_stats* stats) {
  if (!c || !cfg || n < 0 || !n_log) return SS_ERR_ARG;
  if (n > 0 && (!prompt_tokens || !prompt_off || !pred_len || !out_tokens || !out_off || !out_len || !out_status || !order))
    return SS_ERR_ARG;
  int rc = validate_sched_cfg(cfg);
  if (rc) return rc;
  if (c->in_batch) return SS_ERR_STATE;
  if (cfg->max_new_tokens > c->rt.max_new_tokens) return SS_ERR_CAPACITY;
  for (int i = 0; i < n; ++i)
    if (out_off[i + 1] - out_off[i] < cfg->max_new_tokens) return SS_ERR_CAPACITY;

  std::vector<int32_t> plen(n);
  for (int i = 0; i < n; ++i) plen[i] = (int32_t)(prompt_off[i + 1] - prompt_off[i]);
  std::vector<int32_t> ord;
  std::vector<ss_batch_desc> plan;
  if ((rc = plan_first_pass(*cfg, plen.data(), pred_len, perm, n, ord, plan))) return rc;

  cudaEvent_t g0 = nullptr, g1 = nullptr;
  if (cudaEventCreate(&g0) != cudaSuccess || cudaEventCreate(&g1) != cudaSuccess) {
    if (g0) cudaEventDestroy(g0);
    return SS_ERR_CUDA;
  }
  auto done = [&](int code) { cudaEventDestroy(g0); cudaEventDestroy(g1); return code; };
  ss_group_stats gs{};
  const int64_t launches0 = c->launches;
  std::vector<int32_t> fails;
  *n_log = 0;
  cudaEventRecord(g0, c->stream);
  // first pass
  rc = run_batch_list(c, cfg, prompt_tokens, prompt_off, eos_at, ord.data(), plan.data(), (int32_t)plan.size(),
                      out_tokens, out_off, out_len, out_status, fails, log, log_cap, n_log, gs);
  if (rc) return done(rc);
  // the rows the caps cut, in collection order, regenerated from their prompts in batches of B0 with cap = max_new
  // (Sec. 4.1, failure collection and recomputation); they are listed behind the first-pass order
  const size_t n_fail = fails.size();
  ord.insert(ord.end(), fails.begin(), fails.end());
  std::vector<ss_batch_desc> again;
  for (size_t i = 0; i < n_fail; i += (size_t)cfg->base_batch)
    again.push_back({(int32_t)(n + i), (int32_t)std::min<size_t>(cfg->base_batch, n_fail - i), cfg->max_new_tokens, 1});
  std::vector<int32_t> fails2;
  rc = run_batch_list(c, cfg, prompt_tokens, prompt_off, eos_at, ord.data(), again.data(), (int32_t)again.size(),
                      out_tokens, out_off, out_len, out_status, fails2, log, log_cap, n_log, gs);
  if (rc) return done(rc);
  gs.n_failed = (int32_t)n_fail;
  for (int i = 0; i < n; ++i) order[i] = ord[i];
  for (size_t i = 0; i < n_fail; ++i) order[n + i] = fails[i];
  for (size_t i = n_fail; i < (size_t)n; ++i) order[n + i] = -1;
  cudaEventRecord(g1, c->stream);
  if (cudaEventSynchronize(g1) != cudaSuccess) return done(SS_ERR_CUDA);
  cudaEventElapsedTime(&gs.total_ms, g0, g1);
  gs.kernel_launches = c->launches - launches0;
  if (stats) *stats = gs;
  return done(SS_OK);
}

}  // extern "C"
