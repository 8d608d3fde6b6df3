// ss_logits_noalloc(): the LM-head projection for callers that cannot allocate device memory.
//
// Who needs this: code that runs where cudaMalloc is off limits -- inside a region that is being
// captured into a CUDA graph by the caller's framework, inside a memory-pool callback, in a
// process whose device memory is fully handed out to another allocator, or in a real-time loop
// where an allocation (and the implicit synchronisation it can bring) is not acceptable.  Such a
// caller owns its inputs and outputs but has nowhere to put the two temporaries the projection
// needs (the normalised bf16 activations and the fp32 split-K partial sums).  Here they live in
// one file-scope __device__ array of fixed size that every GPU which loads this library carries
// until the process exits.
//
// Same arithmetic as the LM head inside ss_prefill()/ss_decode_step(): x = RMSNorm(h) * g in bf16,
// the tcgen05 weight-streaming GEMM with fp32 partials, partials added in CTA order.
#include <mutex>

#include "ss_gemm.cuh"

using namespace ss;

namespace {

constexpr size_t kScratchBytes = 8u << 20;            // 8 MiB, all of it
constexpr int kNoAllocMaxRows = 16;                    // tokens per call
constexpr int kNoAllocMaxD = 8192;
constexpr size_t kXBytes = (size_t)kNoAllocMaxRows * kNoAllocMaxD * 2;   // bf16 activations, 256 KiB
constexpr int kMaxDevices = 64;

static __device__ __align__(256) unsigned char g_noalloc_scratch[kScratchBytes];

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

struct DeviceSetup {
  bool ready = false;
  unsigned char* scratch = nullptr;     // device address of g_noalloc_scratch on this device
  int n_sm = 0;
};
std::mutex g_mu;
DeviceSetup g_dev[kMaxDevices];
EncodeTiledFn g_encode = nullptr;

// x[r] = RMSNorm(h[r]) * g as bf16; rows r >= n_rows of the 16-row operand are zeroed; the status word starts at zero.
// One pass: 256 threads hold the row (d a multiple of 64, at most 8192) as 8 x 4 values each.  `vec`: h is 16-byte and g
// 8-byte aligned (the caller's pointers need not be).
__global__ void __launch_bounds__(256)
noalloc_rmsnorm_kernel(const float* __restrict__ h, const __nv_bfloat16* __restrict__ g, __nv_bfloat16* __restrict__ x,
                       int n_rows, int d, float eps, int vec, uint32_t* status) {
  __shared__ float red[8];
  pdl_launch_dependents();
  const int r = blockIdx.x, d4 = d >> 2;
  if (r == 0 && threadIdx.x == 0) *status = 0u;
  uint2* out = reinterpret_cast<uint2*>(x + (size_t)r * d);
  if (r >= n_rows) {
    for (int i = threadIdx.x; i < d4; i += 256) out[i] = make_uint2(0u, 0u);
    return;
  }
  const float* hr = h + (size_t)r * d;
  float4 v[8];
  float ss = 0.f;
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const int i = threadIdx.x + k * 256;
    v[k] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (i < d4) v[k] = vec ? __ldg(reinterpret_cast<const float4*>(hr) + i) : make_float4(hr[4 * i], hr[4 * i + 1], hr[4 * i + 2], hr[4 * i + 3]);
    ss += v[k].x * v[k].x + v[k].y * v[k].y + v[k].z * v[k].z + v[k].w * v[k].w;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = ss;
  __syncthreads();
  float tot = 0.f;
#pragma unroll
  for (int w = 0; w < 8; ++w) tot += red[w];
  const float inv = rsqrtf(tot / d + eps);
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const int i = threadIdx.x + k * 256;
    if (i < d4) {
      __nv_bfloat162 g01, g23;
      if (vec) {
        const uint2 gb = __ldg(reinterpret_cast<const uint2*>(g) + i);
        g01 = *reinterpret_cast<const __nv_bfloat162*>(&gb.x);
        g23 = *reinterpret_cast<const __nv_bfloat162*>(&gb.y);
      } else {
        g01 = __nv_bfloat162(g[4 * i], g[4 * i + 1]);
        g23 = __nv_bfloat162(g[4 * i + 2], g[4 * i + 3]);
      }
      const float2 a = __bfloat1622float2(g01), b = __bfloat1622float2(g23);
      out[i] = make_uint2(pack_bf16x2(v[k].x * inv * a.x, v[k].y * inv * a.y), pack_bf16x2(v[k].z * inv * b.x, v[k].w * inv * b.y));
    }
  }
}

// logits[r][v] = sum of the partials of output row v for token r, in CTA order.  If a bounded wait of the
// projection gave up (status word non-zero) the partials are not all there: the whole output becomes NaN,
// which is how this call, having already returned, reports the failure.
// grid (128-row tiles, rows / kReduceRows), block 128 (thread = vocabulary row of the tile).  The tile's segments follow from
// the split arithmetic, 32-bit here: (CTAs + 1) x (tiles x k-blocks) is far below 2^31 for every size the array holds.
constexpr int kReduceRows = 4;
__global__ void __launch_bounds__(128)
noalloc_reduce_kernel(const float* __restrict__ partial, SplitInfo sp, float* __restrict__ logits, int V, int n_rows,
                      const uint32_t* __restrict__ status) {
  const int tile = blockIdx.x, v = tile * 128 + threadIdx.x, total = (int)sp.total;
  auto begin = [&](int c) { return c * total / sp.gridx; };
  auto owner = [&](int x) {
    int c = (int)((unsigned int)x * (unsigned int)sp.gridx / (unsigned int)total);
    while (c + 1 < sp.gridx && begin(c + 1) <= x) ++c;
    return c;
  };
  const int c0 = owner(tile * sp.kb), c1 = owner(tile * sp.kb + sp.kb - 1);
  const int slot0 = c0 * sp.max_seg + tile - begin(c0) / sp.kb;
  const size_t slot_stride = (size_t)sp.NT * 128, cta_stride = slot_stride * sp.max_seg;
  pdl_wait();
  const bool failed = *status != 0u;
  const int r0 = blockIdx.y * kReduceRows;
  float acc[kReduceRows];
#pragma unroll
  for (int j = 0; j < kReduceRows; ++j)
    acc[j] = r0 + j < n_rows ? __ldcg(partial + (size_t)slot0 * slot_stride + (size_t)(r0 + j) * 128 + threadIdx.x) : 0.f;
  for (int c = c0 + 1; c <= c1; ++c)
#pragma unroll
    for (int j = 0; j < kReduceRows; ++j)
      if (r0 + j < n_rows) acc[j] += __ldcg(partial + (size_t)c * cta_stride + (size_t)(r0 + j) * 128 + threadIdx.x);
  if (v >= V) return;
#pragma unroll
  for (int j = 0; j < kReduceRows; ++j)
    if (r0 + j < n_rows) logits[(size_t)(r0 + j) * V + v] = failed ? __int_as_float(0x7fc00000) : acc[j];
}

// A launch that, if `early`, may start before the kernel in front of it has finished; it waits for it itself
// (griddepcontrol.wait, which passes at once behind an ordinary launch).
template <class... KArgs, class... Args>
cudaError_t launch_after(bool early, void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream, Args... args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = early ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kern, KArgs(args)...);
}

int setup_device(int dev, DeviceSetup** out) {
  if (dev < 0 || dev >= kMaxDevices) return SS_ERR_UNSUPPORTED;
  std::lock_guard<std::mutex> lock(g_mu);
  DeviceSetup& s = g_dev[dev];
  if (!s.ready) {
    // The array's name is only a host-side handle; the kernels need its address on THIS device.
    void* p = nullptr;
    if (cudaGetSymbolAddress(&p, g_noalloc_scratch) != cudaSuccess || !p) return SS_ERR_CUDA;
    int n = 0;
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n < 1) return SS_ERR_CUDA;
    if (cudaFuncSetAttribute(gemm_wx_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024) != cudaSuccess)
      return SS_ERR_CUDA;
    if (!g_encode) {
      void* fn = nullptr;
      cudaDriverEntryPointQueryResult qr;
      if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &qr) != cudaSuccess || !fn)
        return SS_ERR_CUDA;
      g_encode = (EncodeTiledFn)fn;
    }
    s.scratch = (unsigned char*)p;
    s.n_sm = n;
    s.ready = true;
  }
  *out = &s;
  return SS_OK;
}

int encode_map(CUtensorMap* m, const void* base, int64_t rows, int64_t cols, int box_rows) {
  cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)cols * 2};
  cuuint32_t box[2] = {(cuuint32_t)kTileK, (cuuint32_t)box_rows};
  cuuint32_t estr[2] = {1, 1};
  return g_encode(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS ? SS_OK : SS_ERR_CUDA;
}

}  // namespace

extern "C" int ss_logits_noalloc(const float* hidden, const void* norm_gain, const void* lm_head, int32_t n_rows,
                                 int32_t d_model, int32_t vocab, float rms_eps, float* logits, void* stream) {
  if (!hidden || !norm_gain || !lm_head || !logits) return SS_ERR_ARG;
  if (n_rows < 1 || d_model < 64 || vocab < 1) return SS_ERR_ARG;
  if (((uintptr_t)lm_head & 15) || (d_model % 64)) return SS_ERR_UNSUPPORTED;
  if (n_rows > kNoAllocMaxRows || d_model > kNoAllocMaxD) return SS_ERR_CAPACITY;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return SS_ERR_CUDA;
  (void)cudaGetLastError();   // an error left behind by the caller's earlier work is not this call's
  DeviceSetup* s = nullptr;
  int rc = setup_device(dev, &s);
  if (rc) return rc;

  // split of the (tile, k-block) space over the SMs, as in the engine's decode step
  GemmPlan p{};
  p.n_out = vocab;
  p.K = d_model;
  p.n_tiles = (vocab + kTileM - 1) / kTileM;
  p.kb = d_model / kTileK;
  p.NT = kNoAllocMaxRows;
  const long long total = (long long)p.n_tiles * p.kb;
  p.gridx = (int)(total < s->n_sm ? total : s->n_sm);
  const int ipc = (int)((total + p.gridx - 1) / p.gridx);
  p.max_seg = (ipc + p.kb - 2) / p.kb + 1;
  const int stage_bytes = kTileM * kTileK * 2 + p.NT * kTileK * 2;
  p.stages = (227 * 1024 - 2048) / stage_bytes;
  if (p.stages > kGemmMaxStages) p.stages = kGemmMaxStages;
  p.smem_bytes = 2048 + p.stages * stage_bytes;
  p.tmem_cols = 32;
  const size_t partial_bytes = (size_t)p.gridx * p.max_seg * p.NT * 128 * sizeof(float);
  if (kXBytes + 256 + partial_bytes > kScratchBytes) return SS_ERR_CAPACITY;   // vocabulary too large for the array

  __nv_bfloat16* x = reinterpret_cast<__nv_bfloat16*>(s->scratch);
  uint32_t* status = reinterpret_cast<uint32_t*>(s->scratch + kXBytes);
  float* partial = reinterpret_cast<float*>(s->scratch + kXBytes + 256);
  cudaStream_t st = (cudaStream_t)stream;

  CUtensorMap mw, mx;
  if (encode_map(&mw, lm_head, vocab, d_model, kTileM) || encode_map(&mx, x, kNoAllocMaxRows, d_model, p.NT))
    return SS_ERR_CUDA;
  // The first kernel starts when the stream's earlier work has finished; the projection may start beside it and fetch its
  // first weights (which are older than the first kernel), the summing kernel beside the projection.
  // Not inside a capture: the graph would hold edges with data of their own, which a framework cannot read with the calls
  // that know plain ones only (captured, us a call with such edges and without: 5 rows x 512 x 1000 6.8 and 8.6, 16 x 4096 x
  // 32000 48.3 and 50.9).
  cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(st, &capture) != cudaSuccess) {
    (void)cudaGetLastError();   // the launches report what is wrong with the stream
    capture = cudaStreamCaptureStatusNone;
  }
  const bool early = capture == cudaStreamCaptureStatusNone;
  const int vec = ((uintptr_t)hidden & 15) == 0 && ((uintptr_t)norm_gain & 7) == 0;
  noalloc_rmsnorm_kernel<<<kNoAllocMaxRows, 256, 0, st>>>(hidden, (const __nv_bfloat16*)norm_gain, x, n_rows, d_model, rms_eps, vec, status);
  GemmArgs a{};
  a.p = p;
  a.n_tok = n_rows;
  a.partial = partial;
  a.status = status;
  a.wait_limit = kDefaultWaitLimit;
  if (launch_after(early, gemm_wx_kernel, dim3(p.gridx), dim3(kGemmThreads), (size_t)p.smem_bytes, st, mw, mx, a) != cudaSuccess) return SS_ERR_CUDA;
  SplitInfo sp;
  sp.gridx = p.gridx; sp.kb = p.kb; sp.max_seg = p.max_seg; sp.NT = p.NT; sp.total = total; sp.tiles = nullptr;
  if (launch_after(early, noalloc_reduce_kernel, dim3(p.n_tiles, (n_rows + kReduceRows - 1) / kReduceRows), dim3(128), 0, st, (const float*)partial, sp, logits,
                   vocab, n_rows, (const uint32_t*)status) != cudaSuccess) return SS_ERR_CUDA;
  return cudaGetLastError() == cudaSuccess ? SS_OK : SS_ERR_CUDA;
}
