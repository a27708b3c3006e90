// Device side of libfcp: launchers behind the C ABI, the HBM-bound kernels (LSE merge, backward
// preprocess, dQ conversion) and the glue around the tensor-core kernels of fcp_fwd.cuh and
// fcp_bwd.cuh.  No call here allocates device memory except fcp_plan_upload, also where the first call of the host entry point
// uploads the plans of its runs.
#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <mutex>
#include <vector>

#include "fcp_bwd.cuh"
#include "fcp_fwd.cuh"

using namespace fcp;

#define FCP_CUDA_CHECK(expr)                                                             \
  do {                                                                                   \
    cudaError_t e_ = (expr);                                                             \
    if (e_ != cudaSuccess) {                                                             \
      fcp_set_error("%s failed: %s (%s:%d)", #expr, cudaGetErrorString(e_), __FILE__, __LINE__); \
      return FCP_ERR_CUDA;                                                               \
    }                                                                                    \
  } while (0)

// ---------------------------------------------------------------------------------------------
// Tensor maps
// ---------------------------------------------------------------------------------------------
namespace {

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn get_encode_fn() {
  static EncodeTiledFn fn = nullptr;
  if (fn) return fn;
  void* p = nullptr;
  cudaDriverEntryPointQueryResult qres;
  if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &qres) != cudaSuccess ||
      qres != cudaDriverEntryPointSuccess)
    return nullptr;
  fn = (EncodeTiledFn)p;
  return fn;
}

// bf16 tensor [T][H][D]; box = 64 columns x 1 head x `box_rows` tokens, 128-byte swizzle, zero fill.
int make_thd_map(CUtensorMap* m, const void* base, int64_t T, int H, int D, int box_rows) {
  EncodeTiledFn fn = get_encode_fn();
  if (!fn) {
    fcp_set_error("cuTensorMapEncodeTiled is not available from the driver");
    return FCP_ERR_CUDA;
  }
  if (((uintptr_t)base & 15) != 0) {
    fcp_set_error("tensor base %p is not 16-byte aligned", base);
    return FCP_ERR_INVALID_ARG;
  }
  const cuuint64_t dims[3] = {(cuuint64_t)D, (cuuint64_t)H, (cuuint64_t)T};
  const cuuint64_t strides[2] = {(cuuint64_t)D * 2, (cuuint64_t)H * D * 2};
  const cuuint32_t box[3] = {64, 1, (cuuint32_t)box_rows};
  const cuuint32_t estr[3] = {1, 1, 1};
  CUresult r = fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box, estr,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) {
    fcp_set_error("cuTensorMapEncodeTiled failed with %d", (int)r);
    return FCP_ERR_CUDA;
  }
  return FCP_OK;
}

// Launch that may begin while the kernel before it in the stream still runs (grid_begin of sm100_ptx.cuh); hides the
// launch latency and the set-up of barriers and tensor memory: 4K-token step, seven queue entries before and four launches now, 59 -> 50 us.
template <typename... P, typename... A>
cudaError_t launch_when(bool early, void (*kernel)(P...), dim3 grid, int threads, size_t smem, cudaStream_t st, A... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr = {};
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = early ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kernel, P(args)...);
}
template <typename... P, typename... A>
cudaError_t launch(void (*kernel)(P...), dim3 grid, int threads, size_t smem, cudaStream_t st, A... args) {
  return launch_when(true, kernel, grid, threads, smem, st, args...);
}

// Records an event pair around a kernel launch when the plan is in profiling mode.
struct ProfScope {
  const fcp_plan* plan;
  int kind;
  cudaStream_t st;
  int slot = -1;
  ProfScope(const fcp_plan* p, int k, cudaStream_t s) : plan(p), kind(k), st(s) {
    if (plan && plan->profiling && plan->prof_ev[kind][0][0]) {
      slot = (int)(plan->prof_n[kind] % 64);
      cudaEventRecord((cudaEvent_t)plan->prof_ev[kind][slot][0], st);
    }
  }
  ~ProfScope() {
    if (slot >= 0) {
      cudaEventRecord((cudaEvent_t)plan->prof_ev[kind][slot][1], st);
      ++plan->prof_n[kind];
    }
  }
};

int check_plan(const fcp_plan* plan) {
  if (!plan) {
    fcp_set_error("plan is NULL");
    return FCP_ERR_INVALID_ARG;
  }
  if (!plan->d_blob) {
    fcp_set_error("plan has no device copy: call fcp_plan_upload first");
    return FCP_ERR_NOT_UPLOADED;
  }
  return FCP_OK;
}

}  // namespace

// ---------------------------------------------------------------------------------------------
// LSE merge (HBM bound).  One thread owns 8 output columns of one (token, head) row: it reads the
// row's slot log-sum-exps, forms the exact weights and accumulates 2 x 128-bit loads per slot.
// ---------------------------------------------------------------------------------------------
template <int D>
__global__ void __launch_bounds__(256) fcp_merge_kernel(const int32_t* __restrict__ units, const int32_t* __restrict__ slot_offset,
                                                        const int32_t* __restrict__ slot_rows, const float* o_partial,
                                                        const float* lse_partial, int head_begin, int head_count,
                                                        int hq, __nv_bfloat16* __restrict__ o, float* __restrict__ o_f32, float* __restrict__ lse) {
  grid_begin();
  constexpr int TPR = D / 8;                 // threads per (token, head) row
  constexpr int RPP = 256 / TPR;             // rows per pass
  const int32_t* U = units + (size_t)blockIdx.x * FCP_MERGE_UNIT_W;
  const int tok0 = U[MU_TOK_BEGIN], ntok = U[MU_N_TOK], chunk = U[MU_CHUNK], ctok0 = U[MU_CHUNK_TOK_BEGIN];
  const int s0 = slot_offset[chunk], ns = slot_offset[chunk + 1] - s0;
  const int sub = threadIdx.x % TPR, rloc = threadIdx.x / TPR;
  const int n_rows = ntok * head_count;
  for (int r = rloc; r < n_rows; r += RPP) {
    const int t = tok0 + r / head_count, hl = r % head_count;
    const int64_t rel = t - ctok0;
    float m = -INFINITY;
    for (int s = 0; s < ns; ++s) m = fmaxf(m, ld_f32(lse_partial + ((int64_t)slot_rows[s0 + s] + rel) * head_count + hl));
    float z = 0.f;
    for (int s = 0; s < ns; ++s)
      z += __expf(ld_f32(lse_partial + ((int64_t)slot_rows[s0 + s] + rel) * head_count + hl) - m);
    const float L = m + __logf(z);
    float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    for (int s = 0; s < ns; ++s) {
      const int64_t prow = ((int64_t)slot_rows[s0 + s] + rel) * head_count + hl;
      const float wgt = __expf(ld_f32(lse_partial + prow) - L);
      const float* src = o_partial + prow * D + sub * 8;
      const float4 a0 = ld_stream_f4(src), a1 = ld_stream_f4(src + 4);
      acc[0] += wgt * a0.x; acc[1] += wgt * a0.y; acc[2] += wgt * a0.z; acc[3] += wgt * a0.w;
      acc[4] += wgt * a1.x; acc[5] += wgt * a1.y; acc[6] += wgt * a1.z; acc[7] += wgt * a1.w;
    }
    const int64_t orow = (int64_t)t * hq + head_begin + hl;
    uint4 pk;
    pk.x = pack_bf16(acc[0], acc[1]); pk.y = pack_bf16(acc[2], acc[3]);
    pk.z = pack_bf16(acc[4], acc[5]); pk.w = pack_bf16(acc[6], acc[7]);
    *reinterpret_cast<uint4*>(o + orow * D + sub * 8) = pk;
    if (o_f32) {
      float4* dst = reinterpret_cast<float4*>(o_f32 + orow * D + sub * 8);
      dst[0] = make_float4(acc[0], acc[1], acc[2], acc[3]);
      dst[1] = make_float4(acc[4], acc[5], acc[6], acc[7]);
    }
    if (sub == 0) lse[orow] = L;
  }
}

// ---------------------------------------------------------------------------------------------
// Backward preprocess (HBM bound): delta[h][t] = -scale * sum_c dO[t,h,c] * O[t,h,c], and minus the forward
// LSE transposed to [h][t] in log2 units, the layout the backward kernel's per-tile loads want.
// ---------------------------------------------------------------------------------------------
// It also clears the dQ accumulator and the work counter of the backward grid: the same bytes as a launch of its own would move
// (268 MB together with the reads on a 32-head 8K batch), but one launch fewer and beside the reads.  One CTA takes DELTA_TOKENS
// tokens of one head, so that the transposed statistics leave as whole sectors.  8K batch 43.6 us (6.2 TB/s), 64K batch
// 325 us (6.6 TB/s, the rate of a plain copy).
constexpr int DELTA_TOKENS = 64;
template <int D>
__global__ void __launch_bounds__(256) fcp_delta_kernel(const __nv_bfloat16* o, const __nv_bfloat16* d_o,
                                                        const float* lse, int64_t T, int hq, int h0, int hc,
                                                        int64_t t_stride, float scale, float* __restrict__ delta_t,
                                                        float* __restrict__ lse2_t, float* __restrict__ dq_acc,
                                                        int32_t* __restrict__ counter) {
  // heads [h0, h0 + hc) of the [T][hq][D] tensors; the outputs hold hc heads, numbered from 0
  grid_begin();
  constexpr int TPR = D / 8, RPP = 256 / TPR, N = DELTA_TOKENS / RPP;    // threads per row, rows per pass, passes
  if (blockIdx.x == 0 && threadIdx.x == 0) *counter = 0;
  const int hl = blockIdx.x % hc, sub = threadIdx.x % TPR;             // heads of a token block run together: they share DRAM pages
  const int64_t t0 = (int64_t)(blockIdx.x / hc) * DELTA_TOKENS + threadIdx.x / TPR;
  uint4 a[N], b[N];
#pragma unroll
  for (int i = 0; i < N; ++i) {
    const int64_t t = t0 + i * RPP;
    if (t < T) {
      const int64_t src = t * hq + h0 + hl;
      a[i] = ld_stream_v4(o + src * D + sub * 8);   // leaves the L2 to dO
      b[i] = ld_v4(d_o + src * D + sub * 8);
    } else {
      a[i] = b[i] = make_uint4(0, 0, 0, 0);
    }
  }
#pragma unroll
  for (int i = 0; i < N; ++i) {
    const int64_t t = t0 + i * RPP;
    if (t < T) {               // any order of the rows does: the whole accumulator is cleared
      float4* z = reinterpret_cast<float4*>(dq_acc + (t * hc + hl) * D);
      z[sub] = z[sub + TPR] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
  }
#pragma unroll
  for (int i = 0; i < N; ++i) {
    const int64_t t = t0 + i * RPP;
    const __nv_bfloat162* pa = reinterpret_cast<const __nv_bfloat162*>(&a[i]);
    const __nv_bfloat162* pb = reinterpret_cast<const __nv_bfloat162*>(&b[i]);
    float acc = 0.f;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float2 fa = __bfloat1622float2(pa[j]), fb = __bfloat1622float2(pb[j]);
      acc += fa.x * fb.x + fa.y * fb.y;
    }
#pragma unroll
    for (int off = TPR / 2; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
    if (t < T && sub == 0) delta_t[hl * t_stride + t] = -acc * scale;
  }
  const int64_t tl = t0 - threadIdx.x / TPR + threadIdx.x;               // a thread per row for the log-sum-exps
  if (threadIdx.x < DELTA_TOKENS && tl < T) lse2_t[hl * t_stride + tl] = ld_f32(lse + tl * hq + h0 + hl) * -1.4426950408889634f;
}

// fp32 dQ accumulator (tiles of dq_tile: [D / 4][rows][4]) -> bf16 dq [T][hq][D], heads from h0 on.  One CTA per (head,
// tile), all in one grid dimension (the others end at 65535): it reads rows * D contiguous floats with lanes along the rows and turns them round in shared memory, so
// that both sides move whole sectors.  Q tiles are cut like key tiles, so the backward units list them.
template <int D>
__global__ void __launch_bounds__(256) fcp_dq_convert_kernel(const float* acc, __nv_bfloat16* __restrict__ dq,
                                                             const int32_t* __restrict__ units, int n_units, int64_t T, int hq, int h0) {
  grid_begin();
  constexpr int PITCH = D + 8;                // bf16 elements per row in shared memory: 16 bytes of padding
  __shared__ __align__(16) __nv_bfloat16 tile[128 * PITCH];
  const int hl = blockIdx.x / n_units;
  const int32_t* U = units + (size_t)(blockIdx.x - hl * n_units) * FCP_BWD_UNIT_W;
  const int64_t t0 = __ldg(U + BU_KV_ROW0);
  const int rows = __ldg(U + BU_KV_ROWS);
  const float* src = acc + ((int64_t)hl * T + t0) * D;
  const int row = threadIdx.x & 127;
  if (row < rows) {
    constexpr int N = 8;                      // loads in flight per thread
#pragma unroll
    for (int c0 = 0; c0 < D / 4; c0 += 2 * N) {
      float4 v[N];
#pragma unroll
      for (int i = 0; i < N; ++i) v[i] = ld_stream_f4(src + ((c0 + 2 * i + (threadIdx.x >> 7)) * rows + row) * 4);
#pragma unroll
      for (int i = 0; i < N; ++i)
        *reinterpret_cast<uint2*>(tile + row * PITCH + (c0 + 2 * i + (threadIdx.x >> 7)) * 4) =
            make_uint2(pack_bf16(v[i].x, v[i].y), pack_bf16(v[i].z, v[i].w));
    }
  }
  __syncthreads();
  constexpr int TPR = D / 8;                  // threads per row, 16 bytes each
  __nv_bfloat16* dst = dq + ((t0 * hq) + h0 + hl) * (int64_t)D;
  for (int r = threadIdx.x / TPR; r < rows; r += 256 / TPR) {
    const int c = (threadIdx.x % TPR) * 8;
    *reinterpret_cast<uint4*>(dst + (int64_t)r * hq * D + c) = *reinterpret_cast<const uint4*>(tile + r * PITCH + c);
  }
}

// ---------------------------------------------------------------------------------------------
// Plan upload / destroy / status
// ---------------------------------------------------------------------------------------------
// Device blocks for the plans' tables.  Every new batch uploads a plan and drops the one before it, and cudaMalloc,
// cudaFree (which waits for the whole device), the device query and the kernel attributes cost milliseconds each time:
// with them a 16K-token batch takes 6.8 ms for 2.8 ms of kernels.  So a destroyed plan's block goes to a short list and
// is handed to the next plan once the event recorded after the last compute call that read it has completed.  The list
// holds at most 8 blocks and 32 MB; larger blocks are never kept, and fcp_release_cached gives all idle ones back.
// Three things still wait for queued work: an upload that finds the list full of blocks in use (for the oldest that
// fits), and, because cudaFree waits for the device, the release of a block that the list has no room for (one whose
// work is done goes first) and of the block of a plan that was captured into a graph.
// Memory, streams and kernel attributes belong to a CUDA context, so each context has a list of its own.
struct PlanPool;
struct PlanBlock {
  void* dev = nullptr;           // tables
  size_t bytes = 0;
  cudaEvent_t used = nullptr;    // after the last compute call that read the block
  PlanPool* pool = nullptr;
};

struct PlanPool {
  unsigned long long context = 0;
  std::mutex mu;                 // the members up to `staging`
  bool ready = false;            // device checked, attributes set, stream created
  int sm_count = 0;
  cudaStream_t copy = nullptr;   // uploads: complete without waiting for the work queued on the caller's stream
  std::vector<PlanBlock*> idle;  // oldest first
  size_t idle_bytes = 0;
  std::mutex staging_mu;         // one upload at a time passes its tables through `staging`
  char* staging = nullptr;
  bool staging_pinned = false;
};

namespace {
constexpr int kMaxDevices = 64;
constexpr size_t kBlockMin = size_t(64) << 10, kBlockKeepMax = size_t(8) << 20, kKeepBytes = size_t(32) << 20;
constexpr size_t kKeepBlocks = 8;
constexpr size_t kStagingBytes = size_t(1) << 20;

// The current context's pool.  Pools are never taken down: the id of a context is not used again.
int current_pool(PlanPool** out) {
  typedef CUresult (*CtxGetIdFn)(CUcontext, unsigned long long*);
  static CtxGetIdFn get_id = [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    return cudaGetDriverEntryPoint("cuCtxGetId", &p, cudaEnableDefault, &q) == cudaSuccess && q == cudaDriverEntryPointSuccess
               ? (CtxGetIdFn)p : nullptr;
  }();
  static std::mutex mu;
  static std::vector<PlanPool*>& pools = *new std::vector<PlanPool*>();
  unsigned long long id = 0;
  if (!get_id || get_id(nullptr, &id) != CUDA_SUCCESS) {
    FCP_CUDA_CHECK(cudaFree(nullptr));           // a thread without a context yet: the runtime makes the device's current
    if (!get_id || get_id(nullptr, &id) != CUDA_SUCCESS) {
      fcp_set_error("cuCtxGetId failed");
      return FCP_ERR_CUDA;
    }
  }
  std::lock_guard<std::mutex> lock(mu);
  for (PlanPool* p : pools)
    if (p->context == id) {
      *out = p;
      return FCP_OK;
    }
  pools.push_back(new PlanPool());
  pools.back()->context = id;
  *out = pools.back();
  return FCP_OK;
}

void free_block(PlanBlock* b) {
  if (b->dev) cudaFree(b->dev);
  if (b->used) cudaEventDestroy(b->used);
  delete b;
}

// Once per context: architecture check, shared-memory opt-in of the tensor-core kernels, the upload stream.
int pool_setup(PlanPool& pool) {
  if (pool.ready) return FCP_OK;
  int dev = 0, major = 0, sms = 0;
  FCP_CUDA_CHECK(cudaGetDevice(&dev));
  FCP_CUDA_CHECK(cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev));
  FCP_CUDA_CHECK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  if (major != 10) {
    fcp_set_error("device %d is not sm_100: this library is built for sm_100a only", dev);
    return FCP_ERR_CUDA;
  }
  FCP_CUDA_CHECK(cudaFuncSetAttribute(fcp_fwd_kernel<64>, cudaFuncAttributeMaxDynamicSharedMemorySize, FwdSmem<64>::DYN_BYTES));
  FCP_CUDA_CHECK(cudaFuncSetAttribute(fcp_fwd_kernel<128>, cudaFuncAttributeMaxDynamicSharedMemorySize, FwdSmem<128>::DYN_BYTES));
  FCP_CUDA_CHECK(cudaFuncSetAttribute(fcp_bwd_kernel<64>, cudaFuncAttributeMaxDynamicSharedMemorySize, BwdSmem<64>::DYN_BYTES));
  FCP_CUDA_CHECK(cudaFuncSetAttribute(fcp_bwd_kernel<128>, cudaFuncAttributeMaxDynamicSharedMemorySize, BwdSmem<128>::DYN_BYTES));
  FCP_CUDA_CHECK(cudaStreamCreateWithFlags(&pool.copy, cudaStreamNonBlocking));
  pool.sm_count = sms;
  pool.ready = true;
  return FCP_OK;
}

// Whether no queued work reads the block any more.  (cudaErrorNotReady is left behind as the thread's last error.)
bool is_free(const PlanBlock* b) {
  const cudaError_t e = cudaEventQuery(b->used);
  if (e != cudaSuccess) cudaGetLastError();
  return e == cudaSuccess;
}

// A block of at least `bytes`: the smallest idle one that fits and that no queued work reads any more; with a full list
// the oldest one that fits, whose event the caller then waits for (a new block would push out one in use, and freeing
// that waits for the whole device); else a new one.
int acquire_block(PlanPool& pool, size_t bytes, PlanBlock** out) {
  size_t best = pool.idle.size();
  for (size_t i = 0; i < pool.idle.size(); ++i) {
    PlanBlock* b = pool.idle[i];
    if (b->bytes >= bytes && (best == pool.idle.size() || b->bytes < pool.idle[best]->bytes) && is_free(b)) best = i;
  }
  if (best == pool.idle.size() && pool.idle.size() >= kKeepBlocks)
    for (best = 0; best < pool.idle.size() && pool.idle[best]->bytes < bytes;) ++best;
  if (best < pool.idle.size()) {
    *out = pool.idle[best];
    pool.idle_bytes -= (*out)->bytes;
    pool.idle.erase(pool.idle.begin() + best);
    return FCP_OK;
  }
  PlanBlock* b = new PlanBlock();
  b->pool = &pool;
  b->bytes = kBlockMin;
  while (b->bytes < bytes && b->bytes < kBlockKeepMax) b->bytes *= 2;
  b->bytes = std::max(b->bytes, bytes);
  cudaError_t e = cudaMalloc(&b->dev, b->bytes);
  if (e == cudaSuccess) e = cudaEventCreateWithFlags(&b->used, cudaEventDisableTiming);
  if (e != cudaSuccess) {
    free_block(b);
    fcp_set_error("plan upload failed: %s", cudaGetErrorString(e));
    return FCP_ERR_CUDA;
  }
  *out = b;
  return FCP_OK;
}

// `keep`: the event of the block covers all work that may still read it.  Otherwise (and for large blocks) the memory
// is freed, which waits for the device.
void return_block(PlanBlock* b, bool keep) {
  if (!keep || b->bytes > kBlockKeepMax) {
    free_block(b);
    return;
  }
  PlanPool& pool = *b->pool;
  std::vector<PlanBlock*> out;
  {
    std::lock_guard<std::mutex> lock(pool.mu);
    pool.idle.push_back(b);
    pool.idle_bytes += b->bytes;
    while (pool.idle.size() > kKeepBlocks || pool.idle_bytes > kKeepBytes) {
      size_t i = 0;              // the oldest whose work is done, else the oldest
      while (i < pool.idle.size() && !is_free(pool.idle[i])) ++i;
      if (i == pool.idle.size()) i = 0;
      out.push_back(pool.idle[i]);
      pool.idle_bytes -= pool.idle[i]->bytes;
      pool.idle.erase(pool.idle.begin() + i);
    }
  }
  for (PlanBlock* x : out) free_block(x);
}

// Host tables -> device, in pieces through the pool's page-locked buffer (a pageable one where that is not to be had): the
// pool keeps 1 MB of it, whatever the plans' number and sizes.  Complete on return.
struct Staging {
  PlanPool& pool;
  char* dst;                     // where the first byte of the buffer goes
  cudaEvent_t done;
  size_t fill = 0;
  cudaError_t flush() {
    if (fill == 0) return cudaSuccess;
    cudaError_t e = cudaMemcpyAsync(dst, pool.staging, fill, cudaMemcpyHostToDevice, pool.copy);
    if (e == cudaSuccess) e = cudaEventRecord(done, pool.copy);
    if (e == cudaSuccess) e = cudaEventSynchronize(done);
    dst += fill;
    fill = 0;
    return e;
  }
  cudaError_t put(const void* src, size_t bytes) {         // src NULL: zeros
    for (size_t i = 0; i < bytes;) {
      const size_t n = std::min(bytes - i, kStagingBytes - fill);
      if (src) memcpy(pool.staging + fill, (const char*)src + i, n);
      else memset(pool.staging + fill, 0, n);
      i += n;
      fill += n;
      if (fill == kStagingBytes)
        if (cudaError_t e = flush(); e != cudaSuccess) return e;
    }
    return cudaSuccess;
  }
};

// At the end of every compute call: the block is in use until the work queued so far on `st` is done (calls on one
// plan are stream-ordered, so the last event covers the earlier calls).  Work recorded into a graph can run at any later
// time: such a plan's block is never handed on.
void mark_used(const fcp_plan* plan, cudaStream_t st) {
  if (!plan->block) return;
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(st, &cs) != cudaSuccess || cs != cudaStreamCaptureStatusNone ||
      cudaEventRecord(plan->block->used, st) != cudaSuccess) {
    plan->block_pinned = true;
    cudaGetLastError();
  }
}
}  // namespace

extern "C" int fcp_release_cached(void) {
  PlanPool* pool = nullptr;
  int rc = current_pool(&pool);
  if (rc != FCP_OK) return rc;
  std::vector<PlanBlock*> out;
  {
    std::lock_guard<std::mutex> lock(pool->mu);
    out.swap(pool->idle);
    pool->idle_bytes = 0;
  }
  for (PlanBlock* b : out) free_block(b);
  std::lock_guard<std::mutex> lock(pool->staging_mu);
  if (pool->staging_pinned) cudaFreeHost(pool->staging);
  else free(pool->staging);
  pool->staging = nullptr;
  return FCP_OK;
}

extern "C" int fcp_plan_upload(fcp_plan* plan, void* stream) {
  (void)stream;                  // the call is complete when it returns, whatever is queued there
  if (!plan) return FCP_ERR_INVALID_ARG;
  if (plan->d_blob) return FCP_OK;
  PlanPool* pool = nullptr;
  int rc = current_pool(&pool);
  if (rc != FCP_OK) return rc;
  constexpr int NT = 13;
  const std::vector<int32_t>* tabs[NT] = {&plan->fwd_units, &plan->bwd_units, &plan->bwd_qranges, &plan->merge_units,
                                          &plan->slot_offset, &plan->slot_rows, &plan->bwd_work, &plan->fused_units,
                                          &plan->row_limit, &plan->first_query, &plan->fwd_groups, &plan->bwd_groups,
                                          &plan->fused_groups};
  size_t off[NT + 1];
  size_t total = 256;  // status words first
  for (int i = 0; i < NT; ++i) {
    off[i] = total;
    total += (tabs[i]->size() * 4 + 255) / 256 * 256;
  }
  off[NT] = total;
  PlanBlock* block = nullptr;
  {
    std::lock_guard<std::mutex> lock(pool->mu);
    rc = pool_setup(*pool);
    if (rc == FCP_OK) rc = acquire_block(*pool, total, &block);
    if (rc != FCP_OK) return rc;
    plan->sm_count = pool->sm_count;
  }
  cudaError_t e = cudaEventSynchronize(block->used);
  if (e == cudaSuccess) {
    std::lock_guard<std::mutex> lock(pool->staging_mu);
    if (!pool->staging) {
      pool->staging_pinned = cudaMallocHost((void**)&pool->staging, kStagingBytes) == cudaSuccess;
      if (!pool->staging_pinned) {
        cudaGetLastError();
        pool->staging = (char*)malloc(kStagingBytes);
      }
    }
    if (!pool->staging) e = cudaErrorMemoryAllocation;
    Staging up{*pool, (char*)block->dev, block->used};
    if (e == cudaSuccess) e = up.put(nullptr, 256);
    for (int i = 0; i < NT && e == cudaSuccess; ++i) {
      e = up.put(tabs[i]->data(), tabs[i]->size() * 4);
      if (e == cudaSuccess) e = up.put(nullptr, off[i + 1] - off[i] - tabs[i]->size() * 4);
    }
    if (e == cudaSuccess) e = up.flush();
  }
  if (e != cudaSuccess) {
    free_block(block);
    fcp_set_error("plan upload failed: %s", cudaGetErrorString(e));
    return FCP_ERR_CUDA;
  }
  void* blob = block->dev;
  plan->block = block;
  plan->block_pinned = false;
  plan->d_blob = blob;
  plan->d_status = (int32_t*)blob;
  plan->d_fwd_units = (int32_t*)((char*)blob + off[0]);
  plan->d_bwd_units = (int32_t*)((char*)blob + off[1]);
  plan->d_bwd_qranges = (int32_t*)((char*)blob + off[2]);
  plan->d_merge_units = (int32_t*)((char*)blob + off[3]);
  plan->d_slot_offset = (int32_t*)((char*)blob + off[4]);
  plan->d_slot_rows = (int32_t*)((char*)blob + off[5]);
  plan->d_bwd_work = (int32_t*)((char*)blob + off[6]);
  plan->d_fused_units = (int32_t*)((char*)blob + off[7]);
  plan->d_fwd_groups = (int32_t*)((char*)blob + off[10]);
  plan->d_bwd_groups = (int32_t*)((char*)blob + off[11]);
  plan->d_fused_groups = (int32_t*)((char*)blob + off[12]);
  plan->d_row_limit = plan->row_limit.empty() ? nullptr : (int32_t*)((char*)blob + off[8]);
  plan->d_first_query = plan->first_query.empty() ? nullptr : (int32_t*)((char*)blob + off[9]);
  return FCP_OK;
}

extern "C" int fcp_plan_set_profiling(fcp_plan* plan, int32_t enable) {
  if (!plan) return FCP_ERR_INVALID_ARG;
  for (int k = 0; k < FCP_KERNEL_KINDS; ++k) {
    plan->prof_n[k] = 0;
    for (int i = 0; i < 64; ++i)
      for (int e = 0; e < 2; ++e) {
        if (enable && !plan->prof_ev[k][i][e]) {
          cudaEvent_t ev;
          FCP_CUDA_CHECK(cudaEventCreate(&ev));
          plan->prof_ev[k][i][e] = ev;
        } else if (!enable && plan->prof_ev[k][i][e]) {
          cudaEventDestroy((cudaEvent_t)plan->prof_ev[k][i][e]);
          plan->prof_ev[k][i][e] = nullptr;
        }
      }
  }
  plan->profiling = enable != 0;
  return FCP_OK;
}

extern "C" int fcp_plan_kernel_ms(const fcp_plan* plan, int32_t kind, int32_t* launches, float* mean_ms) {
  if (!plan || kind < 0 || kind >= FCP_KERNEL_KINDS || !launches || !mean_ms) return FCP_ERR_INVALID_ARG;
  const int n = (int)std::min<int64_t>(plan->prof_n[kind], 64);
  double sum = 0.0;
  for (int i = 0; i < n; ++i) {
    float ms = 0.f;
    FCP_CUDA_CHECK(cudaEventElapsedTime(&ms, (cudaEvent_t)plan->prof_ev[kind][i][0], (cudaEvent_t)plan->prof_ev[kind][i][1]));
    sum += ms;
  }
  *launches = (int32_t)plan->prof_n[kind];
  *mean_ms = n ? (float)(sum / n) : 0.f;
  return FCP_OK;
}

extern "C" int fcp_plan_destroy(fcp_plan* plan) {
  if (!plan) return FCP_OK;
  for (HostCut& cut : plan->host_cuts) {
    for (fcp_plan* g : cut.groups) fcp_plan_destroy(g);
    for (void* e : cut.events) if (e) cudaEventDestroy((cudaEvent_t)e);
  }
  if (plan->host_in) cudaStreamDestroy((cudaStream_t)plan->host_in);
  if (plan->host_out) cudaStreamDestroy((cudaStream_t)plan->host_out);
  if (plan->host_lane) cudaStreamDestroy((cudaStream_t)plan->host_lane);
  plan->host_in = plan->host_out = plan->host_lane = nullptr;
  fcp_plan_set_profiling(plan, 0);
  if (plan->block) return_block(plan->block, !plan->block_pinned);
  delete plan;
  return FCP_OK;
}

extern "C" int fcp_last_device_status(const fcp_plan* plan, int32_t* status) {
  if (!status) return FCP_ERR_INVALID_ARG;
  int rc = check_plan(plan);
  if (rc != FCP_OK) return rc;
  FCP_CUDA_CHECK(cudaDeviceSynchronize());
  FCP_CUDA_CHECK(cudaMemcpy(status, plan->d_status, 4 * sizeof(int32_t), cudaMemcpyDeviceToHost));
  // kernels launched by the host entry point report into the status words of its sequence groups
  for (const HostCut& cut : plan->host_cuts)
    for (const fcp_plan* g : cut.groups) {
      if (status[0] != 0) break;
      FCP_CUDA_CHECK(cudaMemcpy(status, g->d_status, 4 * sizeof(int32_t), cudaMemcpyDeviceToHost));
    }
  return FCP_OK;
}

// scratch layout of fcp_attn_bwd: [dq fp32 accumulator T*hq*D] [delta_t hq*Tpad] [lse2_t hq*Tpad]
static inline int64_t bwd_tpad(int64_t T) { return (T + 255) / 256 * 256 + 256; }

extern "C" int fcp_plan_workspace_bytes(const fcp_plan* plan, int32_t heads_per_pass, int64_t* o_partial_bytes,
                                        int64_t* lse_partial_bytes, int64_t* bwd_scratch_bytes) {
  if (!plan || heads_per_pass <= 0 || heads_per_pass > plan->params.hq) {
    fcp_set_error("fcp_plan_workspace_bytes: invalid argument");
    return FCP_ERR_INVALID_ARG;
  }
  const int64_t D = plan->params.head_dim;
  if (o_partial_bytes) *o_partial_bytes = plan->R * heads_per_pass * D * 4;
  if (lse_partial_bytes) *lse_partial_bytes = plan->R * heads_per_pass * 4;
  if (bwd_scratch_bytes)
    *bwd_scratch_bytes = plan->T * plan->params.hq * D * 4 + 2 * bwd_tpad(plan->T) * plan->params.hq * 4;
  return FCP_OK;
}

// ---------------------------------------------------------------------------------------------
// Compute calls
// ---------------------------------------------------------------------------------------------
static int check_heads(const fcp_plan* plan, int head_begin, int head_count) {
  if (head_begin < 0 || head_count <= 0 || head_begin + head_count > plan->params.hq) {
    fcp_set_error("head range [%d, %d) outside [0, %d)", head_begin, head_begin + head_count, plan->params.hq);
    return FCP_ERR_INVALID_ARG;
  }
  return FCP_OK;
}

namespace {
// `fused`: run the merge-on-the-fly units (every row goes straight to o_direct / lse_direct, no partials).
// `lane`: which work counter of the plan to use (two calls that may overlap use different ones).
int launch_fwd(const fcp_plan* plan, const void* q, const void* k, const void* v, int32_t head_begin, int32_t head_count,
               float* o_partial, float* lse_partial, void* o_direct, float* lse_direct, float* o_f32_direct, bool fused,
               void* stream, int lane = 0) {
  int rc = check_plan(plan);
  if (rc != FCP_OK) return rc;
  if (!q || !k || !v || (!fused && (!o_partial || !lse_partial)) || (fused && (!o_direct || !lse_direct))) {
    fcp_set_error("forward attention: NULL buffer");
    return FCP_ERR_INVALID_ARG;
  }
  if ((rc = check_heads(plan, head_begin, head_count)) != FCP_OK) return rc;
  if (!fused && !plan->row_limit.empty()) {
    fcp_set_error("the per-item partial path (fcp_attn_fwd, fcp_attn_fwd_merged) is causal only; a plan with "
                  "bidirectional spans runs through fcp_attn_fwd_fused");
    return FCP_ERR_UNSUPPORTED;
  }
  const fcp_params& P = plan->params;
  CUtensorMap tq, tk, tv;
  if ((rc = make_thd_map(&tq, q, plan->T, P.hq, P.head_dim, 128)) != FCP_OK) return rc;
  if ((rc = make_thd_map(&tk, k, plan->T, P.hkv, P.head_dim, 128)) != FCP_OK) return rc;
  if ((rc = make_thd_map(&tv, v, plan->T, P.hkv, P.head_dim, 128)) != FCP_OK) return rc;
  FwdArgs a;
  a.units = fused ? plan->d_fused_units : plan->d_fwd_units;
  a.n_units = (int32_t)((fused ? plan->fused_units.size() : plan->fwd_units.size()) / FCP_FWD_UNIT_W);
  a.groups = fused ? plan->d_fused_groups : plan->d_fwd_groups;
  a.head_begin = head_begin;
  a.head_count = head_count;
  a.hq = P.hq;
  a.hkv = P.hkv;
  {
    const int g = P.hq / P.hkv;
    a.head_group = (head_begin % g == 0 && head_count % g == 0) ? g : 1;
  }
  a.scale_log2 = P.scale * 1.4426950408889634f;
  a.o_partial = o_partial;
  a.lse_partial = lse_partial;
  a.o_direct = (__nv_bfloat16*)o_direct;
  a.lse_direct = lse_direct;
  a.o_f32_direct = o_f32_direct;
  a.row_limit = fused ? plan->d_row_limit : nullptr;
  a.status = plan->d_status;
  if (head_count == P.hq && plan->sm_count == FCP_PLAN_SMS)
    a.split = fused ? plan->fused_split : plan->fwd_split;
  else
    a.split = split_units(fused ? plan->fused_units : plan->fwd_units, fused ? plan->fused_groups : plan->fwd_groups,
                          head_count / a.head_group, a.head_group, plan->sm_count);
  const int64_t n_work = (int64_t)a.n_units * head_count << a.split;
  if (n_work >= int64_t(1) << 31) {
    fcp_set_error("forward attention: %lld work items exceed the 2^31 limit", (long long)n_work);
    return FCP_ERR_INVALID_ARG;
  }
  const int grid = (int)std::min<int64_t>(n_work, plan->sm_count);
  if (grid == 0) return FCP_OK;
  cudaStream_t st = (cudaStream_t)stream;
  // the grid's work counter (status block: words 16 + 2 * lane backward, 17 + 2 * lane forward): zero from the upload on
  a.work_counter = plan->d_status + 17 + 2 * lane;
  ProfScope prof(plan, 0, st);
  if (P.head_dim == 128)
    FCP_CUDA_CHECK(launch(fcp_fwd_kernel<128>, grid, FWD_THREADS, FwdSmem<128>::DYN_BYTES, st, tq, tk, tv, a));
  else
    FCP_CUDA_CHECK(launch(fcp_fwd_kernel<64>, grid, FWD_THREADS, FwdSmem<64>::DYN_BYTES, st, tq, tk, tv, a));
  return FCP_OK;
}

int launch_merge(const fcp_plan* plan, const float* o_partial, const float* lse_partial, int32_t head_begin,
                 int32_t head_count, void* o, float* o_f32, float* lse, int n_units, void* stream) {
  const fcp_params& P = plan->params;
  if (n_units == 0) return FCP_OK;
  cudaStream_t st = (cudaStream_t)stream;
  ProfScope prof(plan, 1, st);
  // Launched early, the CTAs go to the first SMs that the forward grid leaves, eight to each, and a grid of few CTAs stays on
  // them (forward + merge, us, early against not; n CTAs): n = 60, 64 heads, D = 64: 327, 287; n = 112, 32 heads, D = 128: 163,
  // 144; n = 448: 389, 375; n = 665: 639, 630; n = 3584: 10570, 10440; where the merge is short the launch costs 1-2 us more.
  const bool early = n_units >= 4 * plan->sm_count;
  if (P.head_dim == 128)
    FCP_CUDA_CHECK(launch_when(early, fcp_merge_kernel<128>, n_units, 256, 0, st, plan->d_merge_units, plan->d_slot_offset, plan->d_slot_rows,
                          o_partial, lse_partial, head_begin, head_count, P.hq, (__nv_bfloat16*)o, o_f32, lse));
  else
    FCP_CUDA_CHECK(launch_when(early, fcp_merge_kernel<64>, n_units, 256, 0, st, plan->d_merge_units, plan->d_slot_offset, plan->d_slot_rows,
                          o_partial, lse_partial, head_begin, head_count, P.hq, (__nv_bfloat16*)o, o_f32, lse));
  FCP_CUDA_CHECK(cudaGetLastError());
  return FCP_OK;
}

// End of a compute call, also of one that failed half-way: part of its work may be queued.
int used(const fcp_plan* plan, void* stream, int rc) {
  if (plan) mark_used(plan, (cudaStream_t)stream);
  return rc;
}
}  // namespace

extern "C" int fcp_attn_fwd(const fcp_plan* plan, const void* q, const void* k, const void* v, int32_t head_begin,
                            int32_t head_count, float* o_partial, float* lse_partial, void* stream) {
  return used(plan, stream, launch_fwd(plan, q, k, v, head_begin, head_count, o_partial, lse_partial, nullptr, nullptr, nullptr, false, stream));
}

extern "C" int fcp_attn_fwd_fused(const fcp_plan* plan, const void* q, const void* k, const void* v, int32_t head_begin,
                                  int32_t head_count, void* o, float* o_f32, float* lse, void* stream) {
  return used(plan, stream, launch_fwd(plan, q, k, v, head_begin, head_count, nullptr, nullptr, o, lse, o_f32, true, stream));
}

extern "C" int fcp_attn_fwd_merged(const fcp_plan* plan, const void* q, const void* k, const void* v, int32_t head_begin,
                                   int32_t head_count, float* o_partial, float* lse_partial, void* o, float* lse,
                                   void* stream) {
  if (!o || !lse) {
    fcp_set_error("fcp_attn_fwd_merged: NULL output");
    return FCP_ERR_INVALID_ARG;
  }
  int rc = launch_fwd(plan, q, k, v, head_begin, head_count, o_partial, lse_partial, o, lse, nullptr, false, stream);
  if (rc == FCP_OK)
    rc = launch_merge(plan, o_partial, lse_partial, head_begin, head_count, o, nullptr, lse, plan->n_merge_multi, stream);
  return used(plan, stream, rc);
}

extern "C" int fcp_lse_merge(const fcp_plan* plan, const float* o_partial, const float* lse_partial,
                             int32_t head_begin, int32_t head_count, void* o, float* o_f32, float* lse,
                             void* stream) {
  int rc = check_plan(plan);
  if (rc != FCP_OK) return rc;
  if (!o_partial || !lse_partial || !o || !lse) {
    fcp_set_error("fcp_lse_merge: NULL buffer");
    return FCP_ERR_INVALID_ARG;
  }
  if ((rc = check_heads(plan, head_begin, head_count)) != FCP_OK) return rc;
  if (!plan->row_limit.empty()) {
    fcp_set_error("fcp_lse_merge: the per-item partial path is causal only; this plan has bidirectional spans");
    return FCP_ERR_UNSUPPORTED;
  }
  return used(plan, stream, launch_merge(plan, o_partial, lse_partial, head_begin, head_count, o, o_f32, lse,
                                         (int)(plan->merge_units.size() / FCP_MERGE_UNIT_W), stream));
}

namespace {
// Everything the backward launches need besides the caller's tensors: device tables, status words,
// work counter, SM count.  fcp_attn_bwd_heads takes them from the uploaded plan, fcp_attn_bwd_noalloc
// from the built-in arena.
struct BwdTables {
  const int32_t *units, *qranges, *order, *groups, *first_query;
  int32_t* status;
  int32_t* counter;
  int sm_count;
};

// scratch layout: [dq fp32 accumulator T*hc*D] [delta_t hc*Tpad] [lse2_t hc*Tpad], hc = query heads of the pass
int64_t bwd_scratch_need(const fcp_plan* plan, int kv_heads) {
  const int64_t hc = (int64_t)kv_heads * (plan->params.hq / plan->params.hkv);
  return plan->T * hc * plan->params.head_dim * 4 + 2 * bwd_tpad(plan->T) * hc * 4;
}

// Launches of one backward pass over KV heads [hk0, hk0 + hkc): clear + delta, main kernel, dQ conversion.
// `prof` may be NULL (no event timing).
int run_bwd(const fcp_plan* plan, const BwdTables& tb, const void* q, const void* k, const void* v, const void* o,
            const void* d_o, const float* lse, int hk0, int hkc, void* dq, void* dk, void* dv, void* scratch,
            const fcp_plan* prof, cudaStream_t st) {
  const fcp_params& P = plan->params;
  const int64_t T = plan->T, D = P.head_dim;
  const int g = P.hq / P.hkv;
  const int h0 = hk0 * g, hc = hkc * g;
  const int64_t tpad = bwd_tpad(T);
  float* dq_acc = (float*)scratch;
  float* delta_t = dq_acc + T * hc * D;
  float* lse2_t = delta_t + tpad * hc;
  int rc;
  {
    ProfScope ps(prof, 2, st);
    const unsigned grid = (unsigned)((T + DELTA_TOKENS - 1) / DELTA_TOKENS * hc);
    if (D == 128)
      FCP_CUDA_CHECK(launch(fcp_delta_kernel<128>, grid, 256, 0, st, (const __nv_bfloat16*)o, (const __nv_bfloat16*)d_o, lse, T, P.hq,
                            h0, hc, tpad, P.scale, delta_t, lse2_t, dq_acc, tb.counter));
    else
      FCP_CUDA_CHECK(launch(fcp_delta_kernel<64>, grid, 256, 0, st, (const __nv_bfloat16*)o, (const __nv_bfloat16*)d_o, lse, T, P.hq,
                            h0, hc, tpad, P.scale, delta_t, lse2_t, dq_acc, tb.counter));
  }
  CUtensorMap tq, tk, tv, tdo;
  if ((rc = make_thd_map(&tq, q, T, P.hq, (int)D, 128)) != FCP_OK) return rc;
  if ((rc = make_thd_map(&tk, k, T, P.hkv, (int)D, 128)) != FCP_OK) return rc;
  if ((rc = make_thd_map(&tv, v, T, P.hkv, (int)D, 128)) != FCP_OK) return rc;
  if ((rc = make_thd_map(&tdo, d_o, T, P.hq, (int)D, 128)) != FCP_OK) return rc;
  BwdArgs a;
  a.units = tb.units;
  a.qranges = tb.qranges;
  a.work = tb.order;
  a.groups = tb.groups;
  a.n_heads = hkc;
  const int32_t n_units = (int32_t)plan->bwd_work.size();
  a.n_work = n_units * hkc;
  a.counter = tb.counter;
  a.hq = P.hq;
  a.hkv = P.hkv;
  a.hk_begin = hk0;
  a.hq_acc = hc;
  a.T = T;
  a.t_stride = tpad;
  a.scale = P.scale;
  a.scale_log2 = P.scale * 1.4426950408889634f;
  a.delta_t = delta_t;
  a.lse2_t = lse2_t;
  a.dq_acc = dq_acc;
  a.first_query = tb.first_query;
  a.dk = (__nv_bfloat16*)dk;
  a.dv = (__nv_bfloat16*)dv;
  a.status = tb.status;
  const int grid = (int)std::min<int64_t>(a.n_work, tb.sm_count);
  if (grid > 0) {
    ProfScope ps(prof, 3, st);
    if (D == 128)
      FCP_CUDA_CHECK(launch(fcp_bwd_kernel<128>, grid, BWD_THREADS, BwdSmem<128>::DYN_BYTES, st, tq, tk, tv, tdo, a));
    else
      FCP_CUDA_CHECK(launch(fcp_bwd_kernel<64>, grid, BWD_THREADS, BwdSmem<64>::DYN_BYTES, st, tq, tk, tv, tdo, a));
  }
  {
    const unsigned grid_c = (unsigned)n_units * hc;
    ProfScope ps(prof, 4, st);
    if (D == 128)
      FCP_CUDA_CHECK(launch(fcp_dq_convert_kernel<128>, grid_c, 256, 0, st, dq_acc, (__nv_bfloat16*)dq, tb.units, n_units, T, P.hq, h0));
    else
      FCP_CUDA_CHECK(launch(fcp_dq_convert_kernel<64>, grid_c, 256, 0, st, dq_acc, (__nv_bfloat16*)dq, tb.units, n_units, T, P.hq, h0));
  }
  return FCP_OK;
}
}  // namespace

extern "C" int fcp_plan_bwd_scratch_bytes(const fcp_plan* plan, int32_t kv_head_count, int64_t* bytes) {
  if (!plan || !bytes || kv_head_count <= 0 || kv_head_count > plan->params.hkv) {
    fcp_set_error("fcp_plan_bwd_scratch_bytes: invalid argument");
    return FCP_ERR_INVALID_ARG;
  }
  *bytes = bwd_scratch_need(plan, kv_head_count);
  return FCP_OK;
}

namespace {
int bwd_heads(const fcp_plan* plan, const void* q, const void* k, const void* v, const void* o, const void* d_o, const float* lse,
              int32_t kv_head_begin, int32_t kv_head_count, void* dq, void* dk, void* dv, void* scratch, int64_t scratch_bytes,
              void* stream, int lane) {
  int rc = check_plan(plan);
  if (rc != FCP_OK) return rc;
  if (!q || !k || !v || !o || !d_o || !lse || !dq || !dk || !dv || !scratch) {
    fcp_set_error("fcp_attn_bwd: NULL buffer");
    return FCP_ERR_INVALID_ARG;
  }
  if (kv_head_begin < 0 || kv_head_count <= 0 || kv_head_begin + kv_head_count > plan->params.hkv) {
    fcp_set_error("KV head range [%d, %d) outside [0, %d)", kv_head_begin, kv_head_begin + kv_head_count, plan->params.hkv);
    return FCP_ERR_INVALID_ARG;
  }
  const int64_t need = bwd_scratch_need(plan, kv_head_count);
  if (scratch_bytes < need) {
    fcp_set_error("fcp_attn_bwd: scratch of %lld bytes, %lld needed", (long long)scratch_bytes, (long long)need);
    return FCP_ERR_WORKSPACE;
  }
  const BwdTables tb{plan->d_bwd_units, plan->d_bwd_qranges, plan->d_bwd_work, plan->d_bwd_groups, plan->d_first_query, plan->d_status,
                     plan->d_status + 16 + 2 * lane, plan->sm_count};
  return used(plan, stream, run_bwd(plan, tb, q, k, v, o, d_o, lse, kv_head_begin, kv_head_count, dq, dk, dv, scratch, plan,
                                    (cudaStream_t)stream));
}
}  // namespace

extern "C" int fcp_attn_bwd_heads(const fcp_plan* plan, const void* q, const void* k, const void* v, const void* o,
                                  const void* d_o, const float* lse, int32_t kv_head_begin, int32_t kv_head_count,
                                  void* dq, void* dk, void* dv, void* scratch, int64_t scratch_bytes, void* stream) {
  return bwd_heads(plan, q, k, v, o, d_o, lse, kv_head_begin, kv_head_count, dq, dk, dv, scratch, scratch_bytes, stream, 0);
}

extern "C" int fcp_attn_bwd(const fcp_plan* plan, const void* q, const void* k, const void* v, const void* o,
                            const void* d_o, const float* lse, void* dq, void* dk, void* dv, void* scratch,
                            int64_t scratch_bytes, void* stream) {
  if (!plan) {
    fcp_set_error("plan is NULL");
    return FCP_ERR_INVALID_ARG;
  }
  return fcp_attn_bwd_heads(plan, q, k, v, o, d_o, lse, 0, plan->params.hkv, dq, dk, dv, scratch, scratch_bytes, stream);
}

// ---------------------------------------------------------------------------------------------
// Whole path from host buffers
// ---------------------------------------------------------------------------------------------
namespace {
struct HostLayout {
  int64_t q, k, v, d_o, o, lse, dq, dk, dv, scratch, total;
};
inline int64_t al(int64_t x) { return (x + 255) / 256 * 256; }

HostLayout host_layout(const fcp_plan* plan) {
  const fcp_params& P = plan->params;
  const int64_t T = plan->T, D = P.head_dim;
  HostLayout L{};
  int64_t off = 0;
  auto take = [&](int64_t bytes) { int64_t o = off; off += al(bytes); return o; };
  L.q = take(T * P.hq * D * 2);
  L.k = take(T * P.hkv * D * 2);
  L.v = take(T * P.hkv * D * 2);
  L.d_o = take(T * P.hq * D * 2);
  L.o = take(T * P.hq * D * 2);
  L.lse = take(T * P.hq * 4);
  L.dq = take(T * P.hq * D * 2);
  L.dk = take(T * P.hkv * D * 2);
  L.dv = take(T * P.hkv * D * 2);
  L.scratch = take(bwd_scratch_need(plan, P.hkv));
  L.total = off;
  return L;
}
}  // namespace

extern "C" int fcp_host_workspace_bytes(const fcp_plan* plan, int64_t* bytes) {
  if (!plan || !bytes) return FCP_ERR_INVALID_ARG;
  *bytes = host_layout(plan).total;
  return FCP_OK;
}

namespace {
// How the host entry point cuts a batch: into passes over whole KV heads (strided slices, 2-D copies; these run at full
// PCIe speed down to 512 bytes per row, 48 of 55 GB/s with both directions busy, 42 at 256 bytes) and, to get to
// kHostSlices, into runs of consecutive sequences (packed tensors are token-major, so a run is one contiguous slice of
// every tensor) with a plan of their own.  About kHostSliceBytes of inputs per slice: what is not overlapped is the
// first slice's way in and the last one's way out (11K tokens of 4 heads, D = 64: 1.4 ms with slices of 32 MB, 1.0 with
// 8 MB; 32K tokens of 32/32 heads: 28.7 ms with 16 passes, 26.5 with 8 in two runs).  Heads come first because every
// pass has the same work; runs of a batch with one long sequence are as unequal as its sequences (32K tokens of 32/8
// heads, half of them one sequence: 23.0 ms with runs only, 17.5 now; the copies alone take 13.6).
constexpr int64_t kHostSliceBytes = int64_t(8) << 20;
//
// That is for batches whose copies take as long as their kernels.  Above kHostFlopsPerByte (kernels at 1000 TFLOP/s against
// input copies at 50 GB/s) the batch is cut by heads alone, into kHostSlices passes where it has as many heads: a run that
// is one long sequence ends with few units left, pass after pass, while a pass over the whole batch has short ones for
// that.  256K tokens with one of 128K, 98 000 flop/byte: 618 ms with runs, 585 without; 64K tokens of the 32/8-head
// log-normal batch, 4 800 flop/byte: 32.1 ms with, 33.2 without.
constexpr int64_t kHostSlices = 16, kHostPasses = 8, kHostFlopsPerByte = 20000;
// Where the copies decide and would be of narrow rows (below kHostNarrowFlops, query rows of a pass of at most kHostNarrowRow
// bytes; or below kHostCopyFlops at any width) and four even runs or more can be had (the longest sequence at most two of them),
// runs come first, up to kHostRuns of kHostRunTokens, and heads are cut only down to K/V rows of kHostRowBytes.  Heads first
// against this (ms, two GPUs where they differ): 32K tokens of 8/8 heads 8.1, 7.3; 64K of 12/4 heads, D = 64: 7.9, 7.2; 700
// sequences of 300 tokens, 32/8 heads: 104, 100; but 64K of 32/32 heads (5800 flop/byte): 50.9, 53.4 and 50.1, 49.5; 64K of 32/8
// heads (1024 bytes): 33.0, 33.9 and 32.5, 31.8.
constexpr int64_t kHostNarrowRow = 512, kHostNarrowFlops = 5000, kHostCopyFlops = 1000, kHostRowBytes = 1024;
constexpr int64_t kHostRuns = 8, kHostRunTokens = 8192;
// Slices with fewer backward units than this per SM take turns on two kernel lanes, so that one fills the SMs that the
// other's last units leave idle (30K tokens of 16/4 heads, D = 64, half a unit: 5.0 ms, one lane 6.7).  Larger ones fill the
// chip by themselves, and two at once share its L2 (384K sequence, 20 units: 8390 ms, one lane 8125; 128K sequence, 7 units:
// 625 and 609; 64K tokens, 2 units: both 32.9).
constexpr int64_t kHostLaneUnits = 4;

// Strided copies of pageable memory run at a fraction of the speed of contiguous ones, and copies wait for one another
// whatever the slices are: such buffers are cut into up to eight runs of at least 8192 tokens and not by heads (8K tokens of
// 32/8 heads: 37 ms by heads, 25 like this; 32K: 155, 104; 64K: 301, 204; 64K of 32/32 heads: 494, 345).

bool is_pageable(const void* p) {
  cudaPointerAttributes a;
  if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
    cudaGetLastError();
    return true;
  }
  return a.type == cudaMemoryTypeUnregistered;
}

// Builds the runs' plans and creates the streams and events the host entry point orders its work with; all of it belongs
// to the plan and is released by fcp_plan_destroy.
int build_host_cut(const fcp_plan* plan, bool pageable, void* stream) {
  HostCut& cut = plan->host_cuts[pageable];
  if (!cut.tok0.empty()) return FCP_OK;
  const int B = plan->B;
  const int64_t T = plan->T;
  const fcp_params& P = plan->params;
  const int64_t in_bytes = 2 * T * (P.hq + P.hkv) * P.head_dim * 2;
  const int64_t slices = std::max<int64_t>(1, std::min<int64_t>(kHostSlices, in_bytes / kHostSliceBytes));
  std::vector<int32_t> lens(B), degs(B);
  double flops = 0;
  for (int b = 0; b < B; ++b) {
    lens[b] = plan->cu_seqlens[b + 1] - plan->cu_seqlens[b];
    degs[b] = (plan->chunk_offset[b + 1] - plan->chunk_offset[b] - 1) / 2;
    flops += 7.0 * lens[b] * lens[b] * P.hq * P.head_dim;
  }
  const bool by_heads = flops > (double)kHostFlopsPerByte * in_bytes;
  const int64_t most = std::min<int64_t>(by_heads ? kHostSlices : kHostPasses, slices);
  int32_t passes = (int32_t)std::min<int64_t>(P.hkv, most);
  int want = by_heads ? 1 : (int)std::max<int64_t>(1, std::min<int64_t>(std::min<int64_t>(slices / passes, B), T / kHostRunTokens));
  const int64_t runs = std::min<int64_t>(std::min<int64_t>(kHostRuns, B), std::min<int64_t>(slices, T / kHostRunTokens));
  const int64_t q_row = (int64_t)P.hq / P.hkv * P.head_dim * 2;
  const bool copies = flops < (double)(q_row <= kHostNarrowRow ? kHostNarrowFlops : kHostCopyFlops) * in_bytes;
  if (copies && runs >= 4 && plan->max_seqlen * runs <= 2 * T) {
    const int64_t kv_row = (int64_t)P.hkv * P.head_dim * 2;
    passes = (int32_t)std::max<int64_t>(1, std::min<int64_t>(std::min<int64_t>(P.hkv, kv_row / kHostRowBytes), kHostSlices / runs));
    want = (int)runs;
  }
  if (pageable) {
    passes = 1;
    want = (int)std::max<int64_t>(1, std::min<int64_t>(std::min<int64_t>(kHostRuns, B), T / kHostRunTokens));
  }
  std::vector<fcp_plan*> groups;
  std::vector<int64_t> tok0;
  auto fail = [&](int rc) {
    for (fcp_plan* x : groups) fcp_plan_destroy(x);
    return rc;
  };
  int b0 = want > 1 ? 0 : B;                     // one run: the plan itself
  if (want == 1) tok0.push_back(0);
  for (int g = 0; g < want && b0 < B; ++g) {
    int b1 = b0 + 1;
    if (g == want - 1) {
      b1 = B;
    } else {
      const int64_t target = T * (g + 1) / want;
      while (b1 < B - (want - 1 - g) && plan->cu_seqlens[b1] < target) ++b1;
    }
    fcp_plan* sub = nullptr;
    int rc;
    if (plan->span_offset.empty()) {
      rc = fcp_plan_blocks(lens.data() + b0, degs.data() + b0, b1 - b0, &plan->params, &sub);
    } else {                                     // the run's spans, offsets counted from its first one
      std::vector<int32_t> so(b1 - b0 + 1);
      for (int b = b0; b <= b1; ++b) so[b - b0] = plan->span_offset[b] - plan->span_offset[b0];
      rc = fcp_plan_blocks_spans(lens.data() + b0, degs.data() + b0, b1 - b0, so.data(),
                                 plan->spans.data() + 2 * (size_t)plan->span_offset[b0], &plan->params, &sub);
    }
    if (rc == FCP_OK) rc = fcp_plan_upload(sub, stream);
    if (rc != FCP_OK) {
      if (sub) fcp_plan_destroy(sub);
      return fail(rc);
    }
    groups.push_back(sub);
    tok0.push_back(plan->cu_seqlens[b0]);
    b0 = b1;
  }
  tok0.push_back(T);
  const size_t total_passes = (tok0.size() - 1) * passes;
  // events: [0] start, [1] last copy out, [2] second lane done, then per (run, pass): q, k, v up; dO up; forward done; backward done
  std::vector<void*> ev(3 + 4 * total_passes, nullptr);
  cudaError_t e = cudaSuccess;
  for (void** st : {&plan->host_in, &plan->host_out, &plan->host_lane})
    if (!*st && e == cudaSuccess) {
      cudaStream_t x = nullptr;
      e = cudaStreamCreateWithFlags(&x, cudaStreamNonBlocking);
      *st = x;
    }
  for (size_t i = 0; i < ev.size() && e == cudaSuccess; ++i) {
    cudaEvent_t x = nullptr;
    e = cudaEventCreateWithFlags(&x, cudaEventDisableTiming);
    ev[i] = x;
  }
  if (e != cudaSuccess) {
    for (void* x : ev) if (x) cudaEventDestroy((cudaEvent_t)x);
    fcp_set_error("fcp_attn_fwd_bwd_host: creating copy streams failed: %s", cudaGetErrorString(e));
    return fail(FCP_ERR_CUDA);
  }
  cut.events = std::move(ev);
  cut.groups = std::move(groups);
  cut.tok0 = std::move(tok0);
  cut.passes = passes;
  return FCP_OK;
}

// On any early exit of the host entry point: wait for the copies and kernels already queued, so that
// nothing still writes into the caller's buffers after the call has returned an error.
struct HostDrain {
  cudaStream_t a, b, c, d;
  bool armed = true;
  ~HostDrain() {
    if (!armed) return;
    cudaStreamSynchronize(a);
    cudaStreamSynchronize(b);
    cudaStreamSynchronize(c);
    cudaStreamSynchronize(d);
  }
};
}  // namespace

extern "C" int fcp_attn_fwd_bwd_host(const fcp_plan* plan, const void* q_host, const void* k_host, const void* v_host,
                                     const void* d_o_host, void* o_host, float* lse_host, void* dq_host, void* dk_host,
                                     void* dv_host, void* workspace, int64_t workspace_bytes, void* stream) {
  int rc = check_plan(plan);
  if (rc != FCP_OK) return rc;
  if (!q_host || !k_host || !v_host || !d_o_host || !o_host || !lse_host || !dq_host || !dk_host || !dv_host ||
      !workspace) {
    fcp_set_error("fcp_attn_fwd_bwd_host: NULL buffer");
    return FCP_ERR_INVALID_ARG;
  }
  const HostLayout L = host_layout(plan);
  if (L.total > workspace_bytes) {
    fcp_set_error("fcp_attn_fwd_bwd_host: workspace of %lld bytes, %lld needed", (long long)workspace_bytes,
                  (long long)L.total);
    return FCP_ERR_WORKSPACE;
  }
  cudaStream_t st = (cudaStream_t)stream;
  bool pageable = false;
  for (const void* p : {q_host, k_host, v_host, d_o_host, (const void*)o_host, (const void*)lse_host, (const void*)dq_host,
                        (const void*)dk_host, (const void*)dv_host})
    pageable = pageable || is_pageable(p);
  if ((rc = build_host_cut(plan, pageable, stream)) != FCP_OK) return rc;
  const HostCut& cut = plan->host_cuts[pageable];
  const fcp_params& P = plan->params;
  const int64_t D = P.head_dim;
  const int64_t rq = (int64_t)P.hq * D * 2, rkv = (int64_t)P.hkv * D * 2, rl = (int64_t)P.hq * 4;   // bytes per token
  char* w = (char*)workspace;
  const int G = (int)cut.tok0.size() - 1;
  // Inputs of later slices come in (s_in) and results of earlier ones go out (s_out) while kernels run.  The kernels of
  // consecutive slices alternate between `stream` and a second lane where a slice has few work units.  Everything is
  // ordered after the work already queued on `stream` and is complete when this call returns.
  cudaStream_t s_in = (cudaStream_t)plan->host_in, s_out = (cudaStream_t)plan->host_out, s_lane = (cudaStream_t)plan->host_lane;
  auto EV = [&](int i) { return (cudaEvent_t)cut.events[i]; };
  // The forward pass of a slice needs q, k, v only: dO follows them and arrives while the forward kernel runs; o leaves
  // while the backward kernels run (they only read it), the log-sum-exps of a run when its last forward pass is done
  // (the few bytes per row of one pass would make a slow strided copy).
  struct Slice { int g, hk0, hkc, ev0; bool last; };
  std::vector<Slice> slices;
  const int per = (P.hkv + cut.passes - 1) / cut.passes;
  int64_t lane_scratch = 0, lane_units = 0;      // scratch and backward units of the largest slice
  {
    int ev0 = 3;
    for (int g = 0; g < G; ++g) {
      const fcp_plan* sub = cut.groups.empty() ? plan : cut.groups[g];
      lane_scratch = std::max(lane_scratch, al(bwd_scratch_need(sub, per)));
      lane_units = std::max(lane_units, (int64_t)(sub->bwd_units.size() / FCP_BWD_UNIT_W) * per);
      for (int hk0 = 0; hk0 < P.hkv; hk0 += per, ev0 += 4)
        slices.push_back(Slice{g, hk0, std::min(per, P.hkv - hk0), ev0, hk0 + per >= P.hkv});
    }
  }
  const bool two_lanes = slices.size() > 1 && lane_units < kHostLaneUnits * plan->sm_count && 2 * lane_scratch <= al(bwd_scratch_need(plan, P.hkv));
  const int gq = P.hq / P.hkv;
  HostDrain drain{s_in, s_out, st, s_lane};
  FCP_CUDA_CHECK(cudaEventRecord(EV(0), st));
  FCP_CUDA_CHECK(cudaStreamWaitEvent(s_in, EV(0), 0));
  FCP_CUDA_CHECK(cudaStreamWaitEvent(s_out, EV(0), 0));
  FCP_CUDA_CHECK(cudaStreamWaitEvent(s_lane, EV(0), 0));
  // copies of the heads [h0, h0 + hc) of nt token rows: width hc * bytes per head, pitch = the row of all heads
  auto copy_heads = [&](char* dst, const char* src, int64_t t0, int64_t nt, int64_t row_bytes, int64_t head_bytes, int h0, int hc,
                        cudaMemcpyKind kind, cudaStream_t cs) {
    return cudaMemcpy2DAsync(dst + t0 * row_bytes + h0 * head_bytes, (size_t)row_bytes, src + t0 * row_bytes + h0 * head_bytes,
                             (size_t)row_bytes, (size_t)(hc * head_bytes), (size_t)nt, kind, cs);
  };
  const int64_t hb = D * 2;   // bytes of one head of one token (bf16)
  for (const Slice& sl : slices) {
    const int64_t t0 = cut.tok0[sl.g], nt = cut.tok0[sl.g + 1] - t0;
    const int h0 = sl.hk0 * gq, hc = sl.hkc * gq;
    FCP_CUDA_CHECK(copy_heads(w + L.q, (const char*)q_host, t0, nt, rq, hb, h0, hc, cudaMemcpyHostToDevice, s_in));
    FCP_CUDA_CHECK(copy_heads(w + L.k, (const char*)k_host, t0, nt, rkv, hb, sl.hk0, sl.hkc, cudaMemcpyHostToDevice, s_in));
    FCP_CUDA_CHECK(copy_heads(w + L.v, (const char*)v_host, t0, nt, rkv, hb, sl.hk0, sl.hkc, cudaMemcpyHostToDevice, s_in));
    FCP_CUDA_CHECK(cudaEventRecord(EV(sl.ev0), s_in));
    FCP_CUDA_CHECK(copy_heads(w + L.d_o, (const char*)d_o_host, t0, nt, rq, hb, h0, hc, cudaMemcpyHostToDevice, s_in));
    FCP_CUDA_CHECK(cudaEventRecord(EV(sl.ev0 + 1), s_in));
  }
  for (size_t i = 0; i < slices.size(); ++i) {
    const Slice& sl = slices[i];
    const fcp_plan* sub = cut.groups.empty() ? plan : cut.groups[sl.g];
    const int lane = two_lanes ? (int)(i & 1) : 0;
    cudaStream_t sk = lane ? s_lane : st;
    const int64_t t0 = cut.tok0[sl.g], nt = cut.tok0[sl.g + 1] - t0;
    const int h0 = sl.hk0 * gq, hc = sl.hkc * gq;
    FCP_CUDA_CHECK(cudaStreamWaitEvent(sk, EV(sl.ev0), 0));
    if ((rc = launch_fwd(sub, w + L.q + t0 * rq, w + L.k + t0 * rkv, w + L.v + t0 * rkv, h0, hc, nullptr, nullptr, w + L.o + t0 * rq,
                         (float*)(w + L.lse + t0 * rl), nullptr, true, sk, lane)) != FCP_OK)
      return rc;
    FCP_CUDA_CHECK(cudaEventRecord(EV(sl.ev0 + 2), sk));
    FCP_CUDA_CHECK(cudaStreamWaitEvent(s_out, EV(sl.ev0 + 2), 0));
    FCP_CUDA_CHECK(copy_heads((char*)o_host, w + L.o, t0, nt, rq, hb, h0, hc, cudaMemcpyDeviceToHost, s_out));
    if (sl.last)
      FCP_CUDA_CHECK(cudaMemcpyAsync((char*)lse_host + t0 * rl, w + L.lse + t0 * rl, nt * rl, cudaMemcpyDeviceToHost, s_out));
    FCP_CUDA_CHECK(cudaStreamWaitEvent(sk, EV(sl.ev0 + 1), 0));
    if ((rc = bwd_heads(sub, w + L.q + t0 * rq, w + L.k + t0 * rkv, w + L.v + t0 * rkv, w + L.o + t0 * rq, w + L.d_o + t0 * rq,
                        (float*)(w + L.lse + t0 * rl), sl.hk0, sl.hkc, w + L.dq + t0 * rq, w + L.dk + t0 * rkv, w + L.dv + t0 * rkv,
                        w + L.scratch + lane * lane_scratch, bwd_scratch_need(sub, sl.hkc), sk, lane)) != FCP_OK)
      return rc;
    FCP_CUDA_CHECK(cudaEventRecord(EV(sl.ev0 + 3), sk));
    FCP_CUDA_CHECK(cudaStreamWaitEvent(s_out, EV(sl.ev0 + 3), 0));
    FCP_CUDA_CHECK(copy_heads((char*)dq_host, w + L.dq, t0, nt, rq, hb, h0, hc, cudaMemcpyDeviceToHost, s_out));
    FCP_CUDA_CHECK(copy_heads((char*)dk_host, w + L.dk, t0, nt, rkv, hb, sl.hk0, sl.hkc, cudaMemcpyDeviceToHost, s_out));
    FCP_CUDA_CHECK(copy_heads((char*)dv_host, w + L.dv, t0, nt, rkv, hb, sl.hk0, sl.hkc, cudaMemcpyDeviceToHost, s_out));
  }
  FCP_CUDA_CHECK(cudaEventRecord(EV(2), s_lane));
  FCP_CUDA_CHECK(cudaStreamWaitEvent(st, EV(2), 0));
  FCP_CUDA_CHECK(cudaEventRecord(EV(1), s_out));
  FCP_CUDA_CHECK(cudaStreamWaitEvent(st, EV(1), 0));
  for (const fcp_plan* sub : cut.groups) mark_used(sub, st);   // after both lanes
  mark_used(plan, st);
  FCP_CUDA_CHECK(cudaStreamSynchronize(st));
  drain.armed = false;
  return FCP_OK;
}

// ---------------------------------------------------------------------------------------------
// Backward pass for callers that must not allocate device memory
// ---------------------------------------------------------------------------------------------
// Everything the backward grid needs besides the caller's tensors lives in this one fixed array:
// status words and work counter, the plan's work tables, and the scratch of fcp_attn_bwd (fp32 dQ
// accumulator, delta and LSE rows).  Each GPU that loads the library carries the array until the
// process exits.  In host code `g_noalloc_arena` is only a handle for the runtime's symbol calls,
// never a device pointer: the address kernels may use comes from cudaGetSymbolAddress.
static __device__ __align__(256) unsigned char g_noalloc_arena[FCP_NOALLOC_MAX_BYTES];

namespace {
// The work groups of the backward list lie in the 256 bytes of the status words, from word 32 on: eight rows fit, and an arena
// of half a group's 64 MB of dQ rows (order_units of fcp_plan.cpp) holds batches of two at most, one and its tail.
constexpr int kNoallocGroupsWord = 32, kNoallocGroupsWords = 32;
unsigned char* g_noalloc_ptr[kMaxDevices] = {};   // device address of the arena, per device
int g_noalloc_sms[kMaxDevices] = {};

// One-time set-up for the current device: arena address, SM count, shared-memory opt-in of the
// backward kernel.  None of these allocates.
int noalloc_setup(int dev) {
  if (g_noalloc_ptr[dev]) return FCP_OK;
  void* p = nullptr;
  FCP_CUDA_CHECK(cudaGetSymbolAddress(&p, g_noalloc_arena));
  int sms = 0, major = 0;
  FCP_CUDA_CHECK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  FCP_CUDA_CHECK(cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev));
  if (major != 10) {
    fcp_set_error("device %d is not sm_100: this library is built for sm_100a only", dev);
    return FCP_ERR_CUDA;
  }
  FCP_CUDA_CHECK(cudaFuncSetAttribute(fcp_bwd_kernel<64>, cudaFuncAttributeMaxDynamicSharedMemorySize, BwdSmem<64>::DYN_BYTES));
  FCP_CUDA_CHECK(cudaFuncSetAttribute(fcp_bwd_kernel<128>, cudaFuncAttributeMaxDynamicSharedMemorySize, BwdSmem<128>::DYN_BYTES));
  g_noalloc_sms[dev] = sms;
  g_noalloc_ptr[dev] = (unsigned char*)p;
  return FCP_OK;
}
}  // namespace

extern "C" int fcp_noalloc_bytes_needed(const fcp_plan* plan, int64_t* bytes) {
  if (!plan || !bytes) return FCP_ERR_INVALID_ARG;
  int64_t scratch = 0;
  fcp_plan_workspace_bytes(plan, 1, nullptr, nullptr, &scratch);
  *bytes = 256 + al((int64_t)plan->bwd_units.size() * 4) + al((int64_t)plan->bwd_qranges.size() * 4) +
           al((int64_t)plan->bwd_work.size() * 4) + al(scratch);
  return FCP_OK;
}

extern "C" int fcp_attn_bwd_noalloc(const fcp_plan* plan, const void* q, const void* k, const void* v, const void* o,
                                    const void* d_o, const float* lse, void* dq, void* dk, void* dv, void* stream) {
  if (!plan || !q || !k || !v || !o || !d_o || !lse || !dq || !dk || !dv) {
    fcp_set_error("fcp_attn_bwd_noalloc: NULL argument");
    return FCP_ERR_INVALID_ARG;
  }
  if (!plan->first_query.empty()) {
    fcp_set_error("fcp_attn_bwd_noalloc: plans with bidirectional spans are not supported here; use fcp_attn_bwd");
    return FCP_ERR_UNSUPPORTED;
  }
  int64_t need = 0;
  fcp_noalloc_bytes_needed(plan, &need);
  if (need > (int64_t)FCP_NOALLOC_MAX_BYTES || plan->bwd_groups.size() > kNoallocGroupsWords) {
    fcp_set_error("fcp_attn_bwd_noalloc: this batch needs %lld bytes of scratch, the built-in arena holds %lld; "
                  "use fcp_attn_bwd with a caller-provided scratch buffer",
                  (long long)need, (long long)FCP_NOALLOC_MAX_BYTES);
    return FCP_ERR_WORKSPACE;
  }
  int dev = 0;
  FCP_CUDA_CHECK(cudaGetDevice(&dev));
  if (dev < 0 || dev >= kMaxDevices) {
    fcp_set_error("fcp_attn_bwd_noalloc: device index %d not supported", dev);
    return FCP_ERR_UNSUPPORTED;
  }
  int rc = noalloc_setup(dev);
  if (rc != FCP_OK) return rc;
  unsigned char* base = g_noalloc_ptr[dev];
  cudaStream_t st = (cudaStream_t)stream;
  const fcp_params& P = plan->params;

  // carve the arena: [status, counter, groups | units | qranges | work | scratch]
  int64_t off = 256;
  int32_t* d_status = (int32_t*)base;
  int32_t* d_units = (int32_t*)(base + off);    off += al((int64_t)plan->bwd_units.size() * 4);
  int32_t* d_qranges = (int32_t*)(base + off);  off += al((int64_t)plan->bwd_qranges.size() * 4);
  int32_t* d_work = (int32_t*)(base + off);     off += al((int64_t)plan->bwd_work.size() * 4);
  int32_t* d_groups = d_status + kNoallocGroupsWord;
  unsigned char* d_scratch = base + off;

  // the arena still holds the previous call's data: status, work counter and the dQ accumulator
  // must start at zero (the first kernel of run_bwd clears the last two); the tables are rewritten from the plan's host copy
  FCP_CUDA_CHECK(cudaMemsetAsync(d_status, 0, 256, st));
  if (!plan->bwd_units.empty())
    FCP_CUDA_CHECK(cudaMemcpyAsync(d_units, plan->bwd_units.data(), plan->bwd_units.size() * 4, cudaMemcpyHostToDevice, st));
  if (!plan->bwd_qranges.empty())
    FCP_CUDA_CHECK(cudaMemcpyAsync(d_qranges, plan->bwd_qranges.data(), plan->bwd_qranges.size() * 4, cudaMemcpyHostToDevice, st));
  if (!plan->bwd_work.empty())
    FCP_CUDA_CHECK(cudaMemcpyAsync(d_work, plan->bwd_work.data(), plan->bwd_work.size() * 4, cudaMemcpyHostToDevice, st));

  if (!plan->bwd_groups.empty())
    FCP_CUDA_CHECK(cudaMemcpyAsync(d_groups, plan->bwd_groups.data(), plan->bwd_groups.size() * 4, cudaMemcpyHostToDevice, st));

  const BwdTables tb{d_units, d_qranges, d_work, d_groups, nullptr, d_status, d_status + 16, g_noalloc_sms[dev]};
  return run_bwd(plan, tb, q, k, v, o, d_o, lse, 0, P.hkv, dq, dk, dv, d_scratch, nullptr, st);
}

extern "C" int fcp_noalloc_device_status(int32_t* status) {
  if (!status) return FCP_ERR_INVALID_ARG;
  int dev = 0;
  FCP_CUDA_CHECK(cudaGetDevice(&dev));
  if (dev < 0 || dev >= kMaxDevices || !g_noalloc_ptr[dev]) {
    fcp_set_error("fcp_noalloc_device_status: fcp_attn_bwd_noalloc has not run on this device");
    return FCP_ERR_INVALID_ARG;
  }
  FCP_CUDA_CHECK(cudaDeviceSynchronize());
  FCP_CUDA_CHECK(cudaMemcpy(status, g_noalloc_ptr[dev], 4 * sizeof(int32_t), cudaMemcpyDeviceToHost));
  return FCP_OK;
}

// ---------------------------------------------------------------------------------------------
// Self-test of the bounded device-side wait
// ---------------------------------------------------------------------------------------------
// One CTA of one warp; lane 0 waits, through the same mbar_wait / wait_teardown the persistent kernels
// use, on a barrier that nobody will ever arrive at.  The wait limit is an argument (a millisecond or
// so instead of the kernels' two seconds), so the launch ends by itself after about that long.  The
// status words are a device array of their own: no plan is involved and none is marked as failed.
static __device__ int32_t g_wait_probe_status[4];

__global__ void __launch_bounds__(32) fcp_wait_probe_kernel(uint32_t limit_ns, int where) {
  __shared__ __align__(8) unsigned long long bar;
  __shared__ int abort_flag;
  const uint32_t b = smem_u32(&bar);
  if (threadIdx.x == 0) {
    abort_flag = 0;
    mbar_init(b, 1);
    fence_mbar_init();
  }
  __syncwarp();
  const WaitCtx ctx{&abort_flag, g_wait_probe_status, limit_ns};
  if (threadIdx.x == 0) (void)mbar_wait(b, 0, ctx, where);     // phase 0 never completes
  __syncwarp();
  wait_teardown(ctx);
}

extern "C" int fcp_selftest_bounded_wait(uint32_t limit_us, int32_t* status, void* stream) {
  if (!status || limit_us == 0 || limit_us > 100000u) {
    fcp_set_error("fcp_selftest_bounded_wait: status is NULL or the limit is outside [1, 100000] microseconds");
    return FCP_ERR_INVALID_ARG;
  }
  cudaStream_t st = (cudaStream_t)stream;
  void* dst = nullptr;
  FCP_CUDA_CHECK(cudaGetSymbolAddress(&dst, g_wait_probe_status));
  FCP_CUDA_CHECK(cudaMemsetAsync(dst, 0, 4 * sizeof(int32_t), st));
  fcp_wait_probe_kernel<<<1, 32, 0, st>>>(limit_us * 1000u, 901);
  FCP_CUDA_CHECK(cudaGetLastError());
  FCP_CUDA_CHECK(cudaMemcpyAsync(status, dst, 4 * sizeof(int32_t), cudaMemcpyDeviceToHost, st));
  FCP_CUDA_CHECK(cudaStreamSynchronize(st));
  return FCP_OK;
}
