// Internal declarations shared by the CUDA translation units of the decode tail.
#pragma once

#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <stdint.h>
#include <math.h>
#include <atomic>
#include <mutex>
#include <utility>
#include <vector>

#include "../../include/brisk.h"

namespace brisk {

constexpr unsigned FULL_MASK = 0xffffffffu;
constexpr float LOG2E = 1.4426950408889634f;   // log2(e): exp(x) = 2^(x log2 e)
constexpr int INVALID_ID = 0x7fffffff;
constexpr float RESID_Z_FLOOR = 1e-6f;         // residual mass below which the verifier argmax is used

// ---------------------------------------------------------------- element access
__device__ __forceinline__ float to_f32(float x) { return x; }
__device__ __forceinline__ float to_f32(__nv_bfloat16 x) { return __bfloat162float(x); }

template <typename T> struct Vec;   // 16-byte vector of T
template <> struct Vec<float> { static constexpr int N = 4; };
template <> struct Vec<__nv_bfloat16> { static constexpr int N = 8; };

// Streaming 16-byte load that skips L1 allocation (each logit is read once).
__device__ __forceinline__ uint4 ld_stream_v4(const void* p) {
  uint4 r;
  asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];"
               : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w) : "l"(p));
  return r;
}

__device__ __forceinline__ void unpack(const uint4& w, float (&f)[8], __nv_bfloat16) {
  const uint32_t u[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    f[2 * j] = __uint_as_float(u[j] << 16);
    f[2 * j + 1] = __uint_as_float(u[j] & 0xffff0000u);
  }
}
__device__ __forceinline__ void unpack(const uint4& w, float (&f)[4], float) {
  f[0] = __uint_as_float(w.x);
  f[1] = __uint_as_float(w.y);
  f[2] = __uint_as_float(w.z);
  f[3] = __uint_as_float(w.w);
}

// Hardware base-2 exponential (MUFU), flushes subnormal results to zero.
__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// ---------------------------------------------------------------- ordering
// Candidate order of the method: logit descending, then id ascending.
__device__ __forceinline__ bool better(float v1, int i1, float v2, int i2) {
  return v1 > v2 || (v1 == v2 && i1 < i2);
}

__device__ __forceinline__ float warp_sum(float x) {
#pragma unroll
  for (int off = 16; off; off >>= 1) x += __shfl_xor_sync(FULL_MASK, x, off);
  return x;
}
__device__ __forceinline__ float warp_max(float x) {
#pragma unroll
  for (int off = 16; off; off >>= 1) x = fmaxf(x, __shfl_xor_sync(FULL_MASK, x, off));
  return x;
}

// Combine per-lane (max, sum of exp(x - max)) pairs into the warp's pair.
__device__ __forceinline__ void warp_lse_combine(float& m, float& s) {
  const float M = warp_max(m);
  float t = (m == -INFINITY) ? 0.f : s * ex2((m - M) * LOG2E);
  t = warp_sum(t);
  m = M;
  s = t;
}

// ---------------------------------------------------------------- contexts
// Unique id of the CUDA context current on this thread (cuCtxGetId; ids are never reused, so a
// device reset, which creates a new context, gives a new id). False when no context is current
// or the driver entry points are unavailable.
bool current_context_id(unsigned long long* id);

// Shared-memory carveouts (KB) the kernels ask for. An SM cannot change its L1/shared split
// while a CTA is resident, and the first kernel to land on an idle SM sets it, so a kernel that
// runs beside another one (the sweep beside the dense products, the verifier-row sweep beside
// the corrector) must leave room in its split for the other's CTAs. Everything not carved out
// is L1, which holds the sweep's loads in flight. Sweeps of 128 x 32 x 126464 alone with 32, 64,
// 100, 132 and 164 KB: 168, 168, 166, 174, 189 us proposal rows; a decode tail of them with 64,
// 100, 132 KB: 395, 381, 389 us.
constexpr int CARVEOUT_SMALL_KB = 100;   // sweep (5.5 KB a CTA), corrector, verification
constexpr int CARVEOUT_FULL_KB = 228;    // dense products, except beside the sweeps
// Prepares `func` in the current context, once: its carveout preference and, for a kernel with dynamic
// shared memory, the most that a block of it may have (process-wide state that another thread's call
// must not lower between this one's and its launch). cudaErrorInvalidValue if `smem` bytes do not fit.
inline cudaError_t set_up_kernel_fn(const void* func, int kb, size_t smem) {
  struct Entry { const void* func; unsigned long long ctx; size_t most; };
  static std::mutex mu;
  static std::vector<Entry> done;
  std::lock_guard<std::mutex> lock(mu);
  unsigned long long ctx = 0;
  const bool known = current_context_id(&ctx);   // (a device reset makes a new context)
  for (const auto& d : done)
    if (known && d.func == func && d.ctx == ctx) return smem <= d.most ? cudaSuccess : cudaErrorInvalidValue;
  int dev = 0, per_sm = 0, per_block = 0;
  cudaFuncAttributes fa;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, func);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&per_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&per_block, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (e != cudaSuccess) return e;
  int pct = per_sm > 0 ? (kb * 1024 * 100 + per_sm - 1) / per_sm : 100;
  if (pct > 100) pct = 100;
  e = cudaFuncSetAttribute(func, cudaFuncAttributePreferredSharedMemoryCarveout, pct);
  const size_t most = smem > 0 ? (size_t)per_block - fa.sharedSizeBytes : 0;
  if (e == cudaSuccess && smem > 0)
    e = cudaFuncSetAttribute(func, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most);
  if (e != cudaSuccess) return e;
  if (known) done.push_back({func, ctx, most});
  return smem <= most ? cudaSuccess : cudaErrorInvalidValue;
}

template <typename Kernel>
inline cudaError_t set_up_kernel(Kernel kernel, int kb, size_t smem = 0) {
  return set_up_kernel_fn(reinterpret_cast<const void*>(kernel), kb, smem);
}

// ---------------------------------------------------------------- mbarriers and bulk copies
// Bounded waits: a wait gives up after a limit of SM cycles (wait_limit_cycles(), set by
// brisk_set_wait_limit and passed to kernels as an argument); the drain of copies still in
// flight after a give-up is bounded by the default limit.
constexpr long long DRAIN_LIMIT_CYCLES = 4000000000ll;  // about 2 s of SM clock
constexpr long long SHORT_WAIT_CYCLES = 1ll << 20;      // below this, waits poll without suspending
long long wait_limit_cycles();

__device__ __forceinline__ uint32_t su32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(su32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(su32(bar)), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(su32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
// Non-blocking test of the phase with the given parity (never suspends the thread).
__device__ __forceinline__ bool mbar_test(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(su32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
// Wait for a phase that is known to complete (the drain after a give-up), bounded by the
// default limit.
__device__ __forceinline__ void mbar_drain(uint64_t* bar, uint32_t parity) {
  const long long t0 = clock64();
  while (!mbar_try_wait(bar, parity) && clock64() - t0 < DRAIN_LIMIT_CYCLES) {
  }
}
// Orders this thread's earlier shared-memory accesses before later async-proxy (TMA, bulk copy)
// accesses of the same memory.
__device__ __forceinline__ void fence_async_smem() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
// Launches `kernel` with the priority of `stream` as a launch attribute. Kernel nodes captured
// into a CUDA graph keep launch attributes, but not the priority of the stream they were captured
// from, so without it a replay of the tail's three-priority schedule runs every kernel at the
// default priority.
// With cluster > 1 the grid runs as clusters of that many CTAs. `started`, if not null, is recorded
// to fire once all of them have begun.
template <typename... KArgs, typename... Args>
inline cudaError_t launch_started(cudaEvent_t started, void (*kernel)(KArgs...), dim3 grid, dim3 block,
                                  size_t smem, cudaStream_t stream, int cluster, Args&&... args) {
  int prio = 0;
  cudaError_t e = cudaStreamGetPriority(stream, &prio);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[3];
  attr[0].id = cudaLaunchAttributePriority;
  attr[0].val.priority = prio;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if (cluster > 1) {
    cudaLaunchAttribute& c = attr[cfg.numAttrs++];
    c.id = cudaLaunchAttributeClusterDimension;
    c.val.clusterDim.x = (unsigned)cluster;
    c.val.clusterDim.y = c.val.clusterDim.z = 1;
  }
  if (started) {
    cudaLaunchAttribute& c = attr[cfg.numAttrs++];
    c.id = cudaLaunchAttributeLaunchCompletionEvent;
    c.val.launchCompletionEvent.event = started;
    c.val.launchCompletionEvent.flags = 0;
  }
  return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}
template <typename... KArgs, typename... Args>
inline cudaError_t launch_cluster(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem,
                                  cudaStream_t stream, int cluster, Args&&... args) {
  return launch_started(nullptr, kernel, grid, block, smem, stream, cluster,
                        std::forward<Args>(args)...);
}
template <typename... KArgs, typename... Args>
inline cudaError_t launch_prio(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem,
                               cudaStream_t stream, Args&&... args) {
  return launch_cluster(kernel, grid, block, smem, stream, 1, std::forward<Args>(args)...);
}

// Every thread of every CTA of the cluster arrives; writes before it are visible after it. (The
// barrier wants its warps whole, which a loop whose lanes leave it in turn does not promise.)
__device__ __forceinline__ void cluster_sync() {
  __syncwarp();
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" :::
               "memory");
}
// 16 bytes at this CTA's shared address p, in the shared memory of CTA `rank` of the cluster.
__device__ __forceinline__ float4 ld_cluster(const float* p, unsigned rank) {
  uint32_t addr;
  float4 v;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(addr) : "r"(su32(p)), "r"(rank));
  asm volatile("ld.shared::cluster.v4.f32 {%0,%1,%2,%3}, [%4];"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
               : "r"(addr)
               : "memory");
  return v;
}

// Stores x at this CTA's shared address p, in the shared memory of CTA `rank` of the cluster.
__device__ __forceinline__ void st_cluster(float* p, unsigned rank, float x) {
  uint32_t addr;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(addr) : "r"(su32(p)), "r"(rank));
  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(addr), "f"(x) : "memory");
}
// Sum, in rank order, of the 16 bytes at this CTA's shared address p in the first n (at most 8)
// CTAs of the cluster, all loads in flight at once.
__device__ __forceinline__ float4 sum_cluster(const float* p, int n) {
  float4 v[8];
#pragma unroll
  for (int o = 0; o < 8; ++o)
    if (o < n) v[o] = ld_cluster(p, o);
  float4 t = v[0];
#pragma unroll
  for (int o = 1; o < 8; ++o)
    if (o < n) {
      t.x += v[o].x; t.y += v[o].y; t.z += v[o].z; t.w += v[o].w;
    }
  return t;
}

__device__ __forceinline__ void set_status(int32_t* status, int code) {
  if (status) atomicCAS(status, 0, code);
}

__device__ __forceinline__ float sigmoidf_(float x) { return 1.f / (1.f + expf(-x)); }

// ---------------------------------------------------------------- sweep
struct SweepSeg {
  const void* logits;     // [rows, V]
  int rows;               // rows in this segment
  int kout;               // entries to output per row (K for proposal rows, 1 for verifier rows)
  int32_t* out_ids;       // [rows, kout]
  float* out_logprob;     // [rows, kout] or nullptr
  float* out_lse;         // [rows]
  float* part_val;        // [rows, nsplit, KP]
  int32_t* part_id;       // [rows, nsplit, KP]
  float* part_m;          // [rows, nsplit]
  float* part_s;          // [rows, nsplit]
  int32_t* counters;      // [rows]
};

struct SweepLaunch {
  SweepSeg seg[2];
  int nseg;
  int V;
  int nsplit;             // segments (CTAs) per row; 1 where a warp sweeps a row
  int KP;
  int dtype;              // brisk_dtype of the logits
  int32_t* status;
};

int sweep_splits(int rows_per_tensor, int V, int dtype, int K);
int kp_for(int K);
cudaError_t launch_sweep(const SweepLaunch& a, cudaStream_t stream);

// ---------------------------------------------------------------- dense products (SIMT, fp32 accumulate)
// C[m, n] = sum_k A(m, k) B(n, k) (+ bias[m % bias_period][n]), A(m,k) = A[m*lda + k],
// B(n,k) = transB ? B[k*ldb + n] : B[n*ldb + k]. call_rows: the most rows of a product of the call.
cudaError_t gemm_simt(int M, int N, int K, const void* A, int a_dt, int lda, const void* B,
                      int b_dt, int ldb, bool transB, float* C, int ldc, cudaStream_t stream,
                      const float* bias = nullptr, int bias_period = 1,
                      int call_rows = 0x7fffffff);
// Tensor-core product on sm_103a: C = A B^T with A [M, K] and B [N, K] bf16 (row strides lda, ldb),
// fp32 accumulation; mode 0 stores fp32 C[m*ldc + n], mode 1 stores three bf16 parts whose sum
// is c to about 2^-24 relative (hi at [m*ldc + n], mid at [m*ldc + N + n], lo at [m*ldc + 2N + n]).
// Up to two independent products of the same kind in one launch.
struct TcSpec {
  int M, N, K;
  const void* A;
  int lda;
  const void* B;
  int ldb;
  int mode;
  void* C;
  int ldc;
  const float* bias;   // optional fp32 [bias_period, N] added to row m as bias[m % bias_period] (mode 0)
  int bias_period;
};
// beside: the products run beside the sweeps and should share SMs with them (the results are the
// same bit for bit). started: recorded to fire once every CTA has begun.
cudaError_t gemm_tc_grouped(const TcSpec* spec, int nprob, int32_t* status, cudaStream_t stream,
                            bool beside = false, cudaEvent_t started = nullptr);
bool gemm_tc_supported(const void* A, int lda, const void* B, int ldb, int K);
// The folds that read the corrector's weights alone, in one launch: see brisk_corrector_prepare.
struct PackArgs {
  int L, r, dt;                  // dt: brisk_dtype of the weights
  const void *Wz, *Wh, *W0, *W_s, *w_g, *pos, *P_phi;
  float *W2, *W0h, *wg, *posG, *Fz, *Fh;
  // bf16 blocks written three times along k (bf16 weights only)
  __nv_bfloat16 *W2s, *W0s, *Wt2s, *W0ts, *Ws3;
};
cudaError_t pack_weights(const PackArgs& a, cudaStream_t stream);

// ---------------------------------------------------------------- corrector scan and verify
struct ScanArgs {
  int B, L, V, K, S, logits_dt;
  int select_mode, verify_mode;
  int do_select, do_verify;
  // corrector inputs
  const void* logits_q;
  const int32_t* cand_ids;
  const float* cand_logprob;
  const int32_t* x0;
  const float* u_sel;
  const float* G;        // [B*L, 2S] hidden and position shares of the GRU pre-activations (z | h)
  const float* G0;       // [B, S]    hidden-state part of Init
  const float* Tzh;      // [V, 2S]   token part of the GRU pre-activations (z | h)
  const float* U;        // [V, S]    residual rows: d = <s, U[c]>
  const float* T0;       // [V, S]    token part of Init

  const float* Fz;       // [S, 5]
  const float* Fh;       // [S, 5]
  const float* wg;       // [S + 5]
  float b_g, alpha;
  // same-state replay (App. B): feed the base selection forward instead of the head's, and
  // record its rank
  int base_prefix;
  int32_t* base_rank;    // [B, L] (base_prefix only)
  int beside_sweep;      // the corrector runs beside the verifier-row sweep
  // set by the launch (see corrector_kernel)
  int ring_depth, tok_ranks, ask_rows;
  int parts;             // CTAs that share a verification's residual walk
  long long wait_limit;
  // select outputs (or verify inputs when do_select == 0)
  int32_t* sel_tokens;   // [B, L]
  float* refined;        // [B, L, K]
  // verify inputs / outputs
  const void* logits_p;
  const int32_t* argmax_p;  // [B, L]
  const float* lse_p;       // [B, L]
  const float* u_acc;
  const float* u_res;
  int32_t* accepted_len;
  int32_t* out_tokens;
  int32_t* correction;
  int32_t* next_anchor;
  int32_t* status;
};

// ---------------------------------------------------------------- distillation loss
struct DistillArgs {
  int B, L, V, K, logits_dt;
  const void* logits_p;        // [B, L, V] verifier logits
  const int32_t* cand_ids;     // [B, L, K]
  const float* cand_logprob;   // [B, L, K]
  const float* refined;        // [B, L, K]
  const int32_t* accepted_len; // [B]
  float beta;
  float* loss;                 // [1]
  float* grad;                 // [B, L, K] or nullptr
  float* partial;              // [B] per-sequence loss sums (workspace)
  int32_t* arrivals;           // zero on entry (workspace)
  int32_t* status;
};
cudaError_t launch_distill(const DistillArgs& a, cudaStream_t stream);

// ---------------------------------------------------------------- same-state replay
struct ReplayArgs {
  int B, L, V, K, logits_dt;
  const void* logits_p;        // [B, L, V]
  const float* lse_p;          // [B, L]
  const int32_t* cand_ids;     // [B, L, K]
  const float* cand_logprob;   // [B, L, K]
  const int32_t* base_rank;    // [B, L]
  const int32_t* head_tokens;  // [B, L]
  const float* u_acc;          // [B, L]
  int32_t* flags;              // [B, L]
  int32_t* first_breaker;      // [B]
  int32_t* status;
};
cudaError_t launch_replay(const ReplayArgs& a, cudaStream_t stream);

size_t scan_smem_bytes(int L, int K, int S, int V);
cudaError_t launch_scan(const ScanArgs& a, cudaStream_t stream);

// ---------------------------------------------------------------- fused tail
// Serialises the use of the library's side streams: held while one call enqueues on them, and
// by graph creation from the start of its capture to the end.
std::mutex& side_stream_mutex();
// brisk_decode_tail with side_stream_mutex() already held by the caller.
brisk_status decode_tail_locked(const brisk_dims* d, const brisk_params* p, const void* tables,
                                const brisk_tail_io* io, int32_t select_mode, int32_t verify_mode,
                                void* ws, const brisk_events* ev, void* stream);

}  // namespace brisk
