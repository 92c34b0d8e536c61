// Tiled fp32 dense products, products of few rows, and the folds of the corrector's own weights. They
// serve the fp32 configurations (the hidden products of a call and the one-off folds of the frozen
// vocabulary rows, App. C.3) and the token folds' fallback; every product accumulates in fp32.
#include "brisk_internal.cuh"

namespace brisk {

namespace {

// One CTA computes a 128 x 64 tile of one product on 256 threads, 8 x 4 outputs a thread in
// packed fp32 pairs, over 16-wide K slices double-buffered in shared memory (the next two slices'
// global loads are in flight while the present one is multiplied). Large products are bound by
// the FMA pipes. A product with few tiles is bound by the K loop's latency instead (12 sequences
// x 24 positions x 1000 by 96: 10 tiles, 145 us on 64 x 64 tiles over the whole K), so there a
// cluster of up to 8 CTAs shares a tile: each takes a part of K, and each adds and stores its
// share of the tile's rows from all parts, in part order, through distributed shared memory.
constexpr int TM = 128, TN = 64, TK = 16;
constexpr int SIMT_THREADS = 256;
constexpr int SIMT_SPLIT_MAX = 8;
constexpr int SIMT_FILL = 152;        // CTAs a split aims for: one an SM
constexpr int SIMT_MIN_SLICES = 2;    // K slices a part has at least

struct SimtProblem {
  int M, N, K;
  const void* A;
  int lda;
  const void* B;
  int ldb;
  int transB;
  float* C;
  int ldc;
  int ntiles;        // tiles along N
  int split;         // CTAs (one cluster) that share a tile, each a part of K
  int vecA, vecB;    // rows may be read as 4-element vectors
  const float* bias; // optional [bias_period, N], row m % bias_period added to row m
  int bias_period;
};

// Elements k .. k + 3 of a row (zero past K).
template <typename T>
__device__ __forceinline__ float4 row4(const T* row, int k, int K, bool vec) {
  if (vec && k + 3 < K) {
    if constexpr (sizeof(T) == 4) {
      return __ldg(reinterpret_cast<const float4*>(row + k));
    } else {
      const uint2 w = __ldg(reinterpret_cast<const uint2*>(row + k));
      return make_float4(__uint_as_float(w.x << 16), __uint_as_float(w.x & 0xffff0000u),
                         __uint_as_float(w.y << 16), __uint_as_float(w.y & 0xffff0000u));
    }
  }
  float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
  if (k < K) v.x = to_f32(row[k]);
  if (k + 1 < K) v.y = to_f32(row[k + 1]);
  if (k + 2 < K) v.z = to_f32(row[k + 2]);
  if (k + 3 < K) v.w = to_f32(row[k + 3]);
  return v;
}

struct SimtSlices {
  float a[2][TK][TM + 4];
  float b[2][TK][TN + 4];
};
union SimtSmem {
  SimtSlices s;
  float part[TM][TN];   // this CTA's partial tile (split K)
};

template <typename TA, typename TB>
__global__ void __launch_bounds__(SIMT_THREADS)
gemm_simt_kernel(const __grid_constant__ SimtProblem P) {
  __shared__ __align__(16) SimtSmem sm;
  const int tid = threadIdx.x;
  const int split = P.split, tile = blockIdx.x / split, part = blockIdx.x - tile * split;
  const int M = P.M, N = P.N, K = P.K;
  const long long m0 = (long long)(tile / P.ntiles) * TM, n0 = (long long)(tile % P.ntiles) * TN;
  const TA* A = static_cast<const TA*>(P.A);
  const TB* B = static_cast<const TB*>(P.B);
  const int slices = (K + TK - 1) / TK, per = (slices + split - 1) / split;
  const int s0 = min(slices, part * per), s1 = min(slices, s0 + per);

  // a thread loads k 4q .. 4q + 3 of rows r and r + 64 of A and of row r of B, q = tid % 4;
  // with transB, columns 4c .. 4c + 3 of row kk of B
  const int q = tid & 3, r = tid >> 2;
  const int kk = tid >> 4, c = tid & 15;
  const bool ra = m0 + r < M, rb = m0 + r + 64 < M, rn = n0 + r < N;
  const TA* arow = A + (m0 + (ra ? r : 0)) * P.lda;
  const TA* brow_a = A + (m0 + (rb ? r + 64 : 0)) * P.lda;
  const TB* brow = B + (P.transB ? 0 : (n0 + (rn ? r : 0)) * P.ldb);
  const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
  struct Slice { float4 a, b, n; };
  auto load = [&](int s) {
    Slice v;
    const int k = s * TK + 4 * q;
    v.a = ra ? row4(arow, k, K, P.vecA) : zero;
    v.b = rb ? row4(brow_a, k, K, P.vecA) : zero;
    if (!P.transB) {
      v.n = rn ? row4(brow, k, K, P.vecB) : zero;
    } else {
      const int kt = s * TK + kk;
      v.n = kt < K ? row4(B + (long long)kt * P.ldb + n0, 4 * c, (int)min((long long)TN, N - n0), P.vecB)
                  : zero;
    }
    return v;
  };
  auto store = [&](int buf, const Slice& v) {
    SimtSlices& z = sm.s;
    z.a[buf][4 * q][r] = v.a.x; z.a[buf][4 * q + 1][r] = v.a.y;
    z.a[buf][4 * q + 2][r] = v.a.z; z.a[buf][4 * q + 3][r] = v.a.w;
    z.a[buf][4 * q][r + 64] = v.b.x; z.a[buf][4 * q + 1][r + 64] = v.b.y;
    z.a[buf][4 * q + 2][r + 64] = v.b.z; z.a[buf][4 * q + 3][r + 64] = v.b.w;
    if (!P.transB) {
      z.b[buf][4 * q][r] = v.n.x; z.b[buf][4 * q + 1][r] = v.n.y;
      z.b[buf][4 * q + 2][r] = v.n.z; z.b[buf][4 * q + 3][r] = v.n.w;
    } else {
      *reinterpret_cast<float4*>(&z.b[buf][kk][4 * c]) = v.n;
    }
  };
  // outputs: rows 8 ty .. 8 ty + 7 in pairs, columns 4 tx .. 4 tx + 3
  const int tx = tid & 15, ty = tid >> 4;
  float2 acc[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = make_float2(0.f, 0.f);
  // two slices on their way while one is multiplied
  Slice next{}, after{};
  if (s0 < s1) store(0, load(s0));
  if (s0 + 1 < s1) next = load(s0 + 1);
  __syncthreads();
  for (int s = s0; s < s1; ++s) {
    const int buf = (s - s0) & 1;
    if (s + 2 < s1) after = load(s + 2);
#pragma unroll
    for (int k = 0; k < TK; ++k) {
      const float4 x0 = *reinterpret_cast<const float4*>(&sm.s.a[buf][k][8 * ty]);
      const float4 x1 = *reinterpret_cast<const float4*>(&sm.s.a[buf][k][8 * ty + 4]);
      const float4 y = *reinterpret_cast<const float4*>(&sm.s.b[buf][k][4 * tx]);
      const float2 x[4] = {make_float2(x0.x, x0.y), make_float2(x0.z, x0.w),
                           make_float2(x1.x, x1.y), make_float2(x1.z, x1.w)};
      const float yv[4] = {y.x, y.y, y.z, y.w};
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j)
          acc[i][j] = __ffma2_rn(x[i], make_float2(yv[j], yv[j]), acc[i][j]);
    }
    if (s + 1 < s1) store(buf ^ 1, next);
    next = after;
    __syncthreads();
  }
  auto bias = [&](long long m, long long n) {
    return P.bias ? P.bias[(m % P.bias_period) * N + n] : 0.f;
  };
  if (split == 1) {
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const long long gm = m0 + 8 * ty + i;
      if (gm >= M) break;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const long long gn = n0 + 4 * tx + j;
        if (gn < N)
          P.C[gm * P.ldc + gn] = (i & 1 ? acc[i / 2][j].y : acc[i / 2][j].x) + bias(gm, gn);
      }
    }
    return;
  }
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const float2* v = acc[i / 2];
    *reinterpret_cast<float4*>(&sm.part[8 * ty + i][4 * tx]) =
        i & 1 ? make_float4(v[0].y, v[1].y, v[2].y, v[3].y)
              : make_float4(v[0].x, v[1].x, v[2].x, v[3].x);
  }
  cluster_sync();
  // this CTA's share of the tile's valid rows: the parts added in part order
  const int rows = (int)min((long long)TM, M - m0);
  const int share = (rows + split - 1) / split;
  const int r0 = part * share, r1 = min(rows, r0 + share);
  for (int e = r0 * 16 + tid; e < r1 * 16; e += SIMT_THREADS) {
    const int row = e >> 4, col = 4 * (e & 15);
    const float4 v = sum_cluster(&sm.part[row][col], split);
    const float x[4] = {v.x, v.y, v.z, v.w};
    float* dst = P.C + (m0 + row) * P.ldc + n0 + col;
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (n0 + col + j < N) dst[j] = x[j] + bias(m0 + row, n0 + col + j);
  }
  cluster_sync();   // the other CTAs have read this one's part
}

// Products of few rows: a warp an output column, whose lanes take four k each of every 128 for every
// row, then a warp sum a row. A tile has nothing to share among so few rows, and its barriers and the
// cluster's cost more than they are worth: a lone corrector of eight positions (d = 96, r = 112) 47 us
// with its products on tiles, 34 so. Up to a k of 128; a longer one only where every product of the
// call has few rows (one sequence of two positions, d = 512, r = 112: 43 us, 26; d = 4096, r = 256: 89,
// 35): with longer products of other rows beside it, a tail's is no faster for it (8 rows, d = 512: 30.9
// us with the context's product of k = 512 on tiles, 34.8 without).
constexpr int FEW_WARPS = 8;
constexpr int FEW_ROWS = 4;             // rows of a call up to which every k is taken so
constexpr int FEW_ROWS_SHORT = 8;       // rows of a product up to which a k of FEW_SHORT_K is (16 in a
constexpr int FEW_SHORT_K = 128;        // tail, k = 128: 38 us, 40)

// UNROLL: four k a lane of the column and of every row that are on their way at once.
template <typename TA, typename TB, int ROWS, int UNROLL>
__global__ void __launch_bounds__(FEW_WARPS * 32)
gemm_few_kernel(const __grid_constant__ SimtProblem P) {
  const int lane = threadIdx.x & 31;
  const long long n = (long long)blockIdx.x * FEW_WARPS + (threadIdx.x >> 5);
  if (n >= P.N) return;
  const TA* A = static_cast<const TA*>(P.A);
  const TB* b = static_cast<const TB*>(P.B) + n * P.ldb;
  float2 acc[ROWS];
#pragma unroll
  for (int m = 0; m < ROWS; ++m) acc[m] = make_float2(0.f, 0.f);
  for (int k0 = 4 * lane; k0 < P.K; k0 += 128 * UNROLL) {
    float4 y[UNROLL], x[UNROLL][ROWS];
#pragma unroll
    for (int u = 0; u < UNROLL; ++u) {
      y[u] = row4(b, k0 + 128 * u, P.K, P.vecB);
#pragma unroll
      for (int m = 0; m < ROWS; ++m)
        if (m < P.M) x[u][m] = row4(A + (long long)m * P.lda, k0 + 128 * u, P.K, P.vecA);
    }
#pragma unroll
    for (int u = 0; u < UNROLL; ++u)
#pragma unroll
      for (int m = 0; m < ROWS; ++m)
        if (m < P.M) {
          acc[m] = __ffma2_rn(make_float2(x[u][m].x, x[u][m].y), make_float2(y[u].x, y[u].y), acc[m]);
          acc[m] = __ffma2_rn(make_float2(x[u][m].z, x[u][m].w), make_float2(y[u].z, y[u].w), acc[m]);
        }
  }
#pragma unroll
  for (int m = 0; m < ROWS; ++m) {
    if (m >= P.M) break;
    const float v = warp_sum(acc[m].x + acc[m].y);
    if (lane == 0)
      P.C[(long long)m * P.ldc + n] = v + (P.bias ? P.bias[(long long)(m % P.bias_period) * P.N + n] : 0.f);
  }
}

// One thread an item: the weight blocks' element (j, t) in every form the products read, then the
// position shares, the feature shares and the gate weights (each a sum of 16 products in order).
// Bound by launches when done block by block: 29 launches took about 100 us.
template <typename T>
__global__ void __launch_bounds__(256) pack_kernel(const __grid_constant__ PackArgs a) {
  const int r = a.r, S = 2 * r, ldw = 2 * r + 32;
  const T *Wz = static_cast<const T*>(a.Wz), *Wh = static_cast<const T*>(a.Wh),
          *W0 = static_cast<const T*>(a.W0), *Ws = static_cast<const T*>(a.W_s),
          *pos = static_cast<const T*>(a.pos), *Pp = static_cast<const T*>(a.P_phi);
  long long e = blockIdx.x * 256ll + threadIdx.x;
  if (e < (long long)S * r) {
    const int j = (int)(e / r), t = (int)(e % r);
    const T z = Wz[(size_t)j * ldw + t], h = Wh[(size_t)j * ldw + t], i = W0[(size_t)j * S + t];
    const size_t at = (size_t)j * r + t, lower = (size_t)S * r + at;
    a.W2[at] = to_f32(z);
    a.W2[lower] = to_f32(h);
    a.W0h[at] = to_f32(i);
    if constexpr (sizeof(T) == 2) {
      const T tz = Wz[(size_t)j * ldw + r + t], th = Wh[(size_t)j * ldw + r + t],
              ti = W0[(size_t)j * S + r + t], ws = Ws[(size_t)t * S + j];
#pragma unroll
      for (int part = 0; part < 3; ++part) {
        const size_t up = (size_t)j * 3 * r + part * r + t, lo = (size_t)S * 3 * r + up;
        a.W2s[up] = z;
        a.W2s[lo] = h;
        a.W0s[up] = i;
        a.Wt2s[up] = tz;
        a.Wt2s[lo] = th;
        a.W0ts[up] = ti;
        a.Ws3[up] = ws;
      }
    }
    return;
  }
  e -= (long long)S * r;
  auto dot16 = [](auto x, auto y) {
    float acc = 0.f;
    for (int t = 0; t < 16; ++t) acc = fmaf(x(t), y(t), acc);
    return acc;
  };
  if (e < (long long)a.L * 2 * S) {        // posG(i, j) = W_{z,h}[j, 2r : 2r + 16] . pos_i
    const int i = (int)(e / (2 * S)), j = (int)(e % (2 * S));
    const T* w = (j < S ? Wz + (size_t)j * ldw : Wh + (size_t)(j - S) * ldw) + 2 * r;
    a.posG[e] = dot16([&](int t) { return to_f32(pos[i * 16 + t]); },
                      [&](int t) { return to_f32(w[t]); });
    return;
  }
  e -= (long long)a.L * 2 * S;
  if (e < 10ll * S) {                       // F(j, f) = sum_t W[j, 2r + 16 + t] P_phi[t, f]
    const int half = (int)(e / (5 * S)), q = (int)(e % (5 * S)), j = q / 5, f = q % 5;
    const T* w = (half ? Wh : Wz) + (size_t)j * ldw + 2 * r + 16;
    (half ? a.Fh : a.Fz)[q] = dot16([&](int t) { return to_f32(w[t]); },
                                    [&](int t) { return to_f32(Pp[t * 5 + f]); });
    return;
  }
  e -= 10ll * S;
  if (e < S + 5) a.wg[e] = to_f32(static_cast<const T*>(a.w_g)[e]);
}

template <typename TA, typename TB>
cudaError_t gemm_t(int M, int N, int K, const void* A, int lda, const void* B, int ldb,
                   bool transB, float* C, int ldc, cudaStream_t stream, const float* bias,
                   int bias_period, bool few) {
  const int ntiles = (N + TN - 1) / TN, slices = (K + TK - 1) / TK;
  const long long tiles = (long long)((M + TM - 1) / TM) * ntiles;
  int split = 1;
  while (split < SIMT_SPLIT_MAX && 2 * split * tiles <= SIMT_FILL &&
         slices >= 2 * split * SIMT_MIN_SLICES)
    split *= 2;
  auto vec = [](const void* p, size_t size, int ld) {
    return reinterpret_cast<uintptr_t>(p) % (4 * size) == 0 && ld % 4 == 0;
  };
  const SimtProblem P{M, N, K, A, lda, B, ldb, transB ? 1 : 0, C, ldc, ntiles, split,
                      vec(A, sizeof(TA), lda), vec(B, sizeof(TB), ldb), bias, bias_period};
  if (!transB && M <= FEW_ROWS_SHORT && (few || K <= FEW_SHORT_K)) {
    auto kernel = M <= FEW_ROWS ? gemm_few_kernel<TA, TB, FEW_ROWS, 4>
                                : gemm_few_kernel<TA, TB, FEW_ROWS_SHORT, 1>;
    const cudaError_t e = launch_prio(kernel, dim3((unsigned)((N + FEW_WARPS - 1) / FEW_WARPS)),
                                      dim3(FEW_WARPS * 32), 0, stream, P);
    return e != cudaSuccess ? e : cudaGetLastError();
  }
  const cudaError_t e = launch_cluster(gemm_simt_kernel<TA, TB>, dim3((unsigned)(tiles * split)),
                                       dim3(SIMT_THREADS), 0, stream, split, P);
  return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace

cudaError_t gemm_simt(int M, int N, int K, const void* A, int a_dt, int lda, const void* B,
                      int b_dt, int ldb, bool transB, float* C, int ldc, cudaStream_t stream,
                      const float* bias, int bias_period, int call_rows) {
  if (M <= 0 || N <= 0) return cudaSuccess;
  const bool few = call_rows <= FEW_ROWS;
  if (a_dt == BRISK_DT_BF16 && b_dt == BRISK_DT_BF16)
    return gemm_t<__nv_bfloat16, __nv_bfloat16>(M, N, K, A, lda, B, ldb, transB, C, ldc, stream,
                                                bias, bias_period, few);
  if (a_dt == BRISK_DT_F32 && b_dt == BRISK_DT_BF16)
    return gemm_t<float, __nv_bfloat16>(M, N, K, A, lda, B, ldb, transB, C, ldc, stream, bias,
                                        bias_period, few);
  if (a_dt == BRISK_DT_BF16 && b_dt == BRISK_DT_F32)
    return gemm_t<__nv_bfloat16, float>(M, N, K, A, lda, B, ldb, transB, C, ldc, stream, bias,
                                        bias_period, few);
  return gemm_t<float, float>(M, N, K, A, lda, B, ldb, transB, C, ldc, stream, bias, bias_period, few);
}

cudaError_t pack_weights(const PackArgs& a, cudaStream_t stream) {
  const long long S = 2ll * a.r, items = S * a.r + a.L * 2 * S + 10 * S + S + 5;
  const unsigned grid = (unsigned)((items + 255) / 256);
  if (a.dt == BRISK_DT_BF16) pack_kernel<__nv_bfloat16><<<grid, 256, 0, stream>>>(a);
  else pack_kernel<float><<<grid, 256, 0, stream>>>(a);
  return cudaGetLastError();
}

}  // namespace brisk
