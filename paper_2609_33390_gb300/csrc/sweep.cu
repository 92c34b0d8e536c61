// Vocabulary sweep: per logit row, the log-partition and the ordered top-K
// (Sec. 3.3 "C_i = TopK(q_i, K)"; App. C.3 ordered candidate set), and for
// verifier rows the argmax (lowest id on ties) and the log-partition.
//
// Two layouts, by the rows and their length (by_warp). Many rows, or short ones: a warp sweeps a row
// alone (sweep_rows_kernel). Else one CTA of SWEEP_WARPS warps sweeps one row, or one of nsplit
// equal segments of a row when there are too few rows to fill the chip:
//
// Its warps take the segment's batches in turn (32 lanes x SWEEP_UNROLL 16-byte streaming loads, all
// in flight at once). Each lane keeps a running (max, sum of exp) pair. The lanes' maxima also give
// the top-K's threshold: every warp publishes its few largest, each of them a logit of the segment,
// and the K-th largest of all published ones is a lower bound on the segment's K-th best. A batch
// whose largest logit is below the threshold costs one comparison; a logit that reaches it (about
// K (1 + ln(batches)) of them a row) is appended to the warp's buffer. At the end every buffered
// entry that reaches the final threshold counts the entries that precede it, which is its place. The
// segments of a row are merged the same way by the last of them to finish (arrival counter, no
// waiting). Which logits are buffered depends on timing; the outputs do not.
//
// Large tensors are bound by memory (see by_warp), small ones by the threshold's and the merge's
// latency. A threshold shared by the CTA's warps is why a row is one CTA's where there are few rows:
// with a list of its own in every warp, each warp paid for its own insertions (16 x 32 rows of 126464
// bf16, K = 8: 50 us, now 28; 32 rows 29, now 10).
#include "brisk_internal.cuh"

namespace brisk {

namespace {

constexpr int SWEEP_WARPS = 8;
constexpr int SWEEP_UNROLL = 8;                         // 16-byte loads in flight per lane
constexpr int SWEEP_BATCH = 32 * SWEEP_UNROLL;          // 16-byte vectors a warp loads at once
constexpr int SWEEP_RESIDENT = 4;                       // CTAs an SM holds at once
constexpr int SWEEP_CTAS = 152 * SWEEP_RESIDENT;
constexpr int SWEEP_BUF = 64;                           // entries a warp buffers
constexpr int SWEEP_MERGE = SWEEP_WARPS * SWEEP_BUF;    // entries merged at most
constexpr int SWEEP_TOPS = 32 / SWEEP_WARPS;            // maxima a warp publishes
constexpr int SWEEP_RAISE = 3;                          // entries between raises of the threshold

// The warp-a-row layout.
constexpr int ROW_WARPS = 2;                            // rows a CTA sweeps
constexpr int ROW_CARVEOUT_KB = 64;
constexpr int ROW_SHORT = 3 * SWEEP_BATCH + 33;         // vectors below which every row takes it
constexpr int ROW_MID = 152 * 12;                       // rows from which three times as many vectors do
constexpr int ROW_MANY = 152 * 16;                      // rows from which every length does for K > 16

// Online log-sum-exp of one logit.
__device__ __forceinline__ void lse_update(float f, float& m, float& s) {
  if (f > m) {
    s *= ex2((m - f) * LOG2E);
    m = f;
  }
  if (m != -INFINITY) s += ex2((f - m) * LOG2E);
}

// The warp's values in ascending lane order (bitonic sort).
__device__ __forceinline__ unsigned warp_sort(unsigned x) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int size = 2; size <= 32; size <<= 1) {
#pragma unroll
    for (int j = size >> 1; j > 0; j >>= 1) {
      const unsigned y = __shfl_xor_sync(FULL_MASK, x, j);
      const bool ascending = (lane & size) == 0;
      const bool lower = (lane & j) == 0;
      x = (lower == ascending) ? min(x, y) : max(x, y);
    }
  }
  return x;
}

// Max of the four logits of a vector.
__device__ __forceinline__ float vec_max(const uint4& w, float) {
  return fmaxf(fmaxf(__uint_as_float(w.x), __uint_as_float(w.y)),
               fmaxf(__uint_as_float(w.z), __uint_as_float(w.w)));
}

__device__ __forceinline__ float vec_max(const uint4& w, __nv_bfloat16) {
  const __nv_bfloat162* v = reinterpret_cast<const __nv_bfloat162*>(&w);
  const __nv_bfloat162 c = __hmax2(__hmax2(v[0], v[1]), __hmax2(v[2], v[3]));
  return fmaxf(__low2float(c), __high2float(c));
}

// Max of a lane's whole batch (bf16: packed maxima, 4 instructions a vector).
__device__ __forceinline__ float batch_max(const uint4 (&w)[SWEEP_UNROLL], __nv_bfloat16) {
  __nv_bfloat162 m[4];
#pragma unroll
  for (int u = 0; u < SWEEP_UNROLL; ++u) {
    const __nv_bfloat162* v = reinterpret_cast<const __nv_bfloat162*>(&w[u]);
#pragma unroll
    for (int j = 0; j < 4; ++j) m[j] = u ? __hmax2(m[j], v[j]) : v[j];
  }
  const __nv_bfloat162 c = __hmax2(__hmax2(m[0], m[1]), __hmax2(m[2], m[3]));
  return fmaxf(__low2float(c), __high2float(c));
}
__device__ __forceinline__ float batch_max(const uint4 (&w)[SWEEP_UNROLL], float) {
  float m = vec_max(w[0], 0.f);
#pragma unroll
  for (int u = 1; u < SWEEP_UNROLL; ++u) m = fmaxf(m, vec_max(w[u], 0.f));
  return m;
}

// Sum of exp(x - m) of a lane's batch for m past FAR_LOGIT in size. The main path multiplies first,
// fma(x, log2 e, -(m log2 e)), and so returns the rounding of m log2 e where x equals m: up to half
// an ulp of m, as the log-partition's own rounding, but 2^-25 of m as an exponent, which overflows
// on a lane whose logits are all a mask of -1e10 (and spoils the row: inf times zero, later). Here
// the difference comes first, which is exact for logits close enough to count.
constexpr float FAR_LOGIT = 1e6f;
template <typename T>
__device__ __forceinline__ float sum_far(const uint4 (&w)[SWEEP_UNROLL], float m, T) {
  const float2 off = make_float2(-m, -m), l2e = make_float2(LOG2E, LOG2E);
  float2 s = make_float2(0.f, 0.f);
#pragma unroll
  for (int u = 0; u < SWEEP_UNROLL; ++u) {
    float f[Vec<T>::N];
    unpack(w[u], f, T());
#pragma unroll
    for (int j = 0; j < Vec<T>::N; j += 2) {
      const float2 arg = __fmul2_rn(__fadd2_rn(make_float2(f[j], f[j + 1]), off), l2e);
      s = __fadd2_rn(s, make_float2(ex2(arg.x), ex2(arg.y)));
    }
  }
  return s.x + s.y;
}

// A batch in a lane's running (max, sum of exp): the max first (returns the batch's own), which moves
// once per batch, so that all of its exponentials share one offset; then the sum, arguments and
// parts in packed fp32 pairs.
template <typename T>
__device__ __forceinline__ float raise_max(const uint4 (&w)[SWEEP_UNROLL], float& m, float& s) {
  const float mx = batch_max(w, T());
  if (mx > m) {
    s *= ex2((m - mx) * LOG2E);
    m = mx;
  }
  return mx;
}
template <typename T>
__device__ __forceinline__ void add_batch(const uint4 (&w)[SWEEP_UNROLL], float m, float& s) {
  constexpr int VN = Vec<T>::N;
  if (fabsf(m) > FAR_LOGIT) {
    if (m != -INFINITY) s += sum_far(w, m, T());
  } else {
    const float nmb = -m * LOG2E;
    const float2 l2e = make_float2(LOG2E, LOG2E), off = make_float2(nmb, nmb);
    float2 acc0 = make_float2(0.f, 0.f), acc1 = make_float2(0.f, 0.f);
#pragma unroll
    for (int u = 0; u < SWEEP_UNROLL; ++u) {
      float f[VN];
      unpack(w[u], f, T());
#pragma unroll
      for (int j = 0; j < VN; j += 2) {
        const float2 arg = __ffma2_rn(make_float2(f[j], f[j + 1]), l2e, off);
        const float2 e = make_float2(ex2(arg.x), ex2(arg.y));
        if ((j / 2 + u) & 1) acc1 = __fadd2_rn(acc1, e);
        else acc0 = __fadd2_rn(acc0, e);
      }
    }
    const float2 acc = __fadd2_rn(acc0, acc1);
    s += acc.x + acc.y;
  }
}

// Order-preserving map of a float (not NaN) to an unsigned key; -0 and +0 map alike.
__device__ __forceinline__ unsigned order_key(float f) {
  const unsigned u = __float_as_uint(f + 0.f);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float key_to_float(unsigned k) {
  return __uint_as_float((k & 0x80000000u) ? (k & 0x7fffffffu) : ~k);
}

struct SweepSmem {
  uint4 stash[SWEEP_WARPS][SWEEP_UNROLL];        // one lane's batch
  float val[SWEEP_WARPS][SWEEP_BUF];             // the warps' buffers, then the entries to merge
  int id[SWEEP_WARPS][SWEEP_BUF];
  unsigned long long top[2][SWEEP_WARPS];        // the warps' largest lane maxima so far (packed)
  int listed;
  float thr;                                     // the final threshold
  float m[SWEEP_WARPS], s[SWEEP_WARPS];
  float best_v[32];                              // the merged list
  int best_i[32];
  int last;
};

// Per-lane state of a warp's sweep; everything but (m, s) is the same in all lanes.
struct WarpState {
  float m, s;      // running max and sum of exp(x - max)
  float thr;       // lower bound on the segment's K-th best
  float kv;        // K-th best of the buffer when it last overflowed: only better ones matter
  int ki;
  int count;       // entries in the warp's buffer
  int fresh;       // of these, appended since the threshold was last raised
};

// Publishes this warp's four largest lane maxima (the largest alone for kout == 1; the four
// largest of either half of the warp for kout > 16), each set as one word that other warps read
// whole, so that no maximum is ever seen twice: 16-bit keys, cut towards smaller values, so still
// lower bounds. With fewer than kout sets the threshold would hang on the warp whose logits are
// smallest (32 of 100003 fp32: 224 us with four maxima a warp, 175 with eight).
__device__ __forceinline__ void publish(SweepSmem& sm, int warp, int kout, float m) {
  const int lane = threadIdx.x & 31;
  const bool halves = kout > 16;
  const unsigned mask = !halves ? FULL_MASK : (lane < 16 ? 0x0000ffffu : 0xffff0000u);
  unsigned key = order_key(m);
  unsigned long long word = __reduce_max_sync(mask, key);
  if (kout > 1) {
    unsigned top = (unsigned)word;
    word >>= 16;
#pragma unroll
    for (int j = 1; j < SWEEP_TOPS; ++j) {
      const unsigned at = __ballot_sync(mask, key == top) & mask;
      if (lane == __ffs(at) - 1) key = 0;
      top = __reduce_max_sync(mask, key);
      word = word << 16 | top >> 16;
    }
  }
  if (lane == 0 || (halves && lane == 16))
    *const_cast<volatile unsigned long long*>(&sm.top[lane >> 4][warp]) = word;
  __syncwarp();
}

// K-th largest of the published maxima: a lower bound on the segment's K-th best.
__device__ __forceinline__ float segment_threshold(const SweepSmem& sm, int kout) {
  const int lane = threadIdx.x & 31, w = lane / SWEEP_TOPS, shift = 16 * (lane % SWEEP_TOPS);
  const volatile unsigned long long* top = &sm.top[0][0];
  if (kout == 1)
    return key_to_float(__reduce_max_sync(FULL_MASK, lane < SWEEP_WARPS ? (unsigned)top[lane] : 0u));
  unsigned key = warp_sort((unsigned)(top[w] >> shift) & 0xffffu);
  if (kout > 16) {
    // the larger 32 of 64: two sorted halves compared end to end
    const unsigned other = warp_sort((unsigned)(top[SWEEP_WARPS + w] >> shift) & 0xffffu);
    key = warp_sort(max(key, __shfl_xor_sync(FULL_MASK, other, 31)));
  }
  const unsigned kth = __shfl_sync(FULL_MASK, key, 32 - kout);
  return kth <= 0x7fu ? -INFINITY : key_to_float(kth << 16);   // (0x7f: the key of -inf)
}

// Cuts a full buffer down to its best kout entries, best first; rare.
__device__ __noinline__ void trim_buffer(SweepSmem& sm, int warp, int kout, WarpState& st) {
  const int lane = threadIdx.x & 31;
  __syncwarp();
  float v[SWEEP_BUF / 32];
  int id[SWEEP_BUF / 32], rank[SWEEP_BUF / 32];
#pragma unroll
  for (int j = 0; j < SWEEP_BUF / 32; ++j) {
    const int e = lane + 32 * j;
    v[j] = e < st.count ? sm.val[warp][e] : -INFINITY;
    id[j] = e < st.count ? sm.id[warp][e] : INVALID_ID;
    rank[j] = 0;
  }
  for (int o = 0; o < st.count; ++o) {
    const float ov = sm.val[warp][o];
    const int oi = sm.id[warp][o];
#pragma unroll
    for (int j = 0; j < SWEEP_BUF / 32; ++j) rank[j] += better(ov, oi, v[j], id[j]) ? 1 : 0;
  }
  __syncwarp();
#pragma unroll
  for (int j = 0; j < SWEEP_BUF / 32; ++j)
    if (id[j] != INVALID_ID && rank[j] < kout) {
      sm.val[warp][rank[j]] = v[j];
      sm.id[warp][rank[j]] = id[j];
    }
  __syncwarp();
  st.count = min(st.count, kout);
  st.kv = sm.val[warp][kout - 1];   // (a trimmed buffer held at least kout entries)
  st.ki = sm.id[warp][kout - 1];
  __syncwarp();
}

// Appends the lanes' elements f (ids id) that reach the threshold.
__device__ __forceinline__ void append(SweepSmem& sm, int warp, int kout, bool in, float f, int id,
                                       WarpState& st) {
  const bool want = in && f >= st.thr && better(f, id, st.kv, st.ki);
  unsigned hit = __ballot_sync(FULL_MASK, want);
  if (!hit) return;
  if (st.count + __popc(hit) > SWEEP_BUF) {
    trim_buffer(sm, warp, kout, st);
    hit = __ballot_sync(FULL_MASK, want && better(f, id, st.kv, st.ki));
  }
  const int lane = threadIdx.x & 31;
  if (hit >> lane & 1) {
    const int at = st.count + __popc(hit & ((1u << lane) - 1));
    sm.val[warp][at] = f;
    sm.id[warp][at] = id;
  }
  st.count += __popc(hit);
  st.fresh += __popc(hit);
}

// The rare path of a batch: the vectors of each lane that holds a logit of at least the threshold
// (mx: the lane's largest) are shared with the warp, which appends the logits that count.
template <typename T>
__device__ __forceinline__ void offer_batch(const uint4 (&w)[SWEEP_UNROLL], float mx, int id0_lane,
                                            int valid, int kout, SweepSmem& sm, WarpState& st) {
  constexpr int VN = Vec<T>::N;
  constexpr int PER_WORD = VN / 4;   // logits in four bytes
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  unsigned lanes = __ballot_sync(FULL_MASK, valid > 0 && mx >= st.thr);
  while (lanes) {
    const int src = __ffs(lanes) - 1;
    lanes &= lanes - 1;
    if (lane == src) {
#pragma unroll
      for (int u = 0; u < SWEEP_UNROLL; ++u) sm.stash[warp][u] = w[u];
    }
    const int id0 = __shfl_sync(FULL_MASK, id0_lane, src);
    const int vecs = __shfl_sync(FULL_MASK, valid, src);
    __syncwarp();
    // lane t reads the four bytes t of every 32 words
#pragma unroll
    for (int q = 0; q < SWEEP_UNROLL / 8; ++q) {
      const int word = 32 * q + lane, u = word / 4;
      const uint32_t bits = reinterpret_cast<const uint32_t*>(sm.stash[warp])[word];
      const int id = id0 + u * 32 * VN + (word % 4) * PER_WORD;
      if constexpr (PER_WORD == 2) {
        append(sm, warp, kout, u < vecs, __uint_as_float(bits << 16), id, st);
        append(sm, warp, kout, u < vecs, __uint_as_float(bits & 0xffff0000u), id + 1, st);
      } else {
        append(sm, warp, kout, u < vecs, __uint_as_float(bits), id, st);
      }
    }
    __syncwarp();
  }
  // ids only grow from one batch to the next: a later logit has to exceed the trimmed buffer's
  // K-th best
  if (st.ki != INVALID_ID) st.thr = fmaxf(st.thr, nextafterf(st.kv, INFINITY));
}

// One batch: SWEEP_UNROLL vectors per lane, lane's vector u holding ids id0_lane + 32 u VN + j;
// vectors u >= valid are padding (-inf) and are never appended.
template <typename T, bool FIRST>
__device__ __forceinline__ void sweep_batch(const uint4 (&w)[SWEEP_UNROLL], int id0_lane, int valid,
                                            int kout, SweepSmem& sm, WarpState& st) {
  const int warp = threadIdx.x >> 5;
  const float mx = raise_max<T>(w, st.m, st.s);
  if constexpr (FIRST) publish(sm, warp, kout, st.m);
  add_batch<T>(w, st.m, st.s);
  if constexpr (FIRST) {   // every warp has published its maxima before anyone needs them
    __syncthreads();
    st.thr = segment_threshold(sm, kout);
  }
  if (!__any_sync(FULL_MASK, mx >= st.thr)) return;
  offer_batch<T>(w, mx, id0_lane, valid, kout, sm, st);
  if (!FIRST && st.fresh >= SWEEP_RAISE) {
    publish(sm, warp, kout, st.m);
    st.thr = fmaxf(st.thr, segment_threshold(sm, kout));
    st.fresh = 0;
  }
}

// This warp's share of the vectors [v0, v1) of the row (its batches interleaved with the other
// warps'), and for warp 0 the row's unaligned head (first segment) and ragged tail (last one);
// then the entries that can be among the segment's best, listed for the merge.
template <typename T>
__device__ __forceinline__ void sweep_segment(const T* rowp, int V, int split, int nsplit, int kout,
                                              SweepSmem& sm, WarpState& st) {
  constexpr int VN = Vec<T>::N;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uintptr_t addr = reinterpret_cast<uintptr_t>(rowp);
  int head = (int)(((16u - (unsigned)(addr & 15u)) & 15u) / sizeof(T));
  if (head > V) head = V;
  const int nvec = (V - head) / VN;
  const int per = (nvec + nsplit - 1) / nsplit;
  const int v0 = min(nvec, split * per), v1 = min(nvec, v0 + per);
  st = WarpState{-INFINITY, 0.f, -INFINITY, -INFINITY, INVALID_ID, 0, 0};
  // the unaligned head (fewer than VN logits, the row's lowest ids)
  if (warp == 0 && split == 0) {
    const bool in = lane < head;
    float f = -INFINITY;
    if (in) {
      f = to_f32(rowp[lane]);
      lse_update(f, st.m, st.s);
    }
    append(sm, warp, kout, in, f, lane, st);
  }
  const uint4* vp = reinterpret_cast<const uint4*>(rowp + head) + lane;
  const uint32_t ninf = VN == 8 ? 0xff80ff80u : 0xff800000u;
  int base = v0 + warp * SWEEP_BATCH;
  uint4 w[SWEEP_UNROLL];
  auto load = [&]() -> int {   // padded with -inf past the segment
    const int left = v1 - base - lane;
    const int valid = left <= 0 ? 0 : min(SWEEP_UNROLL, (left + 31) / 32);
#pragma unroll
    for (int u = 0; u < SWEEP_UNROLL; ++u)
      w[u] = u < valid ? ld_stream_v4(vp + base + 32 * u) : make_uint4(ninf, ninf, ninf, ninf);
    return valid;
  };
  int valid = load();
  sweep_batch<T, true>(w, head + (base + lane) * VN, valid, kout, sm, st);
  base += SWEEP_WARPS * SWEEP_BATCH;
  // full batches: no bounds checks
  for (; base + SWEEP_BATCH <= v1; base += SWEEP_WARPS * SWEEP_BATCH) {
#pragma unroll
    for (int u = 0; u < SWEEP_UNROLL; ++u) w[u] = ld_stream_v4(vp + base + 32 * u);
    sweep_batch<T, false>(w, head + (base + lane) * VN, SWEEP_UNROLL, kout, sm, st);
  }
  if (base < v1) {
    valid = load();
    sweep_batch<T, false>(w, head + (base + lane) * VN, valid, kout, sm, st);
  }
  // the ragged tail (fewer than VN logits, the row's highest ids)
  if (warp == 0 && split == nsplit - 1) {
    const int e = head + nvec * VN + lane;
    float f = -INFINITY;
    if (e < V) {
      f = to_f32(rowp[e]);
      lse_update(f, st.m, st.s);
    }
    append(sm, warp, kout, e < V, f, e, st);
  }
  publish(sm, warp, kout, st.m);
  warp_lse_combine(st.m, st.s);
  __syncthreads();
  if (warp == 0) {   // (one warp's work: the others leave their issue slots to other CTAs)
    const float t = segment_threshold(sm, kout);
    if (lane == 0) sm.thr = t;
  }
  __syncthreads();
  // the entries that reach it, through registers: the list takes the buffers' place
  const float thr = sm.thr;
  float v[SWEEP_BUF / 32];
  int id[SWEEP_BUF / 32], at[SWEEP_BUF / 32];
#pragma unroll
  for (int j = 0; j < SWEEP_BUF / 32; ++j) {
    const int e = lane + 32 * j;
    v[j] = sm.val[warp][e];
    id[j] = sm.id[warp][e];
    const unsigned hit = __ballot_sync(FULL_MASK, e < st.count && v[j] >= thr);
    int first = 0;
    if (lane == 0 && hit) first = atomicAdd(&sm.listed, __popc(hit));
    first = __shfl_sync(FULL_MASK, first, 0);
    at[j] = hit >> lane & 1 ? first + __popc(hit & ((1u << lane) - 1)) : -1;
  }
  __syncthreads();
#pragma unroll
  for (int j = 0; j < SWEEP_BUF / 32; ++j)
    if (at[j] >= 0) {
      (&sm.val[0][0])[at[j]] = v[j];
      (&sm.id[0][0])[at[j]] = id[j];
    }
}

// The best kout of the n listed entries, best first, into best_v / best_i (-inf, INVALID_ID past
// the real ones): an entry's place is the number of entries that precede it. CTA-wide.
__device__ __forceinline__ void merge_by_rank(SweepSmem& sm, int n, int kout) {
  const int tid = threadIdx.x;
  if (tid < 32) {
    sm.best_v[tid] = -INFINITY;
    sm.best_i[tid] = INVALID_ID;
  }
  __syncthreads();
  const float* list_v = &sm.val[0][0];
  const int* list_i = &sm.id[0][0];
  for (int e = tid; e < n; e += SWEEP_WARPS * 32) {
    const float v = list_v[e];
    const int i = list_i[e];
    int rank = 0;
#pragma unroll 4
    for (int o = 0; o < n; ++o) rank += better(list_v[o], list_i[o], v, i) ? 1 : 0;
    if (i != INVALID_ID && rank < kout) {
      sm.best_v[rank] = v;
      sm.best_i[rank] = i;
    }
  }
  __syncthreads();
}

// A row's outputs, by one warp: its (max, sum of exp) and, in lane k < kout, the k-th best.
__device__ __forceinline__ void write_row(const SweepSeg& sg, size_t row, int kout, float m, float s,
                                          float v, int id, int32_t* status) {
  const int lane = threadIdx.x & 31;
  const float lse = m + logf(s);
  if (!isfinite(lse) && lane == 0) set_status(status, BRISK_ERR_NUMERIC);
  if (lane < kout) {
    sg.out_ids[row * kout + lane] = id;
    if (sg.out_logprob) sg.out_logprob[row * kout + lane] = v - lse;
  }
  if (lane == 0) sg.out_lse[row] = lse;
}

// At most 64 registers a thread: four CTAs of eight warps an SM.
template <typename T>
__global__ void __launch_bounds__(SWEEP_WARPS * 32, SWEEP_RESIDENT)
sweep_kernel(const __grid_constant__ SweepLaunch a) {
  __shared__ SweepSmem sm;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int nsplit = a.nsplit;
  const long long ctas0 = (long long)a.seg[0].rows * nsplit;
  const int si = (long long)blockIdx.x < ctas0 ? 0 : 1;
  const SweepSeg& sg = a.seg[si];
  const unsigned t = si ? (unsigned)(blockIdx.x - ctas0) : blockIdx.x;
  const int row = (int)(t / nsplit), split = (int)(t % nsplit);
  const int kout = sg.kout;
  const T* rowp = reinterpret_cast<const T*>(sg.logits) + (size_t)row * a.V;
  if (tid == 0) sm.listed = 0;   // (ordered before its use by the segment's barriers)
  WarpState st;
  sweep_segment<T>(rowp, a.V, split, nsplit, kout, sm, st);
  if (lane == 0) {
    sm.m[warp] = st.m;
    sm.s[warp] = st.s;
  }
  __syncthreads();
  merge_by_rank(sm, sm.listed, kout);
  float m = -INFINITY, s = 0.f;
  if (warp == 0) {
    if (lane < SWEEP_WARPS) {
      m = sm.m[lane];
      s = sm.s[lane];
    }
    warp_lse_combine(m, s);
  }
  if (nsplit > 1) {
    // publish this segment; the last of the row's segments to arrive merges all of them
    const size_t p0 = (size_t)row * nsplit;
    if (warp == 0) {
      if (lane < kout) {
        sg.part_val[(p0 + split) * a.KP + lane] = sm.best_v[lane];
        sg.part_id[(p0 + split) * a.KP + lane] = sm.best_i[lane];
      }
      if (lane == 0) {
        sg.part_m[p0 + split] = m;
        sg.part_s[p0 + split] = s;
      }
      __threadfence();
      __syncwarp();
      if (lane == 0) sm.last = atomicAdd(&sg.counters[row], 1) == nsplit - 1;
    }
    __syncthreads();
    if (!sm.last) return;
    __threadfence();
    for (int e = tid; e < nsplit * kout; e += SWEEP_WARPS * 32) {
      const size_t q = (p0 + e / kout) * a.KP + e % kout;
      (&sm.val[0][0])[e] = __ldcg(sg.part_val + q);
      (&sm.id[0][0])[e] = __ldcg(sg.part_id + q);
    }
    merge_by_rank(sm, nsplit * kout, kout);
    if (warp == 0) {
      m = -INFINITY;
      s = 0.f;
      for (int c = lane; c < nsplit; c += 32) {
        const float pm = __ldcg(sg.part_m + p0 + c), ps = __ldcg(sg.part_s + p0 + c);
        if (pm == -INFINITY) continue;
        const float top = fmaxf(m, pm);
        s = (m == -INFINITY ? 0.f : s * ex2((m - top) * LOG2E)) + ps * ex2((pm - top) * LOG2E);
        m = top;
      }
      warp_lse_combine(m, s);
      if (lane == 0) sg.counters[row] = 0;
    }
  }
  if (warp == 0) write_row(sg, row, kout, m, s, sm.best_v[lane], sm.best_i[lane], a.status);
}


// ---------------------------------------------------------------- a warp a row
// Many rows, or short ones: a warp sweeps a row alone and keeps its best-first list over the lanes
// (lane k holds the k-th best), into which the few logits that reach the K-th best are inserted one
// by one. Bound by memory from some 3000 rows (4096 rows of 126464 bf16, K = 8: 6.7 TB/s) given L1 for
// its loads in flight, 128 KB an SM: with 100 KB of shared memory carved out instead of 64, 185 us
// instead of 156.
struct RowState {
  float m, s;      // this lane's running max and sum of exp(x - max)
  float wv;        // this lane's entry of the list
  int wi;
  float thr;       // lower bound on the row's K-th best, the same in all lanes
};

// Inserts (v, id), the same in all lanes; entries past kout keep (-inf, INVALID_ID).
__device__ __forceinline__ void list_insert(float v, int id, int kout, RowState& st) {
  const int lane = threadIdx.x & 31;
  const bool ahead = lane < kout && !better(v, id, st.wv, st.wi);   // entries that stay before it
  const int pos = __popc(__ballot_sync(FULL_MASK, ahead));
  const float uv = __shfl_up_sync(FULL_MASK, st.wv, 1);
  const int ui = __shfl_up_sync(FULL_MASK, st.wi, 1);
  if (lane < kout && lane >= pos) {
    st.wv = lane == pos ? v : uv;
    st.wi = lane == pos ? id : ui;
  }
  st.thr = fmaxf(st.thr, __shfl_sync(FULL_MASK, st.wv, kout - 1));
}

// Inserts the lanes' elements f (ids id) that reach the threshold and come before the list's last
// (not the many at a mask's value once the list is full of them).
__device__ __forceinline__ void insert_lanes(bool in, float f, int id, int kout, RowState& st) {
  const float last_v = __shfl_sync(FULL_MASK, st.wv, kout - 1);
  const int last_i = __shfl_sync(FULL_MASK, st.wi, kout - 1);
  unsigned hit = __ballot_sync(FULL_MASK, in && f >= st.thr && better(f, id, last_v, last_i));
  while (hit) {
    const int src = __ffs(hit) - 1;
    hit &= hit - 1;
    const float v = __shfl_sync(FULL_MASK, f, src);
    const int i = __shfl_sync(FULL_MASK, id, src);
    if (v >= st.thr) list_insert(v, i, kout, st);
  }
}

// One batch (as in sweep_batch). stash: 32 vectors of shared memory.
template <typename T>
__device__ __forceinline__ void row_batch(const uint4 (&w)[SWEEP_UNROLL], int id0_lane, int valid,
                                          int kout, uint4* stash, RowState& st) {
  constexpr int VN = Vec<T>::N;
  const int lane = threadIdx.x & 31;
  const float mx = raise_max<T>(w, st.m, st.s);
  add_batch<T>(w, st.m, st.s);
  const unsigned lanes = __ballot_sync(FULL_MASK, valid > 0 && mx >= st.thr);
  if (!lanes) return;
  if (__popc(lanes) >= kout) {   // kout lanes each hold a logit at least as large as this
    const unsigned key = order_key(mx);
    const unsigned kth = kout == 1 ? __reduce_max_sync(FULL_MASK, key)
                                   : __shfl_sync(FULL_MASK, warp_sort(key), 32 - kout);
    st.thr = fmaxf(st.thr, key_to_float(kth));
  }
#pragma unroll
  for (int u = 0; u < SWEEP_UNROLL; ++u) {
    unsigned hit = __ballot_sync(FULL_MASK, u < valid && vec_max(w[u], T()) >= st.thr);
    if (!hit) continue;
    stash[lane] = w[u];
    __syncwarp();
    do {   // lane j < VN reads logit j of the vector of lane src
      const int src = __ffs(hit) - 1;
      hit &= hit - 1;
      const T* e = reinterpret_cast<const T*>(stash + src);
      const float f = lane < VN ? to_f32(e[lane]) : -INFINITY;
      const int id = __shfl_sync(FULL_MASK, id0_lane, src) + u * 32 * VN + lane;
      insert_lanes(lane < VN, f, id, kout, st);
    } while (hit);
    __syncwarp();
  }
  // ids only grow from one batch to the next: a later logit has to exceed a full list's last
  const float last = __shfl_sync(FULL_MASK, st.wv, kout - 1);
  if (__shfl_sync(FULL_MASK, st.wi, kout - 1) != INVALID_ID)
    st.thr = fmaxf(st.thr, nextafterf(last, INFINITY));
}

// At most 64 registers a thread: 32 rows an SM.
template <typename T>
__global__ void __launch_bounds__(ROW_WARPS * 32, 32 / ROW_WARPS)
sweep_rows_kernel(const __grid_constant__ SweepSeg sg, int V, int32_t* status) {
  constexpr int VN = Vec<T>::N;
  __shared__ uint4 stash[ROW_WARPS][32];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int row = (int)blockIdx.x * ROW_WARPS + warp;
  if (row >= sg.rows) return;
  const int kout = sg.kout;
  const T* rowp = reinterpret_cast<const T*>(sg.logits) + (size_t)row * V;
  const uintptr_t addr = reinterpret_cast<uintptr_t>(rowp);
  const int head = min(V, (int)(((16u - (unsigned)(addr & 15u)) & 15u) / sizeof(T)));
  const int nvec = (V - head) / VN;
  RowState st{-INFINITY, 0.f, -INFINITY, INVALID_ID, -INFINITY};
  // the unaligned head and, at the end, the ragged tail: fewer than VN logits each
  auto ragged = [&](int first, int n) {
    const bool in = lane < n;
    const float f = in ? to_f32(rowp[first + lane]) : -INFINITY;
    if (in) lse_update(f, st.m, st.s);
    insert_lanes(in, f, first + lane, kout, st);
  };
  ragged(0, head);
  const uint4* vp = reinterpret_cast<const uint4*>(rowp + head) + lane;
  const uint32_t ninf = VN == 8 ? 0xff80ff80u : 0xff800000u;
  uint4 w[SWEEP_UNROLL];
  int base = 0;
  auto load = [&]() -> int {   // padded with -inf past the row
    const int left = nvec - base - lane;
    const int valid = left <= 0 ? 0 : min(SWEEP_UNROLL, (left + 31) / 32);
#pragma unroll
    for (int u = 0; u < SWEEP_UNROLL; ++u)
      w[u] = u < valid ? ld_stream_v4(vp + base + 32 * u) : make_uint4(ninf, ninf, ninf, ninf);
    return valid;
  };
  int valid = load();
  row_batch<T>(w, head + lane * VN, valid, kout, stash[warp], st);
  // full batches: no bounds checks
  for (base = SWEEP_BATCH; base + SWEEP_BATCH <= nvec; base += SWEEP_BATCH) {
#pragma unroll
    for (int u = 0; u < SWEEP_UNROLL; ++u) w[u] = ld_stream_v4(vp + base + 32 * u);
    row_batch<T>(w, head + (base + lane) * VN, SWEEP_UNROLL, kout, stash[warp], st);
  }
  if (base < nvec) {
    valid = load();
    row_batch<T>(w, head + (base + lane) * VN, valid, kout, stash[warp], st);
  }
  ragged(head + nvec * VN, V - head - nvec * VN);
  warp_lse_combine(st.m, st.s);
  write_row(sg, row, kout, st.m, st.s, st.wv, st.wi, status);
}

// Whether a warp sweeps a row alone (KP: K or a power of two above it). In short rows fewer than four
// warps of a CTA have a logit in every lane, too few for K <= 32 maxima to be published, and nothing
// would be screened out (4096 bf16 rows of 1000, K = 8: 161 us on a CTA a row, 16 so; 32 rows of
// 4000, K = 32: 91, 27). And where one warp a row fills the chip it spares the CTA's barriers and merge
// (4096 rows of 16000, K = 8: 53 us, 33; 2048 of 32000: 44, 40; of 64000: 62, 62; of 126464: 98, 101;
// 1536 of 32000: 36, 38). Past 3 vectors a row's length for every row a call of these rows alone
// still gains (4096 of 126464, K = 8: 175 us, 156), but beside the products of a tail it depends on
// which kernel is placed first (128 sequences: 372 or 374 us on a CTA a row, 352 or 379 so; 64 of 64
// rows of 151936: 524 or 533, 539 or 534; 2560 rows of 104000: 222, 234); with K > 16 it stays well
// ahead (4096 of 126464: 326, 197).
bool by_warp(int rows, int V, int dtype, int KP) {
  const int nvec = V / (dtype == BRISK_DT_BF16 ? 8 : 4);
  return nvec < ROW_SHORT || (rows >= ROW_MID && nvec <= 3ll * rows) || (rows >= ROW_MANY && KP > 16);
}

template <typename T>
cudaError_t launch_t(const SweepLaunch& a, cudaStream_t stream) {
  long long rows = a.seg[0].rows;
  if (a.nseg > 1) rows += a.seg[1].rows;
  if (by_warp(a.seg[0].rows, a.V, a.dtype, a.KP)) {
    cudaError_t e = set_up_kernel(sweep_rows_kernel<T>, ROW_CARVEOUT_KB);
    for (int i = 0; i < a.nseg && e == cudaSuccess; ++i)
      e = launch_prio(sweep_rows_kernel<T>, dim3((unsigned)((a.seg[i].rows + ROW_WARPS - 1) / ROW_WARPS)),
                      dim3(ROW_WARPS * 32), 0, stream, a.seg[i], a.V, a.status);
    return e != cudaSuccess ? e : cudaGetLastError();
  }
  cudaError_t e = set_up_kernel(sweep_kernel<T>, CARVEOUT_SMALL_KB);
  if (e != cudaSuccess) return e;
  e = launch_prio(sweep_kernel<T>, dim3((unsigned)(rows * a.nsplit)), dim3(SWEEP_WARPS * 32), 0, stream, a);
  if (e != cudaSuccess) return e;
  return cudaGetLastError();
}

}  // namespace

int kp_for(int K) {
  int kp = 4;
  while (kp < K) kp *= 2;
  return kp;
}

// Segments per row: enough CTAs to fill the chip once (16 sequences on one CTA a row would leave
// 96 of the 608 that fit idle, one sequence 576), each with at least one batch a warp, and
// no more than the merge holds. Independent of the device, so that the summation order, and hence
// every rounded result, is the same on every run.
int sweep_splits(int rows_per_tensor, int V, int dtype, int K) {
  const int vn = dtype == BRISK_DT_BF16 ? 8 : 4;
  const int batches = (V / vn + SWEEP_BATCH - 1) / SWEEP_BATCH;
  if (by_warp(rows_per_tensor, V, dtype, K)) return 1;
  int c = SWEEP_CTAS / rows_per_tensor;
  const int most = (batches + SWEEP_WARPS - 1) / SWEEP_WARPS;
  if (c > most) c = most;
  if (c > SWEEP_MERGE / K) c = SWEEP_MERGE / K;
  return c < 1 ? 1 : c;
}

cudaError_t launch_sweep(const SweepLaunch& a, cudaStream_t stream) {
  if (a.dtype == BRISK_DT_BF16) return launch_t<__nv_bfloat16>(a, stream);
  return launch_t<float>(a, stream);
}

}  // namespace brisk
