// Corrector scan and verification, one CTA per sequence.
//
// Corrector (Sec. 3.3 Eqs. 4-5; App. C.3 Eq. 9; Algorithm 1(b) loop). The
// minimal-GRU pre-activations are linear in the input blocks
// [P_h m_i ; P_e E_in(x_{i-1}) ; pos_i ; P_phi phi_i], so each block's share is
// read from a precomputed source:
//   hidden share   G[b,i]          (one dense product over all b, i, before the scan)
//   token share    Tzh[x_{i-1}]    (vocabulary table folded once per weight set)
//   position share posz[i], posh[i]
//   feature share  Fz phi_i, Fh phi_i   (S x 5 folded matrices)
// and the residual d_{i,k} = <W_s s_i, W_c E_out(c)> = <s_i, U[c]> with
// U = (E_out W_c^T) W_s. Init is u_0 = tanh(G0[b] + T0[x0]). What stays
// sequential per position is O(S) element work, K+1 dot products of length S
// and the K-way Select.
//
// Verification (Sec. 3.1; Sec. 3.3; App. B Eq. 6) runs in the same CTA after
// the scan, or alone (brisk_verify_block), through the same device code.
#include "brisk_internal.cuh"

namespace brisk {

namespace {

// Verification CTA: 128 threads, or 512 under stochastic verification, where a rejection
// resamples from a residual over the whole vocabulary row (a 126464-entry row: 112 us on 128
// threads with element loads and the precise exponential, 28 with 512 threads, vector loads and
// the hardware one, 12 with a cluster of 8 CTAs).
constexpr int VERIFY_THREADS = 128;
constexpr int VERIFY_THREADS_MAX = 512;
constexpr int VERIFY_CTAS = 152;       // CTAs up to which a residual walk is shared
constexpr int VERIFY_SHARE = 4096;     // ids of it a CTA has at least

struct Smem {
  int* cid;        // [L][K]
  int* sel;        // [L]
  int* rank;       // [L]
  float* ref;      // [L][K]
  float* bsum;     // [nblk]  residual block sums
  float* misc;     // [16]
  int* imisc;      // [16]
};

__host__ __device__ inline size_t align16(size_t x) { return (x + 15) & ~size_t(15); }

constexpr int RES_BLOCK = 256;  // residual-sampling block: 32 lanes x 8 ids
constexpr int RES_FLIGHT = 4;   // blocks whose logits a warp loads at once

__host__ __device__ inline size_t smem_layout(int L, int K, int S, int V, char* base, Smem* sm) {
  size_t off = 0;
  auto take = [&](size_t bytes) {
    const size_t o = off;
    off = align16(off + bytes);
    return base ? base + o : nullptr;
  };
  (void)S;
  const int nblk = (V + RES_BLOCK - 1) / RES_BLOCK;
  char* p_cid = take(sizeof(int) * L * K);
  char* p_sel = take(sizeof(int) * L);
  char* p_rank = take(sizeof(int) * L);
  char* p_ref = take(sizeof(float) * L * K);
  char* p_bsum = take(sizeof(float) * nblk);
  char* p_misc = take(sizeof(float) * 16);
  char* p_imisc = take(sizeof(int) * 16);
  if (sm) {
    sm->cid = (int*)p_cid; sm->sel = (int*)p_sel; sm->rank = (int*)p_rank; sm->ref = (float*)p_ref;
    sm->bsum = (float*)p_bsum; sm->misc = (float*)p_misc; sm->imisc = (int*)p_imisc;
  }
  return off;
}

__device__ __forceinline__ float4 ld4(const float* p) { return *reinterpret_cast<const float4*>(p); }

__device__ __forceinline__ float load_logit(const void* base, int dt, size_t idx) {
  if (dt == BRISK_DT_BF16) return __bfloat162float(reinterpret_cast<const __nv_bfloat16*>(base)[idx]);
  return reinterpret_cast<const float*>(base)[idx];
}

// Largest of one float per lane, none of them NaN (one warp reduction).
__device__ __forceinline__ float redux_max(float x) {
  float r;
  asm volatile("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(r) : "f"(x));
  return r;
}

// Select with lane k holding refined score k (lanes >= K hold -inf), K <= NP; the same in every
// lane.
// Greedy: argmax, the lowest rank on ties. Sample: the first rank whose cumulative softmax mass
// exceeds u * total (warp prefix sums), else the last rank with mass.
template <int NP = 32>
__device__ __forceinline__ int select_warp(float ref, int K, int mode, float u) {
  const int lane = threadIdx.x & 31;
  if (mode == BRISK_SELECT_GREEDY) {
    // a NaN score ranks as -inf, so every lane agrees on one rank in [0, K) whatever the
    // scores hold: the lowest rank holding the warp's largest score
    const float bv = (lane < K && !isnan(ref)) ? ref : -INFINITY;
    const float mx = redux_max(bv);   // (by the whole warp)
    const unsigned hit = __ballot_sync(FULL_MASK, lane < K && bv == mx);
    return hit ? __ffs(hit) - 1 : 0;
  }
  const float mx = redux_max(isnan(ref) ? -INFINITY : ref);
  const float w = lane < K ? expf(ref - mx) : 0.f;
  float cum = w;
#pragma unroll
  for (int off = 1; off < NP; off <<= 1) {
    const float o = __shfl_up_sync(FULL_MASK, cum, off);
    if (lane >= off) cum += o;
  }
  const float tot = __shfl_sync(FULL_MASK, cum, NP - 1);
  const unsigned hit = __ballot_sync(FULL_MASK, lane < K && cum > u * tot);
  if (hit) return __ffs(hit) - 1;
  const unsigned pos = __ballot_sync(FULL_MASK, w > 0.f);
  return pos ? 31 - __clz(pos) : 0;
}

// pi_i(rank r) of the proposal law induced by the Select rule.
__device__ __forceinline__ float proposal_mass(const float* ref, int K, int mode, int r) {
  if (mode == BRISK_SELECT_GREEDY) return 1.f;
  float mx = ref[0];
  for (int k = 1; k < K; ++k) mx = fmaxf(mx, ref[k]);
  float tot = 0.f;
  for (int k = 0; k < K; ++k) tot += expf(ref[k] - mx);
  return expf(ref[r] - mx) / tot;
}

// The logits of the 8 ids [v0, v0 + 8) owned by this lane (v0 is a multiple of 8, so a
// 16-byte-aligned row gives aligned 16-byte vector loads; ragged ends and unaligned rows take
// element loads). -inf past V.
__device__ __forceinline__ void logits8(const void* rowp, int dt, int V, int v0, float (&l)[8]) {
  const bool vec = v0 + 8 <= V && (reinterpret_cast<uintptr_t>(rowp) & 15u) == 0;
  if (vec && dt == BRISK_DT_BF16) {
    unpack(__ldg(reinterpret_cast<const uint4*>(reinterpret_cast<const __nv_bfloat16*>(rowp) + v0)),
           l, __nv_bfloat16());
  } else if (vec) {
    const uint4* q = reinterpret_cast<const uint4*>(reinterpret_cast<const float*>(rowp) + v0);
    float a[4], b[4];
    unpack(__ldg(q), a, 0.f);
    unpack(__ldg(q + 1), b, 0.f);
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      l[e] = a[e];
      l[4 + e] = b[e];
    }
  } else {
#pragma unroll
    for (int e = 0; e < 8; ++e) l[e] = v0 + e < V ? load_logit(rowp, dt, (size_t)(v0 + e)) : -INFINITY;
  }
}

// Residual R(v) = max(0, p(v) - pi(v)) of the 8 ids [v0, v0 + 8) with logits l, with
// p(v) = 2^(l(v) log2 e - lse log2 e) on the hardware exponential. Lanes k < K hold candidate k:
// (cand_id, cand_mass).
__device__ __forceinline__ void residual8(const float (&l)[8], float lse, int v0, int blk0,
                                         int cand_id, float cand_mass, int K, float (&R)[8]) {
  const int lane = threadIdx.x & 31;
  const float nlb = -lse * LOG2E;
#pragma unroll
  for (int e = 0; e < 8; ++e) R[e] = ex2(fmaf(l[e], LOG2E, nlb));
  const bool mine = lane < K && cand_id >= blk0 && cand_id < blk0 + RES_BLOCK;
  unsigned mask = __ballot_sync(FULL_MASK, mine);
  while (mask) {
    const int k = __ffs(mask) - 1;
    mask &= mask - 1;
    const int cid = __shfl_sync(FULL_MASK, cand_id, k);
    const float cm = __shfl_sync(FULL_MASK, cand_mass, k);
    const int rel = cid - v0;
#pragma unroll
    for (int e = 0; e < 8; ++e)
      if (rel == e) R[e] -= cm;
  }
#pragma unroll
  for (int e = 0; e < 8; ++e) R[e] = fmaxf(R[e], 0.f);
}

// Draw from the normalised [p - pi]_+ of verifier row `rowp` with uniform u, walking ids in
// ascending order; the verifier argmax when the residual mass is <= RESID_Z_FLOOR. CTA-wide.
// With `parts` CTAs of a cluster sharing the walk, each sums every parts-th run of blocks into the
// first CTA's shared memory, which goes on alone (the others return -1).
__device__ int residual_sample(const Smem& sm, const void* rowp, int dt, int V, float lse,
                               const int* cid, const float* ref, int K, int select_mode,
                               int sel_rank, float u, int argmax_p, int part, int parts) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nblk = (V + RES_BLOCK - 1) / RES_BLOCK;
  // candidate k's proposal mass, held by lane k
  int cand_id = -1;
  float cand_mass = 0.f;
  if (lane < K) {
    cand_id = cid[lane];
    if (select_mode == BRISK_SELECT_GREEDY) cand_mass = (lane == sel_rank) ? 1.f : 0.f;
    else cand_mass = proposal_mass(ref, K, select_mode, lane);
  }
  // pass 1: block sums, blocks interleaved over warps, the logits of RES_FLIGHT blocks on their
  // way at once (one at a time, the walk of a 126464-entry row waited 31 times for memory:
  // a call waits for memory most of the time)
  const int nw = (int)(blockDim.x >> 5) * parts;
  for (int base = part * (int)(blockDim.x >> 5) + warp; base < nblk; base += RES_FLIGHT * nw) {
    float l[RES_FLIGHT][8];
#pragma unroll
    for (int u = 0; u < RES_FLIGHT; ++u)   // (a block past the row reads as -inf)
      logits8(rowp, dt, V, (base + u * nw) * RES_BLOCK + lane * 8, l[u]);
#pragma unroll
    for (int u = 0; u < RES_FLIGHT; ++u) {
      const int blk = base + u * nw, blk0 = blk * RES_BLOCK;
      if (blk >= nblk) break;
      float R[8];
      residual8(l[u], lse, blk0 + lane * 8, blk0, cand_id, cand_mass, K, R);
      float t = 0.f;
#pragma unroll
      for (int e = 0; e < 8; ++e) t += R[e];
      t = warp_sum(t);
      if (lane == 0) {
        if (parts > 1) st_cluster(sm.bsum + blk, 0, t);
        else sm.bsum[blk] = t;
      }
    }
  }
  if (parts > 1) {
    cluster_sync();
    if (part) return -1;
  }
  __syncthreads();
  // warp 0: total mass and the block holding the target
  if (warp == 0) {
    const int per = (nblk + 31) / 32;
    const int b0 = lane * per, b1 = min(nblk, b0 + per);
    float mine = 0.f;
    for (int b = b0; b < b1; ++b) mine += sm.bsum[b];
    float incl = mine;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const float o = __shfl_up_sync(FULL_MASK, incl, off);
      if (lane >= off) incl += o;
    }
    const float Z = __shfl_sync(FULL_MASK, incl, 31);
    const float target = u * Z;
    int found = -1;
    float before = 0.f;
    // first lane whose run holds the target, then the block inside the run
    const unsigned hit = __ballot_sync(FULL_MASK, incl > target && b1 > b0);
    if (hit) {
      const int l = __ffs(hit) - 1;
      if (lane == l) {
        float acc = incl - mine;
        for (int b = b0; b < b1; ++b) {
          if (acc + sm.bsum[b] > target) { found = b; break; }
          acc += sm.bsum[b];
        }
        if (found < 0) found = b1 - 1;
        before = acc;
        sm.imisc[0] = found;
        sm.imisc[3] = 0;
        sm.misc[0] = before;
      }
    } else if (lane == 0) {
      // rounding put the target at or past the end: the last id with mass
      int lastb = -1;
      for (int b = nblk - 1; b >= 0; --b)
        if (sm.bsum[b] > 0.f) { lastb = b; break; }
      sm.imisc[0] = lastb;
      sm.imisc[3] = 1;
      sm.misc[0] = 0.f;
    }
    if (lane == 0) {
      sm.misc[1] = Z;
      sm.misc[2] = target;
    }
  }
  __syncthreads();
  const float Z = sm.misc[1];
  if (!(Z > RESID_Z_FLOOR)) return argmax_p;
  const int blk = sm.imisc[0];
  if (blk < 0) return argmax_p;
  // warp 0 walks the block: lane prefix sums, then the lane's 8 ids in order
  if (warp == 0) {
    const int blk0 = blk * RES_BLOCK;
    float l[8], R[8];
    logits8(rowp, dt, V, blk0 + lane * 8, l);
    residual8(l, lse, blk0 + lane * 8, blk0, cand_id, cand_mass, K, R);
    float mine = 0.f;
#pragma unroll
    for (int e = 0; e < 8; ++e) mine += R[e];
    float incl = mine;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const float o = __shfl_up_sync(FULL_MASK, incl, off);
      if (lane >= off) incl += o;
    }
    const float before = sm.misc[0];
    const float target = sm.misc[2];
    const bool past_end = sm.imisc[3] != 0;
    const unsigned hit = past_end ? 0u : __ballot_sync(FULL_MASK, before + incl > target);
    int pick = -1;
    if (hit) {
      const int l = __ffs(hit) - 1;
      if (lane == l) {
        float acc = before + incl - mine;
        int lastpos = -1;
        for (int e = 0; e < 8; ++e) {
          if (R[e] > 0.f) lastpos = e;
          acc += R[e];
          if (acc > target) { pick = blk0 + lane * 8 + e; break; }
        }
        if (pick < 0) pick = blk0 + lane * 8 + (lastpos < 0 ? 0 : lastpos);
      }
      pick = __shfl_sync(FULL_MASK, pick, l);
    } else {
      // the last id of the block with positive residual
      const unsigned pos = __ballot_sync(FULL_MASK, mine > 0.f);
      if (pos) {
        const int l = 31 - __clz(pos);
        if (lane == l) {
          int lastpos = 0;
          for (int e = 0; e < 8; ++e)
            if (R[e] > 0.f) lastpos = e;
          pick = blk0 + lane * 8 + lastpos;
        }
        pick = __shfl_sync(FULL_MASK, pick, l);
      } else {
        pick = argmax_p;
      }
    }
    if (lane == 0) sm.imisc[1] = pick;
  }
  __syncthreads();
  return sm.imisc[1];
}

// Left-to-right verification of sm.sel against the verifier rows of sequence b. part of parts:
// this CTA's place in a cluster that shares the residual walk (all of them find the same first
// rejection).
__device__ void verify_sequence(const ScanArgs& a, const Smem& sm, int b, int part = 0,
                                int parts = 1) {
  const int tid = threadIdx.x;
  const int L = a.L, K = a.K;
  if (tid == 0) sm.imisc[2] = L;
  __syncthreads();
  for (int t = tid; t < L; t += (int)blockDim.x) {
    const size_t bi = (size_t)b * L + t;
    const int x = sm.sel[t];
    bool ok;
    if (a.verify_mode == BRISK_VERIFY_GREEDY) {
      ok = (x == a.argmax_p[bi]);
    } else {
      const float lpx = load_logit(a.logits_p, a.logits_dt, bi * a.V + x);
      const float px = expf(lpx - a.lse_p[bi]);
      const float pim = proposal_mass(sm.ref + (size_t)t * K, K, a.select_mode, sm.rank[t]);
      const float alpha = fminf(1.f, px / pim);
      ok = a.u_acc[bi] < alpha;
    }
    if (!ok) atomicMin(&sm.imisc[2], t);
  }
  __syncthreads();
  const int j = sm.imisc[2];
  int corr = -1;
  if (j < L) {
    const size_t bj = (size_t)b * L + j;
    if (a.verify_mode == BRISK_VERIFY_GREEDY) {
      corr = a.argmax_p[bj];
    } else {
      const void* rowp = (a.logits_dt == BRISK_DT_BF16)
                             ? (const void*)(reinterpret_cast<const __nv_bfloat16*>(a.logits_p) + bj * a.V)
                             : (const void*)(reinterpret_cast<const float*>(a.logits_p) + bj * a.V);
      corr = residual_sample(sm, rowp, a.logits_dt, a.V, a.lse_p[bj], sm.cid + (size_t)j * K,
                             sm.ref + (size_t)j * K, K, a.select_mode, sm.rank[j], a.u_res[bj],
                             a.argmax_p[bj], part, parts);
    }
  }
  if (part) return;
  if (tid == 0) {
    a.accepted_len[b] = j;
    a.correction[b] = (j < L) ? corr : -1;
    if (a.next_anchor) a.next_anchor[b] = (j < L) ? corr : sm.sel[L - 1];
  }
  for (int t = tid; t < L; t += (int)blockDim.x)
    a.out_tokens[(size_t)b * L + t] = t < j ? sm.sel[t] : (t == j ? corr : -1);
}

// Verification of one sequence per CTA (Sec. 3.1; Sec. 3.3; App. B Eq. 6), reading the
// selections and refined scores the corrector wrote.
__global__ void __launch_bounds__(VERIFY_THREADS_MAX)
verify_kernel(const __grid_constant__ ScanArgs a) {
  extern __shared__ __align__(16) char smem_raw[];
  Smem sm;
  smem_layout(a.L, a.K, a.S, a.V, smem_raw, &sm);
  const int b = blockIdx.x / a.parts;
  const int tid = threadIdx.x;
  const int L = a.L, K = a.K, V = a.V;
  const size_t bL = (size_t)b * L;
  if (a.parts > 1) cluster_sync();   // every CTA runs before its shared memory is written
  // Ids are gathered with below, so out-of-range ones (a row with no finite logit leaves
  // placeholder ids; caller-provided ids may be anything) are replaced by 0 and reported.
  const int nt = (int)blockDim.x;
  for (int e = tid; e < L * K; e += nt) {
    int c = a.cand_ids[bL * K + e];
    if (c < 0 || c >= V) { set_status(a.status, BRISK_ERR_NUMERIC); c = 0; }
    sm.cid[e] = c;
    sm.ref[e] = a.refined[bL * K + e];
  }
  for (int e = tid; e < L; e += nt) {
    int x = a.sel_tokens[bL + e];
    if (x < 0 || x >= V) { set_status(a.status, BRISK_ERR_INVALID_ARG); x = 0; }
    sm.sel[e] = x;
  }
  __syncthreads();
  // each selection's rank in its candidate list
  for (int i = tid; i < L; i += nt) {
    int r = 0;
    for (int k = 0; k < K; ++k)
      if (sm.cid[i * K + k] == sm.sel[i]) { r = k; break; }
    sm.rank[i] = r;
  }
  __syncthreads();
  verify_sequence(a, sm, b, (int)blockIdx.x - b * a.parts, a.parts);
}

// ---------------------------------------------------------------- corrector
constexpr int CORR_SPAN = 128;   // state elements a computing warp owns, 4 a lane
constexpr int CORR_PART = 8;     // slots for the dots' parts: S <= 1024, so at most 8 warps
constexpr int CORR_DEPTH = 4;    // positions the ring holds at most
constexpr int CORR_AHEAD = 3;    // positions whose rows are asked into L2 ahead of use
constexpr int CORR_OTHERS = 64;  // threads of a sequence that do not compute

struct CorrSmem {
  uint64_t* full;  // [CORR_DEPTH] mbarriers: a stage's rows have landed
  int* gave_up;    // set once a computing thread's wait has run out
  int* cid;        // [L][K], with K copies of x0 before it
  float* clp;      // [L][K]
  float4* feat;    // [L][K]  features 2, 3, 4 given that rank k of the position before was fed on,
                   //         and the gate's share of all five features
  float2* gap;     // [L]     features 0 and 1
  float* usel;     // [L]
  int* base;       // [L]     base selections (same-state replay)
  float* red;      // [2][32][CORR_PART] the residual dots' parts, zero past the computing warps
  float* gpart;    // [2][CORR_PART]     the gate's parts
  float* ring;     // [depth][stage]: the token rows and residual rows of a position
  Smem v;          // selections, ranks and refined scores kept for verification in the same CTA
};

// Floats of one ring stage: the token rows of the first R candidates of the position before (2S
// each) and, with rows, the residual rows of the K candidates (S each).
__host__ __device__ inline int corr_stage(int K, int S, int R, bool rows) {
  return 2 * S * R + (rows ? K * S : 0);
}

// Shared memory of one sequence.
__host__ __device__ inline size_t corr_layout(int L, int K, int S, int V, int depth, int stage,
                                              bool verify, char* base, CorrSmem* sm) {
  size_t off = 0;
  auto take = [&](size_t bytes) {
    const size_t o = off;
    off = align16(off + bytes);
    return base ? base + o : nullptr;
  };
  char* pb = take(sizeof(uint64_t) * CORR_DEPTH);
  char* pc = take(sizeof(int) * (L + 1) * K);
  char* pl = take(sizeof(float) * L * K);
  char* pf = take(sizeof(float4) * L * K);
  char* pg = take(sizeof(float2) * L);
  char* pu = take(sizeof(float) * L);
  char* pq = take(sizeof(int) * L);
  char* pr = take(sizeof(float) * 2 * 32 * CORR_PART);
  char* pp = take(sizeof(float) * 2 * CORR_PART);
  char* pt = take(sizeof(float) * depth * stage);
  char* pw = take(sizeof(int));
  const size_t voff = off;
  if (sm) {
    sm->full = (uint64_t*)pb;
    sm->gave_up = (int*)pw;
    sm->cid = (int*)pc + K; sm->clp = (float*)pl; sm->feat = (float4*)pf; sm->gap = (float2*)pg;
    sm->usel = (float*)pu; sm->base = (int*)pq; sm->red = (float*)pr; sm->gpart = (float*)pp; sm->ring = (float*)pt;
  }
  // with verification in the same CTA its tables follow (the candidate table is the corrector's)
  if (!verify) return off;
  Smem v;
  off = voff + smem_layout(L, K, S, V, base ? base + voff : nullptr, sm ? &v : nullptr);
  if (sm) {
    sm->v = v;
    sm->v.cid = sm->cid;
  }
  return off;
}

// Warp reduce-scatter of NP values per lane (NP = 8, 16 or 32): afterwards lane l holds the
// warp-wide sum of value (l >> log2(32 / NP)) & (NP - 1), that is value k sits in lane
// k * (32 / NP).
template <int NP>
__device__ __forceinline__ float reduce_scatter_n(float (&v)[NP]) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int m = 16, n = NP; n > 1; m >>= 1, n >>= 1) {
    const bool upper = (lane & m) != 0;
#pragma unroll
    for (int j = 0; j < n / 2; ++j) {
      const float send = upper ? v[j] : v[j + n / 2];
      const float keep = upper ? v[j + n / 2] : v[j];
      v[j] = keep + __shfl_xor_sync(FULL_MASK, send, m);
    }
  }
  float r = v[0];
#pragma unroll
  for (int m = 32 / NP / 2; m >= 1; m >>= 1) r += __shfl_xor_sync(FULL_MASK, r, m);
  return r;
}

// Asynchronous bulk copy of `bytes` (a multiple of 16) into shared memory, counted on `bar`.
__device__ __forceinline__ void bulk_load(float* dst, const float* src, unsigned bytes,
                                          uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
          su32(dst)),
      "l"(src), "r"(bytes), "r"(su32(bar))
      : "memory");
}
// Asks for `bytes` (a multiple of 16) at p in L2, to be kept there ahead of streamed data (a
// concurrent sweep replaces the whole of L2 within 20 us).
__device__ __forceinline__ uint64_t keep_policy() {
  uint64_t p;
  asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(p));
  return p;
}
__device__ __forceinline__ void prefetch_l2(const float* p, unsigned bytes, uint64_t policy) {
  asm volatile("cp.async.bulk.prefetch.L2.global.L2::cache_hint [%0], %1, %2;" ::"l"(p), "r"(bytes),
               "l"(policy));
}
// The block's barrier, for code that only some warps run. (It wants its warps whole, which a wait
// that lanes leave one by one does not promise.)
__device__ __forceinline__ void block_sync(int threads) {
  __syncwarp();
  asm volatile("bar.sync 0, %0;" ::"r"(threads) : "memory");
}
// Bounded wait for the phase of the given parity (more than `limit` SM cycles: false).
__device__ __forceinline__ bool mbar_wait_limit(uint64_t* bar, uint32_t parity, long long limit) {
  if (mbar_test(bar, parity)) return true;
  const long long t0 = clock64();
  while (!mbar_test(bar, parity))
    if (clock64() - t0 > limit) return false;
  return true;
}
// Packed fp32 pairs of four elements: w x + y, and the sum of x y.
__device__ __forceinline__ float4 fma4(const float4& w, const float2& x, const float4& y) {
  const float2 lo = __ffma2_rn(make_float2(w.x, w.y), x, make_float2(y.x, y.y));
  const float2 hi = __ffma2_rn(make_float2(w.z, w.w), x, make_float2(y.z, y.w));
  return make_float4(lo.x, lo.y, hi.x, hi.y);
}
__device__ __forceinline__ float4 fma4(const float4& w, float x, const float4& y) {
  return fma4(w, make_float2(x, x), y);
}
__device__ __forceinline__ float4 add4(const float4& x, const float4& y) {
  const float2 lo = __fadd2_rn(make_float2(x.x, x.y), make_float2(y.x, y.y));
  const float2 hi = __fadd2_rn(make_float2(x.z, x.w), make_float2(y.z, y.w));
  return make_float4(lo.x, lo.y, hi.x, hi.y);
}
__device__ __forceinline__ float dot4(const float4& x, const float4& y) {
  const float2 p = __ffma2_rn(make_float2(x.z, x.w), make_float2(y.z, y.w),
                              __fmul2_rn(make_float2(x.x, x.y), make_float2(y.x, y.y)));
  return p.x + p.y;
}
// Logistic function on the hardware exponential and reciprocal (relative error about 1e-7 for small
// |x|, 1e-6 at -20: that of the exponential's rounded argument).
__device__ __forceinline__ float rcp_hw(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float sigmoid_hw(float x) { return rcp_hw(1.f + ex2(-LOG2E * x)); }

// The sequential corrector (Sec. 3.3 Eqs. 4-5; App. C.3 Eq. 9; Algorithm 1(b) loop). What bounds
// it is the number of instructions on the dependent chain of a position (a lone warp issues one
// about every 8 cycles), and beside it the ones that every warp repeats; so few warps compute and
// the rest of the work is done by others or beforehand (32 positions, S = 512, K = 8: one sequence
// 41 us with eight computing warps that load for themselves, now 27; 16 sampled ones 63, now 41). A
// sequence has ceil(S / 128) computing warps that own four state elements a lane. A position is:
//  - the minimal-GRU step on the lane's elements, its residual-dot and gate partials (packed
//    fp32 pairs), a warp reduce-scatter, the warps' parts to shared memory, one barrier;
//  - gate, refined scores and Select, in every warp alike: lane k adds the parts of candidate k.
// A copying warp fetches the token rows of the first R candidates (one of which is usually fed
// forward) and, with ROWS, the residual rows into a ring of `depth` positions by bulk copies, a
// row a lane; a rank past R reads its token row through L2, and without ROWS the computing warps
// load the residual rows themselves. One more warp asks rows into L2 some positions ahead (where
// the ring is shallow) and stores the outputs. A warp issues a copy or an ask in some 50 cycles,
// which bounds positions with many candidates, so it asks for no token rows past the first R (with
// all K of them 128 sequences of K = 32, S = 512 took 173 us, now 115; K = 16, S = 1024 123, now 113). The
// features of every (position, rank fed forward) pair are tabulated first; the shares of a position
// that do not depend on the selection are summed before the barrier of the position before. (One CTA
// an SM is asked of the compiler: left to itself it settles on 80 to 103 registers, some spilled on
// the chain, and one sequence's graph replay takes 61 us, not 51.)
// LONE does not change the code: it makes a separate kernel whose shared-memory carveout preference
// gives a call without a sweep beside it all that an SM has. Not without ROWS: the residual rows'
// loads then want L1 (K = 32, one sequence of 61 positions: S = 864 180 us with it, 163 without;
// S = 1024 187, 169).
template <int NP, bool ROWS, bool SAMPLE, bool VERIFY, bool LONE>
__global__ void __launch_bounds__(32 * CORR_PART + CORR_OTHERS, 1)
corrector_kernel(const __grid_constant__ ScanArgs a) {
  extern __shared__ __align__(16) char smem_raw[];
  const int L = a.L, K = a.K, S = a.S, V = a.V, R = a.tok_ranks, D = a.ring_depth;
  const int stage = corr_stage(K, S, R, ROWS);
  const int b = blockIdx.x, NT = blockDim.x;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int NC = NT - CORR_OTHERS;   // computing threads
  auto sync = [&] { block_sync(NT); };
  CorrSmem sm;
  corr_layout(L, K, S, V, D, stage, VERIFY, smem_raw, &sm);
  const size_t bL = (size_t)b * L;
  constexpr int MODE = SAMPLE ? BRISK_SELECT_SAMPLE : BRISK_SELECT_GREEDY;

  // Prologue: the candidate table, then what depends on it.
  int x0 = a.x0[b];
  if (x0 < 0 || x0 >= V) {
    if (tid == 0) set_status(a.status, BRISK_ERR_INVALID_ARG);
    x0 = 0;
  }
  for (int e = tid; e < L * K; e += NT) {
    int c = a.cand_ids[bL * K + e];
    if (c < 0 || c >= V) { set_status(a.status, BRISK_ERR_NUMERIC); c = 0; }
    sm.cid[e] = c;
    sm.clp[e] = a.cand_logprob[bL * K + e];
  }
  if (tid < K) sm.cid[tid - K] = x0;
  for (int i = tid; i < L; i += NT) sm.usel[i] = SAMPLE ? a.u_sel[bL + i] : 0.f;
  for (int e = tid; e < 2 * 32 * CORR_PART; e += NT) sm.red[e] = 0.f;
  if (tid < 2 * CORR_PART) sm.gpart[tid] = 0.f;
  if (tid == 0) {
    *sm.gave_up = 0;
    for (int d = 0; d < CORR_DEPTH; ++d) mbar_init(&sm.full[d], 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    fence_async_smem();
  }
  sync();

  // the features of every position for every rank that may be fed forward (position 0: x0)
  auto features = [&] {
    const void* lq = a.logits_q;
    float w[5];
#pragma unroll
    for (int f = 0; f < 5; ++f) w[f] = a.wg[S + f];
    for (int e = tid; e < L * K; e += NT) {
      const int i = e / K, k = e - i * K;
      const int* ci = sm.cid + i * K;
      const int x = sm.cid[e - K];
      const size_t row = (bL + i) * V;
      const float l0 = load_logit(lq, a.logits_dt, row + ci[0]);
      const float l1 = load_logit(lq, a.logits_dt, row + ci[1]);
      const float l3 = load_logit(lq, a.logits_dt, row + ci[3]);
      const float lx = load_logit(lq, a.logits_dt, row + x);
      const float phi0 = l0 - l1, phi1 = l0 - l3, phi4 = l0 - lx;
      const float phi2 = x == ci[0] ? 1.f : 0.f;
      const float phi3 = x == ci[0] || x == ci[1] || x == ci[2] || x == ci[3] ? 1.f : 0.f;
      if (k == 0) sm.gap[i] = make_float2(phi0, phi1);
      float g = a.b_g;
      g = fmaf(w[0], phi0, g); g = fmaf(w[1], phi1, g); g = fmaf(w[2], phi2, g);
      g = fmaf(w[3], phi3, g); g = fmaf(w[4], phi4, g);
      sm.feat[e] = make_float4(phi2, phi3, phi4, g);
    }
  };

  const float sig_alpha = sigmoidf_(a.alpha);
  // gate, refined scores and Select of position i: every lane gets the selection, lane k the
  // refined score of candidate k; `share` is the gate's share of the features
  auto decide = [&](int i, float share, float& ref) -> int {
    const float* red = sm.red + ((i & 1) * 32 + lane) * CORR_PART;
    const float* gp = sm.gpart + (i & 1) * CORR_PART;
    const float lp = lane < K ? sm.clp[i * K + lane] : -INFINITY;
    const float4 d0 = ld4(red), q0 = ld4(gp);
    float dk = (d0.x + d0.y) + (d0.z + d0.w);
    float gs = (q0.x + q0.y) + (q0.z + q0.w);
    if (NC > 128) {
      const float4 d1 = ld4(red + 4), q1 = ld4(gp + 4);
      dk += (d1.x + d1.y) + (d1.z + d1.w);
      gs += (q1.x + q1.y) + (q1.z + q1.w);
    }
    ref = fmaf(sig_alpha * sigmoid_hw(share + gs), dk, lp);   // (lanes past K: dk = 0)
    return select_warp<NP>(ref, K, MODE, SAMPLE ? sm.usel[i] : 0.f);
  };
  // the token fed forward: the head's selection, or in a same-state replay the base selection
  // (the Select rule on the base scores log q, same draw), which is tabulated too
  auto base_ranks = [&] {
    if (!a.base_prefix) return;
    for (int i = warp; i < L; i += NT / 32) {
      const int pick = select_warp<NP>(lane < K ? sm.clp[i * K + lane] : -INFINITY, K, MODE,
                                       SAMPLE ? sm.usel[i] : 0.f);
      if (lane == 0) {
        sm.base[i] = pick;
        a.base_rank[bL + i] = pick;
      }
    }
  };

  if (tid < NC) {
    const bool owns = 4 * tid < S;           // state elements 4 tid .. 4 tid + 3
    const int e4 = owns ? 4 * tid : 0;       // (others keep a zero state)
    const float4 g0 = __ldcg(reinterpret_cast<const float4*>(a.G0 + (size_t)b * S + e4));
    const float4 t0 = __ldcg(reinterpret_cast<const float4*>(a.T0 + (size_t)x0 * S + e4));
    const float* gp = a.G + bL * 2 * S + e4;
    float4 zb = __ldcg(reinterpret_cast<const float4*>(gp));
    float4 hb = __ldcg(reinterpret_cast<const float4*>(gp + S));
    float4 fz[5], fh[5];                     // feature shares of the four elements, by feature
    {
      float z[20], h[20];
#pragma unroll
      for (int q = 0; q < 5; ++q) {
        *reinterpret_cast<float4*>(z + 4 * q) = ld4(a.Fz + 5 * e4 + 4 * q);
        *reinterpret_cast<float4*>(h + 4 * q) = ld4(a.Fh + 5 * e4 + 4 * q);
      }
#pragma unroll
      for (int f = 0; f < 5; ++f) {
        fz[f] = make_float4(z[f], z[5 + f], z[10 + f], z[15 + f]);
        fh[f] = make_float4(h[f], h[5 + f], h[10 + f], h[15 + f]);
      }
    }
    const float4 wg = ld4(a.wg + e4);
    features();
    base_ranks();
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);   // s_{-1} = u_0 = Init(h_c, E(x0))
    if (owns) s = make_float4(tanhf(g0.x + t0.x), tanhf(g0.y + t0.y), tanhf(g0.z + t0.z),
                              tanhf(g0.w + t0.w));
    auto give_up = [&] {                     // tells the copying warp
      *const_cast<volatile int*>(sm.gave_up) = 1;
      return false;
    };
    bool alive = mbar_wait_limit(&sm.full[0], 0, a.wait_limit) || give_up();
    sync();
    {
      const float2 gap = sm.gap[0];
      zb = fma4(fz[0], gap.x, fma4(fz[1], gap.y, zb));
      hb = fma4(fh[0], gap.x, fma4(fh[1], gap.y, hb));
    }
    const float* st = sm.ring + e4;          // this lane's place in the present stage
    int prank = 0, slot = 0, parity = 0;
    for (int i = 0; i < L; ++i) {
      const bool more = i + 1 < L;
      const float4 ft = sm.feat[i * K + prank];
      float4 tz, th;
      if (prank < R) {
        const float* t = st + 2 * S * prank;
        tz = ld4(t);
        th = ld4(t + S);
      } else {
        const float* t = a.Tzh + (size_t)sm.cid[(i - 1) * K + prank] * 2 * S + e4;
        tz = __ldcg(reinterpret_cast<const float4*>(t));
        th = __ldcg(reinterpret_cast<const float4*>(t + S));
      }
      float4 nz, nh;                          // the next position's hidden shares, on their way
      if (more) {
        gp += 2 * S;
        nz = __ldcg(reinterpret_cast<const float4*>(gp));
        nh = __ldcg(reinterpret_cast<const float4*>(gp + S));
      }
      // minimal-GRU step: s + z (h - s)
      zb = fma4(fz[2], ft.x, fma4(fz[3], ft.y, fma4(fz[4], ft.z, zb)));
      hb = fma4(fh[2], ft.x, fma4(fh[3], ft.y, fma4(fh[4], ft.z, hb)));
      const float4 z = add4(zb, tz);
      float4 h = add4(hb, th);
      h = fma4(s, -1.f, h);
      if (owns) {
        const float2 lo = __ffma2_rn(make_float2(sigmoid_hw(z.x), sigmoid_hw(z.y)),
                                     make_float2(h.x, h.y), make_float2(s.x, s.y));
        const float2 hi = __ffma2_rn(make_float2(sigmoid_hw(z.z), sigmoid_hw(z.w)),
                                     make_float2(h.z, h.w), make_float2(s.z, s.w));
        s = make_float4(lo.x, lo.y, hi.x, hi.y);
      }
      // residual-dot and gate partials
      float part[NP];
      const float* ur = st + 2 * S * R;
#pragma unroll
      for (int k = 0; k < NP; ++k) {
        const int kk = k < K ? k : K - 1;
        float4 u;
        if constexpr (ROWS) u = ld4(ur + kk * S);
        else u = __ldcg(reinterpret_cast<const float4*>(a.U + (size_t)sm.cid[i * K + kk] * S + e4));
        part[k] = dot4(u, s);
      }
      const float g = warp_sum(dot4(wg, s));
      const float r = reduce_scatter_n<NP>(part);
      constexpr int LSTEP = 32 / NP;
      if ((lane & (LSTEP - 1)) == 0)
        sm.red[((i & 1) * 32 + lane / LSTEP) * CORR_PART + warp] = r;
      if (lane == 0) sm.gpart[(i & 1) * CORR_PART + warp] = g;
      if (more) {
        const float2 gap = sm.gap[i + 1];
        zb = fma4(fz[0], gap.x, fma4(fz[1], gap.y, nz));
        hb = fma4(fh[0], gap.x, fma4(fh[1], gap.y, nh));
        // the next position's rows: a wait that gave up is not repeated
        st += stage;
        if (++slot == D) {
          slot = 0;
          parity ^= 1;
          st = sm.ring + e4;
        }
        if (alive && !mbar_wait_limit(&sm.full[slot], parity, a.wait_limit)) alive = give_up();
      }
      sync();
      float ref;
      const int pick = decide(i, ft.w, ref);
      prank = a.base_prefix ? sm.base[i] : pick;
    }
    if (!alive) set_status(a.status, BRISK_ERR_TIMEOUT);
  } else if (tid < NC + 32) {
    // Rows of position p into a stage, a row a lane: token rows, residual rows. The computing warps
    // have waited for the stage's previous rows, so it may be armed again, unless a thread of theirs
    // gave up: they may still be on their way then, and nothing more is fetched. Position i's wait
    // (and flag) comes before the sync that opens pass i below; the flag is read, by the whole warp
    // at once, in that pass, and position i's stage is armed again in the next one. (A look at the
    // barrier itself, or a vote on the flag, makes narrow states 2 to 4 % slower.)
    const int rows = R + (ROWS ? K : 0);
    int armed = 0;                        // positions fetched so far
    bool live = true;
    auto fetch = [&](int p, int slot) {
      if (p >= L || !live) return;
      armed = p + 1;
      float* base = sm.ring + slot * stage;
      const int* id = sm.cid + p * K;
      if (lane == 0) mbar_expect_tx(&sm.full[slot], (unsigned)stage * 4);
      __syncwarp();
      for (int j = lane; j < rows; j += 32) {
        if (j < R) bulk_load(base + 2 * S * j, a.Tzh + (size_t)id[j - K] * 2 * S, 8 * S, &sm.full[slot]);
        else bulk_load(base + 2 * S * R + (j - R) * S, a.U + (size_t)id[j - R] * S, 4 * S, &sm.full[slot]);
      }
      __syncwarp();
    };
    for (int p = 0; p < D - 1; ++p) fetch(p, p);
    features();
    base_ranks();
    sync();
    int slot = D - 1;                     // of position i + D - 1
    int stop = 0;
    for (int i = 0; i < L; ++i) {
      live = live && !stop;
      fetch(i + D - 1, slot);             // (its stage was last read before the sync just passed)
      slot = slot + 1 == D ? 0 : slot + 1;
      stop = *const_cast<volatile int*>(sm.gave_up);
      sync();
    }
    // a computing warp that gave up waiting leaves copies in flight: they end before the CTA does
    if (lane == 0)
      for (int p = max(0, armed - D); p < armed; ++p) mbar_drain(&sm.full[p % D], (p / D) & 1);
  } else {
    const uint64_t keep = keep_policy();
    auto ask = [&](int p) {
      if (!a.ask_rows || p >= L) return;
      if (lane == 0) prefetch_l2(a.G + (bL + p) * 2 * S, S * 8, keep);
      if (lane >= K) return;
      prefetch_l2(a.U + (size_t)sm.cid[p * K + lane] * S, S * 4, keep);
      if (lane < R && p + 1 < L)
        prefetch_l2(a.Tzh + (size_t)sm.cid[p * K + lane] * 2 * S, S * 8, keep);
    };
    for (int p = 0; p < CORR_AHEAD; ++p) ask(p);
    features();
    base_ranks();
    sync();
    int prank = 0;
    bool bad = false;
    for (int i = 0; i < L; ++i) {
      ask(i + CORR_AHEAD);
      sync();
      float ref;
      const int pick = decide(i, sm.feat[i * K + prank].w, ref);
      if (lane < K) a.refined[(bL + i) * K + lane] = ref;
      bad |= isnan(ref);
      if (lane == 0) a.sel_tokens[bL + i] = sm.cid[i * K + pick];
      if constexpr (VERIFY) {
        if (lane < K) sm.v.ref[i * K + lane] = ref;
        if (lane == 0) {
          sm.v.sel[i] = sm.cid[i * K + pick];
          sm.v.rank[i] = pick;
        }
      }
      prank = a.base_prefix ? sm.base[i] : pick;
    }
    if (bad) set_status(a.status, BRISK_ERR_NUMERIC);
  }
  // verification of this sequence in the same CTA (the verifier rows' statistics are complete:
  // their sweep ran before this kernel)
  if constexpr (VERIFY) {
    __syncthreads();
    verify_sequence(a, sm.v, b);
  }
}

}  // namespace

size_t scan_smem_bytes(int L, int K, int S, int V) {
  return smem_layout(L, K, S, V, nullptr, nullptr);
}

namespace {

// Shared memory a CTA may take; beside the verifier-row sweep (128 sequences, S = 512, K = 8):
// 377 us a decode tail with the corrector's 69 KB beside sweep CTAs, 382 us with two sequences'
// 210 KB on half as many SMs, which no sweep CTA shares.
constexpr size_t CORR_SMEM = 220 * 1024;
constexpr size_t CORR_SMEM_BESIDE = 76 * 1024;
constexpr int CORR_SMS = 152;

template <int NP, bool ROWS, bool SAMPLE, bool VERIFY, bool LONE>
cudaError_t launch_corrector_k(const ScanArgs& a, cudaStream_t stream) {
  const size_t smem = corr_layout(a.L, a.K, a.S, a.V, a.ring_depth,
                                  corr_stage(a.K, a.S, a.tok_ranks, ROWS), VERIFY, nullptr, nullptr);
  auto kernel = corrector_kernel<NP, ROWS, SAMPLE, VERIFY, LONE>;
  cudaError_t e = set_up_kernel(kernel, LONE ? CARVEOUT_FULL_KB : CARVEOUT_SMALL_KB, smem);
  if (e != cudaSuccess) return e;
  const int threads = 32 * ((a.S + CORR_SPAN - 1) / CORR_SPAN) + CORR_OTHERS;
  e = launch_prio(kernel, dim3(a.B), dim3(threads), smem, stream, a);
  if (e != cudaSuccess) return e;
  return cudaGetLastError();
}

template <int NP, bool ROWS, bool SAMPLE>
cudaError_t launch_corrector_m(const ScanArgs& a, cudaStream_t stream) {
  if (a.do_verify) return launch_corrector_k<NP, ROWS, SAMPLE, true, ROWS>(a, stream);
  return a.beside_sweep ? launch_corrector_k<NP, ROWS, SAMPLE, false, false>(a, stream)
                        : launch_corrector_k<NP, ROWS, SAMPLE, false, ROWS>(a, stream);
}
template <int NP>
cudaError_t launch_corrector_n(const ScanArgs& a, bool rows, cudaStream_t stream) {
  if (a.select_mode == BRISK_SELECT_SAMPLE)
    return rows ? launch_corrector_m<NP, true, true>(a, stream)
                : launch_corrector_m<NP, false, true>(a, stream);
  return rows ? launch_corrector_m<NP, true, false>(a, stream)
              : launch_corrector_m<NP, false, false>(a, stream);
}

cudaError_t launch_corrector(const ScanArgs& args, cudaStream_t stream) {
  ScanArgs a = args;
  a.wait_limit = wait_limit_cycles();
  auto bytes = [&](int depth, int ranks, bool rows) {
    return corr_layout(a.L, a.K, a.S, a.V, depth, corr_stage(a.K, a.S, ranks, rows),
                       a.do_verify != 0, nullptr, nullptr);
  };
  // Beside the verifier-row sweep a CTA stays within the sweep's carveout, with room for sweep CTAs
  // on its SM, where it can. Alone, more sequences than SMs share them (a state of up to 128, 256, 512
  // leaves registers for four, three, two) as far as the smallest ring with residual rows allows:
  // 608 sequences of 32 positions, K = 8: S = 128 97 us with the deepest ring, 74 so; S = 512 228,
  // 170; K = 32, S = 128 274, 170. (Rows left out of the ring for one more CTA an SM: 134 us there
  // with 4000 ids, but 407 instead of 358 with S = 512 and 60000 ids.)
  size_t room = a.beside_sweep && bytes(2, 1, true) <= CORR_SMEM_BESIDE ? CORR_SMEM_BESIDE : CORR_SMEM;
  if (!a.beside_sweep) {
    int n = a.S <= 128 ? 4 : (a.S <= 256 ? 3 : (a.S <= 512 ? 2 : 1));
    if (n > (a.B + CORR_SMS - 1) / CORR_SMS) n = (a.B + CORR_SMS - 1) / CORR_SMS;
    while (n > 1 && bytes(2, 1, true) > CORR_SMEM / n - 1024) --n;
    if (n > 1) room = CORR_SMEM / n - 1024;
  }
  // the ring's depth, the token rows a stage holds, and whether it holds the residual rows: the
  // first of these that fits
  struct Shape { int depth, ranks; bool rows; };
  const Shape shapes[] = {{4, 4, true}, {3, 4, true}, {3, 2, true}, {3, 1, true}, {2, 2, true},
                          {2, 1, true}, {4, 4, false}, {3, 2, false}, {2, 1, false}};
  bool rows = false;
  for (const Shape& s : shapes) {
    a.ring_depth = s.depth;
    a.tok_ranks = s.ranks;
    rows = s.rows;
    if (bytes(s.depth, s.ranks, s.rows) <= room) break;
  }
  a.ask_rows = a.ring_depth < 4;
  if (a.K <= 8) return launch_corrector_n<8>(a, rows, stream);
  if (a.K <= 16) return launch_corrector_n<16>(a, rows, stream);
  return launch_corrector_n<32>(a, rows, stream);
}

}  // namespace

// The corrector (do_select; with do_verify also the verification in the same CTA) or the
// verification alone (do_verify) for every sequence.
cudaError_t launch_scan(const ScanArgs& a, cudaStream_t stream) {
  if (a.do_select) return launch_corrector(a, stream);
  ScanArgs v = a;
  // A rejection walks a whole vocabulary row: clusters of up to 8 CTAs a sequence while there are
  // SMs for them (16 sequences: 28 us alone, 12 us so).
  v.parts = 1;
  if (a.verify_mode == BRISK_VERIFY_STOCHASTIC)
    while (v.parts < 8 && 2 * v.parts * a.B <= VERIFY_CTAS && a.V >= 2 * v.parts * VERIFY_SHARE)
      v.parts *= 2;
  const size_t smem = scan_smem_bytes(a.L, a.K, a.S, a.V);
  cudaError_t e = set_up_kernel(verify_kernel, CARVEOUT_SMALL_KB, smem);
  if (e != cudaSuccess) return e;
  const int threads = a.verify_mode == BRISK_VERIFY_STOCHASTIC ? VERIFY_THREADS_MAX : VERIFY_THREADS;
  e = launch_cluster(verify_kernel, dim3(a.B * v.parts), dim3(threads), smem, stream, v.parts, v);
  if (e != cudaSuccess) return e;
  return cudaGetLastError();
}

}  // namespace brisk
