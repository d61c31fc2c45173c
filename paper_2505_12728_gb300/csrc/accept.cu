// accept.cu -- fused speculative acceptance for sm_103a.
//
// The verification rule (Sec. 3.1; Sec. 3.3 names it the usual token-by-token
// accept/reject rule of speculative sampling): with
// p_i = softmax(target_logits_i / tau) and
// the draft distribution q_i, draft T'_{i+1} = x_i is accepted iff
// u_i * q_i(x_i) < p_i(x_i) (probability min(1, p/q)); decisions are taken in
// order up to the first rejection j; the token at position j is drawn by
// inverse CDF from norm(max(0, p_j - q_j)), or from the bonus row p_k when all
// k drafts were accepted.  tau <= 0 is greedy decoding (Sec. 4.2): accept iff
// x_i is the argmax of row i, and emit the argmax of row j.
//
// GB300 design.  The whole cost is streaming the (k+1) x V fp32 logits once
// (plus one row of q for the draw), so every kernel is a coalesced 128-bit
// streaming reduction spread over many CTAs, with no tensor cores, and the
// critical path is a short chain of memory round trips.  Three launch plans:
//  * V <= 16 x 2048: accept_cluster_kernel, one thread-block cluster per
//    sequence, the phases separated by cluster barriers (below);
//  * larger V: accept_chunks_kernel (every row in 1024-token chunks over
//    all SMs; the warp that completes a row combines its run records, the
//    one that completes a sequence takes the decisions) then
//    accept_draw_kernel (the residual draw in C2 CTAs per sequence over row
//    j, the last CTA of a sequence scanning for u_k * S);
//  * behind the fused LM head, whose projection already left per-CTA row
//    statistics: accept_decide_kernel then accept_draw_kernel (few rows,
//    one draft or many sequences of V <= 16 x 2048: the cluster kernel on the
//    projection's logits).
// Every launch uses programmatic stream serialisation: a kernel is resident
// while the previous one drains and waits for it (griddepcontrol.wait)
// before reading its results.
// Arithmetic: per-element terms are fp32 (2^x by the hardware approximation
// of explicitly rounded differences and products; the decisions' p(x) by
// expf on a float-float difference; a term recomputed within a draw is
// recomputed identically); sums, scans and the accept tests use float-float
// numbers (an unevaluated sum hi + lo of two fp32 values, ~44 significant
// bits) built from exactly rounded fp32 operations, accumulated in a fixed
// order (results are deterministic).
// GB300's fp64 pipe is far too slow for this latency-bound path, and
// float-float gives the accuracy the decisions need.
#include <climits>
#include <cmath>
#include <map>
#include <mutex>
#include <tuple>

#include "chunk_split.h"
#include "ff_math.cuh"
#include "sf_device.cuh"
#include "sf_host.h"

namespace sf {

constexpr int kAccThreads = kFfThreads;
constexpr int kAccWarps = kFfWarps;
// Rows are cut into segments of 1024 tokens (a warp, eight float4 per lane):
// the unit of the chunk records and of the draw's partial sums.
constexpr int kSegTokens = 1024;


struct alignas(16) RowStat {  // a target row, or a run of its chunks (one 16-byte load)
  float m;         // largest raw logit
  int arg;         // its first index
  ff S;            // sum of exp((x - m) / tau); 0 for greedy rows
};

struct alignas(16) SeqState {  // what the draw needs, in one 16-byte load
  int j1;          // first rejected position (k if none) + 1; 0: no decision (between calls; greedy)
  float m;         // row j's largest raw logit
  ff S;            // row j's sum of exp((x - m) / tau)
};

struct alignas(32) DrawPart {  // one segment of row j: a 32-byte sector, written by one warp
  ff sum_r;        // residual (or bonus) mass of the segment
  ff sum_p;        // target mass of the segment (fallback when the residual is 0)
};

struct AccParams {
  const float *logits;     // [B][k+1][V]
  const float *q;          // [B][k][V]
  const int32_t *tokens;   // [B][k]
  const float *u;          // [B][k+1]
  const float *tau;        // [B]
  int32_t *num_accepted;   // [B]
  int32_t *out_tokens;     // [B][k+1]
  float *ratio;            // [B][k] or null
  uint32_t *status;
  uint32_t *draw_tickets;  // [B]
  uint32_t *row_tickets;   // [B][k+1]: runs of a row whose record is written (chunk kernel)
  uint32_t *seq_tickets;   // [B]: rows of a sequence whose statistics are final
  RowStat *runs;           // [B][k+1][C1]: per row, one record per run of the chunk kernel
  RowStat *rows;           // [B][k+1]
  SeqState *seqs;          // [B]
  DrawPart *parts;         // [B][C1]
  int B, k, V;
  int C1;                  // segments per row: ceil(V / kSegTokens)
  int C2;                  // draw CTAs per row: ceil(C1 / kAccWarps)
  int NW1;                 // warps of the chunk kernel
  int vec4;                // rows are 16-byte aligned and V % 4 == 0
};


// exp((x - m) / tau) for the per-token loops (sums and draw terms); the
// decisions' p(x) use exp_diff_accurate.  Terms are summed four at a time in
// fp32 before each float-float add (a few 2^-24 of the partial).
__device__ __forceinline__ float exp_scaled(float x, float m, float tau) {
  const float d = __fsub_rn(x, m);
  return exp_fast(tau == 1.0f ? d : __fdiv_rn(d, tau));
}

__device__ __forceinline__ float sum4(float a, float b, float c, float d) {
  return __fadd_rn(__fadd_rn(a, b), __fadd_rn(c, d));
}

// Residual (j < k) or bonus (j == k) mass of one token and its target mass.
__device__ __forceinline__ void draw_terms(float x, float qx, bool residual, float m, float tau,
                                           float invS, float &r, float &pz) {
  pz = __fmul_rn(exp_scaled(x, m, tau), invS);
  r = residual ? fmaxf(__fsub_rn(pz, qx), 0.0f) : pz;
}

// What the decisions leave to the draw: the first rejected position j (k if
// none) and row j's largest logit and sum.
struct Decision {
  int j;
  float m;
  ff S;
};

// The k accept/reject decisions of sequence b by one warp.  Lane i <= k holds
// the final statistics of row i (max rm, first argmax rarg, float-float sum rS);
// lane i < k tests draft i: its token, uniform, the token's logit lx and draft
// probability qx (0 outside the vocabulary).  With `write`, every output is
// written except, for a sampled sequence, out_tokens[j], which the draw writes.
__device__ __forceinline__ Decision decide_core(const AccParams &p, int b, float tau, float rm, int rarg, ff rS,
                                                int tok, float u, float lx, float qx, bool write) {
  const int lane = threadIdx.x & 31, k = p.k;
  const bool greedy = !(tau > 0.0f);
  const bool in_range = tok >= 0 && tok < p.V;
  int acc = 0;
  if (lane < k) {
    float ratio = 0.f;
    if (!in_range) {
      if (write) set_status(p.status, SF_DEVICE_BAD_TOKEN);  // treated as a rejection
    } else if (greedy) {
      acc = tok == rarg;
      ratio = acc ? 1.f : 0.f;
    } else {
      // p(x) = exp((l_x - m) / tau) / S; accept iff u * q(x) < p(x), with the
      // product u * q kept exactly as float-float
      const float px = ff_div_to_f(exp_diff_accurate(lx, rm, tau), rS);
      const float uq = __fmul_rn(u, qx);
      const ff uqf = ff{uq, __fmaf_rn(u, qx, -uq)};
      acc = ff_lt(uqf, ff_of(px)) ? 1 : 0;
      ratio = qx > 0.f ? fminf(1.f, __fdiv_rn(px, qx)) : 1.f;
    }
    if (write && p.ratio) p.ratio[(size_t)b * k + lane] = ratio;
  }
  const unsigned rejected = __ballot_sync(0xffffffffu, lane < k && !acc);
  const int j = rejected ? __ffs(rejected) - 1 : k;
  const int arg_j = __shfl_sync(0xffffffffu, rarg, j);
  const Decision d = {j, __shfl_sync(0xffffffffu, rm, j),
                      ff{__shfl_sync(0xffffffffu, rS.hi, j), __shfl_sync(0xffffffffu, rS.lo, j)}};
  if (write && lane <= k) {
    int v = -1;
    if (lane < j) v = tok;
    else if (lane == j && greedy) v = arg_j;
    if (!(lane == j && !greedy)) p.out_tokens[(size_t)b * (k + 1) + lane] = v;
    if (lane == 0) p.num_accepted[b] = j;
  }
  return d;
}

// Lane i < k of a warp: draft token i of sequence b, its uniform, logit and
// draft probability (0 outside the vocabulary).
struct DraftEntry {
  int tok;
  float u, lx, qx;
};

__device__ __forceinline__ DraftEntry load_draft(const AccParams &p, int b) {
  const int lane = threadIdx.x & 31, k = p.k;
  DraftEntry d = {-1, 0.f, 0.f, 0.f};
  if (lane < k) {
    d.tok = p.tokens[(size_t)b * k + lane];
    d.u = p.u[(size_t)b * (k + 1) + lane];
    if (d.tok >= 0 && d.tok < p.V) {
      d.lx = p.logits[((size_t)b * (k + 1) + lane) * p.V + d.tok];
      d.qx = p.q[((size_t)b * k + lane) * p.V + d.tok];
    }
  }
  return d;
}

// Single-kernel acceptance for V <= 16 * kClusterMaxSlice: one thread-block
// cluster of cs CTAs per sequence, CTA `rank` owning tokens [rank * slice,
// (rank + 1) * slice) of every row.  It is a chain of latencies (a row is 128 KB
// at most), so the chain is short and its code, which runs once per launch and
// is fetched cold, is rolled over the rows:
//  1. every row's slice is copied to shared memory at once, or `bufs` rows at a
//     time (one bulk copy per row; with q_ahead also the draft rows' slices, of
//     which the draw needs one that is not known yet), and the draft tokens'
//     logits and probabilities are on their way meanwhile;
//  2. per row and warp the maximum, its first index and the float-float sum of
//     exp((x - max)/tau), combined over the slice and pushed into every CTA of
//     the cluster;
//  3. after the first cluster barrier every CTA combines the cs records of
//     each row in rank order and takes the decisions, identically; CTA 0
//     writes them.  Greedy clusters leave here;
//  4. each thread forms the residual (or bonus) terms of 8 consecutive tokens of
//     row j in registers; the slice's masses are pushed into every CTA;
//  5. after the second cluster barrier the CTA holding u_k * S finds the token
//     by a float-float scan over its threads' terms.
// Nobody touches a peer's shared memory after the second barrier.  Measured
// back to back (V = 32000): B = 1, k = 5 17.5 -> 11.4 us, greedy 5.2 -> 4.4; B = 16,
// k = 8 32.7 -> 23.1; B = 64, k = 4 77.3 -> 38.3 us, against the same phases with
// four barriers, the decisions in CTA 0 alone, row j read again from memory
// and the sums combined warp by warp.
constexpr int kClusterMax = 16;
constexpr int kClusterMaxSlice = 2048;
constexpr int kClusterPerThread = kClusterMaxSlice / kAccThreads;  // 8
// Draft rows are fetched ahead of the decision while they are few (B k V 4
// bytes, about a microsecond of the memory's time): the draw then doesn't wait
// for memory once more.
constexpr long long kAheadBytes = 8 << 20;
constexpr int kClusterFewBufs = 5;  // rows in shared memory at a time, where not all

struct alignas(16) ClusterRec {  // one row of one CTA's slice
  float m;
  int arg;
  ff S;
};

struct alignas(16) ClusterDraw {  // row j's terms in one CTA's slice
  ff sum;    // their mass
  int last;  // last index with mass (-1 if none)
  int pad;
};
static_assert(sizeof(ClusterRec) == 16 && sizeof(ClusterDraw) == 16, "record sizes");

// Dynamic shared memory: `bufs` rows' slices, then the k draft rows'.
static size_t cluster_smem(int k, int slice, int bufs, bool ahead) {
  return sizeof(float) * static_cast<size_t>(slice) * (bufs + (ahead ? k : 0));
}

// A partial sum relative to the maximum m, relative to the larger maximum to.
template <bool kExact>
__device__ __forceinline__ ff scale_sum(ff S, float m, float to, float tau) {
  if constexpr (kExact) return ff_mul(S, exp_diff_ff(m, to, tau));
  else return ff_mul(S, exp_diff_accurate(m, to, tau));
}

// kExact (behind the fused LM head): the row sums have the precision of the
// projection's statistics, which other sizes use there: terms of expf on a
// float-float difference, each added in float-float.  A slice's sum is scaled to
// the row's maximum by a float-float factor, since at most 16 factors, and not
// 152, average their errors.  Acceptance ratios against 64 bits, 40594 of nine
// sizes and three temperatures (rms / largest error): the statistics 5.7e-8 /
// 2.3e-7, this 5.7e-8 / 2.3e-7; the sums of sf_accept 7.4e-8 / 2.5e-7.
template <bool kExact>
__global__ void __launch_bounds__(kAccThreads)
accept_cluster_kernel(const __grid_constant__ AccParams p, int cs, int slice, int bufs, int q_ahead) {
  extern __shared__ __align__(128) float s_rows[];  // [bufs][slice], then [k][slice] of q
  __shared__ ClusterRec s_all[kClusterMax][SF_MAX_DRAFT + 1];  // pushed by every CTA of the cluster
  __shared__ ClusterDraw s_draws[kClusterMax];
  __shared__ float s_wm[SF_MAX_DRAFT + 1][kAccWarps];
  __shared__ int s_wi[SF_MAX_DRAFT + 1][kAccWarps];
  __shared__ ff s_part[SF_MAX_DRAFT + 1][kAccWarps];
  __shared__ float s_rm[SF_MAX_DRAFT + 1];
  __shared__ int s_rarg[SF_MAX_DRAFT + 1];
  __shared__ ff s_rS[SF_MAX_DRAFT + 1];
  __shared__ Decision s_dec;
  __shared__ ff s_scan[kAccWarps];
  __shared__ int s_last[kAccWarps], s_tok;
  __shared__ uint64_t s_bars[SF_MAX_DRAFT + 2];

  const int rank = blockIdx.x, b = blockIdx.y;
  const int tid = threadIdx.x, lane = tid & 31, warp = uniform_warp_id();
  const int k = p.k, V = p.V;
  const int x0 = min(V, rank * slice), len = min(V, x0 + slice) - x0;
  const uint32_t bars = smem_addr(s_bars);
  float *s_q = s_rows + static_cast<size_t>(bufs) * slice;
  if (tid == 0) {
    for (int r = 0; r <= k + 1; ++r) mbar_init(bars + 8u * r, 1);
    fence_mbar_init();
    s_tok = INT_MAX;
  }
  __syncthreads();
  cluster_arrive();        // this CTA has started
  grid_dependency_wait();  // logits, q, tokens and the outputs follow the previous kernel
  grid_launch_dependents();

  // ---- 1. copies ----
  const float *rows = p.logits + (size_t)b * (k + 1) * V + x0;
  const float *qrows = p.q + (size_t)b * k * V + x0;
  const bool bulk = p.vec4;  // rows are 16-byte aligned and their slices multiples of 16 bytes
  // rows r0 .. r0 + n - 1 into the buffers
  auto fetch = [&](int r0, int n) {
    if (bulk) {
      const uint32_t bytes = static_cast<uint32_t>(len) * 4u;
      for (int i = warp; i < n; i += kAccWarps) {
        if (elect_one()) {
          mbar_arrive_expect_tx(bars + 8u * i, bytes);
          bulk_copy_g2s(smem_addr(s_rows + static_cast<size_t>(i) * slice), rows + (size_t)(r0 + i) * V, bytes,
                        bars + 8u * i);
        }
        __syncwarp();
      }
    } else {
      for (int i = 0; i < n; ++i) {
#pragma unroll
        for (int t = 0; t < kClusterPerThread; ++t) {
          const int e = tid + kAccThreads * t;
          if (e < len) s_rows[static_cast<size_t>(i) * slice + e] = rows[(size_t)(r0 + i) * V + e];
        }
      }
      __syncthreads();
    }
  };
  fetch(0, min(bufs, k + 1));
  const float tau = p.tau[b];
  const bool greedy = !(tau > 0.0f);
  DraftEntry ent = {-1, 0.f, 0.f, 0.f};
  if (warp == 0) ent = load_draft(p, b);
  const float u_k = p.u[(size_t)b * (k + 1) + k];
  const bool ahead = q_ahead && !greedy;
  if (ahead) {
    const uint32_t bytes = static_cast<uint32_t>(len) * 4u, qb = bars + 8u * (k + 1);
    if (warp == kAccWarps - 1) {
      if (elect_one()) mbar_arrive_expect_tx(qb, bytes * static_cast<uint32_t>(k));
      __syncwarp();
      for (int r = 0; r < k; ++r) {
        if (elect_one())
          bulk_copy_g2s(smem_addr(s_q + static_cast<size_t>(r) * slice), qrows + (size_t)r * V, bytes, qb);
        __syncwarp();
      }
    }
  }
  bool landed = true;  // every copy waited for so far
  auto sum8 = [](const float (&t)[8]) {
    return ff_add(ff_add(two_sum(t[0], t[1]), two_sum(t[2], t[3])), ff_add(two_sum(t[4], t[5]), two_sum(t[6], t[7])));
  };

  // ---- 2. the slice's statistics: warp w takes tokens [256 w, 256 w + 256)
  // of every row, lane l tokens 128 h + 4 l .. + 3 of them ----
  auto load8 = [&](int buf, float (&v)[8]) {
    const float *row = s_rows + static_cast<size_t>(buf) * slice;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int e = 256 * warp + 128 * h + 4 * lane;
      const float4 x = e < slice ? *reinterpret_cast<const float4 *>(row + e) : make_float4(0.f, 0.f, 0.f, 0.f);
      v[4 * h] = e < len ? x.x : -INFINITY;
      v[4 * h + 1] = e + 1 < len ? x.y : -INFINITY;
      v[4 * h + 2] = e + 2 < len ? x.z : -INFINITY;
      v[4 * h + 3] = e + 3 < len ? x.w : -INFINITY;
    }
  };
  int r0 = 0;  // the buffers hold rows r0 .. r0 + bufs - 1
#pragma unroll 1
  for (uint32_t lap = 0;; ++lap) {
    const int n = min(bufs, k + 1 - r0);
#pragma unroll 1
    for (int i = 0; i < n; ++i) {
      if (bulk) landed &= mbar_wait_bounded(bars + 8u * i, lap & 1u);
      float v[8];
      load8(i, v);
      float bv = -INFINITY;
      int bi = INT_MAX;
#pragma unroll
      for (int t = 0; t < 8; ++t) {
        const int e = x0 + 256 * warp + 128 * (t / 4) + 4 * lane + (t % 4);
        if (better(v[t], e, bv, bi)) { bv = v[t]; bi = e; }
      }
      warp_argmax(bv, bi);
      ff S = ff_of(0.f);
      if (!greedy) {
        const float ref = bv == -INFINITY ? 0.f : bv;  // all masked: every term is 0
        if constexpr (kExact) {
          if (tau == 1.0f) {  // one branch for all: the divisions are skipped together
#pragma unroll
            for (int t = 0; t < 8; ++t) v[t] = exp_diff_accurate(v[t], ref, 1.0f);
          } else {
#pragma unroll
            for (int t = 0; t < 8; ++t) v[t] = exp_diff_accurate(v[t], ref, tau);
          }
          S = sum8(v);
        } else {
#pragma unroll
          for (int t = 0; t < 8; ++t) v[t] = __fsub_rn(v[t], ref);
          if (tau != 1.0f) {
#pragma unroll
            for (int t = 0; t < 8; ++t) v[t] = __fdiv_rn(v[t], tau);
          }
#pragma unroll
          for (int t = 0; t < 8; ++t) v[t] = exp_fast(v[t]);
          S = two_sum(sum4(v[0], v[1], v[2], v[3]), sum4(v[4], v[5], v[6], v[7]));
        }
        S = warp_sum_ff(S);
      }
      if (lane == 0) {
        s_wm[r0 + i][warp] = bv;
        s_wi[r0 + i][warp] = bi;
        s_part[r0 + i][warp] = S;
      }
    }
    if (r0 + bufs > k) break;
    if (bulk) fence_proxy_async_smem();  // this thread's reads before the next copies
    __syncthreads();
    r0 += bufs;
    fetch(r0, min(bufs, k + 1 - r0));
  }
  __syncthreads();
  cluster_wait();  // every peer has started
  for (int r = warp; r <= k; r += kAccWarps) {
    // the eight warps' records of row r, in warp order
    const float wm = lane < kAccWarps ? s_wm[r][lane] : -INFINITY;
    float mv = wm;
    int mi = lane < kAccWarps ? s_wi[r][lane] : INT_MAX;
    warp_argmax(mv, mi);
    ff S = lane < kAccWarps ? s_part[r][lane] : ff_of(0.f);
    if (ff_pos(S)) S = scale_sum<kExact>(S, wm, mv, tau);
    S = shfl_ff(warp_sum_ff<kAccWarps>(S), 0);
    if (lane < cs) {
      const uint32_t at = dsmem_addr(smem_addr(&s_all[rank][r]), static_cast<uint32_t>(lane));
      st_dsmem_f32x2(at, mv, __int_as_float(mi));
      st_dsmem_f32x2(at + 8, S.hi, S.lo);
    }
  }
  cluster_sync();

  // ---- 3. combine the slices of every row, in rank order, and decide ----
  for (int r = warp; r <= k; r += kAccWarps) {
    float cm = -INFINITY;
    int ci = INT_MAX;
    ff cS = ff_of(0.f);
    if (lane < cs) {
      cm = s_all[lane][r].m;
      ci = s_all[lane][r].arg;
      cS = s_all[lane][r].S;
    }
    float mv = cm;
    int mi = ci;
    warp_argmax(mv, mi);
    ff Sr = ff_of(0.f);
    if (!greedy && mv != -INFINITY) {
      if (lane < cs && ff_pos(cS)) Sr = scale_sum<kExact>(cS, cm, mv, tau);
      Sr = warp_sum_ff<kClusterMax>(Sr);
    }
    if (lane == 0) {
      s_rm[r] = mv;
      s_rarg[r] = mi;
      s_rS[r] = Sr;
    }
  }
  __syncthreads();
  if (warp == 0) {
    const int r = lane <= k ? lane : 0;
    const Decision d =
        decide_core(p, b, tau, s_rm[r], s_rarg[r], s_rS[r], ent.tok, ent.u, ent.lx, ent.qx, rank == 0);
    if (lane == 0) s_dec = d;
  }
  if (!__all_sync(0xffffffffu, landed) && lane == 0) set_status(p.status, SF_DEVICE_TIMEOUT);
  if (greedy) return;  // uniform over the cluster: the sequence is complete
  __syncthreads();

  // ---- 4. row j's residual (or bonus) terms, tokens 8 tid .. 8 tid + 7 ----
  const Decision dec = s_dec;
  const int j = dec.j;
  const bool residual = j < k;
  const float invS = ff_div_to_f(1.0f, dec.S);
  const int e0 = 8 * tid;
  float tr[8], tp[8];
  {
    float xv[8], qv[8];
    const bool here = j >= r0;  // row j is still in its buffer
    const float *row = s_rows + static_cast<size_t>(here ? j - r0 : 0) * slice;
    // four tokens of a row of the slice in global memory
    auto fetch4 = [&](const float *g, int e, float pad) -> float4 {
      if (bulk) return *reinterpret_cast<const float4 *>(g + e);
      return make_float4(g[e], e + 1 < len ? g[e + 1] : pad, e + 2 < len ? g[e + 2] : pad,
                         e + 3 < len ? g[e + 3] : pad);
    };
    if (ahead) {  // also when all drafts were accepted: the copies must have landed before the CTA ends
      if (!__all_sync(0xffffffffu, mbar_wait_bounded(bars + 8u * (k + 1), 0)) && lane == 0)
        set_status(p.status, SF_DEVICE_TIMEOUT);
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int e = e0 + 4 * h;
      float4 x = make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY), q = make_float4(0.f, 0.f, 0.f, 0.f);
      if (e < len) {
        x = here ? *reinterpret_cast<const float4 *>(row + e) : fetch4(rows + (size_t)j * V, e, -INFINITY);
        if (residual)
          q = ahead ? *reinterpret_cast<const float4 *>(s_q + static_cast<size_t>(j) * slice + e)
                    : fetch4(qrows + (size_t)j * V, e, 0.f);
      }
      xv[4 * h] = x.x; xv[4 * h + 1] = x.y; xv[4 * h + 2] = x.z; xv[4 * h + 3] = x.w;
      qv[4 * h] = q.x; qv[4 * h + 1] = q.y; qv[4 * h + 2] = q.z; qv[4 * h + 3] = q.w;
    }
#pragma unroll
    for (int t = 0; t < 8; ++t) tr[t] = tp[t] = 0.f;
    // the temperature is tested once, not once per term (its divisions are
    // skipped together)
    if (tau == 1.f) {
#pragma unroll
      for (int t = 0; t < 8; ++t)
        if (e0 + t < len) draw_terms(xv[t], qv[t], residual, dec.m, 1.f, invS, tr[t], tp[t]);
    } else {
#pragma unroll
      for (int t = 0; t < 8; ++t)
        if (e0 + t < len) draw_terms(xv[t], qv[t], residual, dec.m, tau, invS, tr[t], tp[t]);
    }
  }
  // the slice's mass of the terms t and its last index with mass, into every
  // CTA's s_draws; returns the thread's exclusive prefix
  auto publish = [&](const float (&t)[8]) -> ff {
    int last = -1;
#pragma unroll
    for (int i = 0; i < 8; ++i)
      if (t[i] > 0.f) last = x0 + e0 + i;
    last = __reduce_max_sync(0xffffffffu, last);
    if (lane == 0) s_last[warp] = last;
    ff tot;
    const ff ex = block_scan2(sum8(t), s_scan, &tot);  // its barriers order s_last too
    if (warp == 0) {
      last = __reduce_max_sync(0xffffffffu, lane < kAccWarps ? s_last[lane] : -1);
      if (lane < cs) {
        const uint32_t at = dsmem_addr(smem_addr(&s_draws[rank]), static_cast<uint32_t>(lane));
        st_dsmem_f32x2(at, tot.hi, tot.lo);
        st_dsmem_f32(at + 8, __int_as_float(last));
      }
    }
    return ex;
  };
  ff excl = publish(tr);
  cluster_sync();

  // ---- 5. the slice holding u_k * S draws the token ----
  // slice l covers [ex, in) of an inclusive scan over the slices, identical in
  // every warp of every CTA
  const bool have = lane < cs;
  ff in, ex, mass, total;
  auto scan_slices = [&]() {
    mass = have ? s_draws[lane].sum : ff_of(0.f);
    in = warp_scan_ff(mass, kClusterMax, &ex);
    total = shfl_ff(in, cs - 1);
  };
  scan_slices();
  if (!ff_pos(total)) {
    // a residual with no mass (rounding only): draw from the target's row
    // instead, the cluster once more round the same steps
#pragma unroll
    for (int t = 0; t < 8; ++t) tr[t] = tp[t];
    cluster_sync();  // every CTA has read its s_draws
    excl = publish(tr);
    cluster_sync();
    scan_slices();
  }
  const ff target = ff_mul(total, u_k);
  const unsigned hit = __ballot_sync(0xffffffffu, have && ff_pos(mass) && ff_lt(target, in) && !ff_lt(target, ex));
  int32_t *out = p.out_tokens + (size_t)b * (k + 1) + j;
  if (!hit) {
    // no slice holds the target (rounding): the last token with positive mass
    const int last = __reduce_max_sync(0xffffffffu, have ? s_draws[lane].last : -1);
    if (rank == 0 && tid == 0) *out = last;
    return;
  }
  const int cross = __ffs(hit) - 1;
  if (cross != rank) return;
  ff c = ff_add(shfl_ff(ex, cross), excl);
#pragma unroll
  for (int t = 0; t < 8; ++t) {
    c = ff_add(c, ff_of(tr[t]));
    if (tr[t] > 0.f && ff_lt(target, c)) {
      atomicMin(&s_tok, x0 + e0 + t);
      break;
    }
  }
  __syncthreads();
  if (tid == 0) *out = s_tok != INT_MAX ? s_tok : s_draws[rank].last;
}

// Combines the n records (max, first argmax, sum) of parts of a target row in
// order, kPer per lane and pass, into the row's max, first argmax and
// float-float sum rescaled to the max.  Executed by one whole warp; all loads
// of a pass are issued before any is used.
template <int kPer>
__device__ __forceinline__ RowStat combine_records(const float4 *rr, int n, float tau, bool greedy) {
  const int lane = threadIdx.x & 31;
  float mv = -INFINITY;
  int mi = INT_MAX;
  ff Sr = ff_of(0.f);
  for (int base = 0; base < n; base += 32 * kPer) {  // one pass unless n > 32 kPer
    float4 a[kPer];
#pragma unroll
    for (int t = 0; t < kPer; ++t) {
      const int i = base + lane + 32 * t;
      a[t] = i < n ? __ldcg(rr + i) : make_float4(-INFINITY, __int_as_float(INT_MAX), 0.f, 0.f);
    }
    float bm = -INFINITY;
    int bi = INT_MAX;
#pragma unroll
    for (int t = 0; t < kPer; ++t)
      if (better(a[t].x, __float_as_int(a[t].y), bm, bi)) { bm = a[t].x; bi = __float_as_int(a[t].y); }
    warp_argmax(bm, bi);
    if (!greedy) {
      // the pass's sums relative to its max, then the running sum moved to
      // the larger of the two maxima
      ff ps = ff_of(0.f);
#pragma unroll
      for (int t = 0; t < kPer; ++t) {
        const ff cS = ff{a[t].z, a[t].w};
        if (ff_pos(cS)) ps = ff_add(ps, ff_mul(cS, exp_diff_accurate(a[t].x, bm, tau)));
      }
      ps = warp_sum_ff(ps);
      if (bm > mv) {
        if (ff_pos(Sr)) Sr = ff_mul(Sr, exp_diff_accurate(mv, bm, tau));
        Sr = ff_add(Sr, ps);
      } else if (ff_pos(ps)) {
        Sr = ff_add(Sr, ff_mul(ps, exp_diff_accurate(bm, mv, tau)));
      }
    }
    if (better(bm, bi, mv, mi)) { mv = bm; mi = bi; }
  }
  return RowStat{mv, mi, Sr};
}

// Fused path: the decisions from the projection's per-CTA row statistics
// (launch_projection_stats, G records per row) instead of a pass over the
// logits.  grid (B), a warp for each of the k + 1 rows, its records in one
// round of loads (up to 160 of them).  With eight warps taking the rows in turn
// and two passes over the records, B = 7, k = 16, V = 32000 took 54.2 us with its
// projection and draw, against 49.8; B = 4, k = 8, V = 152064 194.3 against 192.1.
__global__ void __launch_bounds__(32 * (SF_MAX_DRAFT + 1))
accept_decide_kernel(const __grid_constant__ AccParams p, const SampStat *stats, int G) {
  __shared__ float s_rm[SF_MAX_DRAFT + 1];
  __shared__ int s_rarg[SF_MAX_DRAFT + 1];
  __shared__ ff s_rS[SF_MAX_DRAFT + 1];
  grid_dependency_wait();  // statistics and logits come from the projection
  grid_launch_dependents();
  const int b = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int k = p.k;
  const float tau = p.tau[b];
  DraftEntry e = {-1, 0.f, 0.f, 0.f};
  if (warp == 0) e = load_draft(p, b);  // in flight with the statistics
  const RowStat rs = combine_records<5>(
      reinterpret_cast<const float4 *>(stats + ((size_t)b * (k + 1) + warp) * G), G, tau, !(tau > 0.0f));
  if (lane == 0) {
    s_rm[warp] = rs.m;
    s_rarg[warp] = rs.arg;
    s_rS[warp] = rs.S;
  }
  __syncthreads();
  if (warp == 0) {
    const int r = lane <= k ? lane : 0;
    const Decision d = decide_core(p, b, tau, s_rm[r], s_rarg[r], s_rS[r], e.tok, e.u, e.lx, e.qx, true);
    if (lane == 0 && tau > 0.0f) p.seqs[b] = SeqState{d.j + 1, d.m, d.S};
  }
}

// The residual (j < k) or bonus (j == k) draw of sequence b (grid (C2, B)
// of kAccThreads threads; rs holds row j's max, argmax and sum).  Warp w of
// CTA c sums the residual and target masses of segment c * kAccWarps + w of
// row j (float-float) into its part; the last CTA of the sequence to finish
// (one atomic ticket; nobody waits) locates the segment holding u_k * S with
// a float-float scan over the segment sums in order, and scans that segment
// in ascending token order, four tokens per thread.
//
// One wave of CTAs and then one CTA per sequence: the kernel is the issue of
// a warp's 32 terms (four warps share a scheduler) and a chain of latencies.
// So the temperature is tested once for all terms, the last index with mass
// is looked for only where rounding asks for it, and the scans take two
// barriers each.  From the release of the kernel to the token, 16
// sequences of V = 152064: 9.0 -> 7.0 us.  Its CTAs have to find room beside two
// CTAs of the statistics kernel, whose rings leave 1.6 KB of the SM's 196 KB
// configuration, 1 KB of it reserved: 3.2 KB of shared memory here cost that
// call 1.7 us.
__device__ void draw_residual(const AccParams &p, int b, int c, int j, RowStat rs, float tau,
                              float u_k) {
  __shared__ ff s_scan[kAccWarps];
  __shared__ ff s_base[kAccWarps];   // of each warp's first thread that holds the target
  __shared__ int s_seg[kAccWarps];
  __shared__ int s_flag, s_owner, s_token;  // s_owner: the first such warp
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int k = p.k, V = p.V, NS = p.C1;
  const bool residual = j < k;
  const float *row = p.logits + ((size_t)b * (k + 1) + j) * V;
  const float *qrow = residual ? p.q + ((size_t)b * k + j) * V : nullptr;
  DrawPart *parts = p.parts + (size_t)b * NS;
  // four consecutive tokens from e (past V: logit -inf and q 0, terms 0)
  auto load4 = [&](int e, float4 &x, float4 &qq) {
    if (p.vec4) {
      x = e < V ? *reinterpret_cast<const float4 *>(row + e)
                : make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
      qq = (e < V && residual) ? __ldcs(reinterpret_cast<const float4 *>(qrow + e))
                               : make_float4(0.f, 0.f, 0.f, 0.f);
    } else {
      x.x = e < V ? row[e] : -INFINITY;
      x.y = e + 1 < V ? row[e + 1] : -INFINITY;
      x.z = e + 2 < V ? row[e + 2] : -INFINITY;
      x.w = e + 3 < V ? row[e + 3] : -INFINITY;
      qq.x = (e < V && residual) ? qrow[e] : 0.f;
      qq.y = (e + 1 < V && residual) ? qrow[e + 1] : 0.f;
      qq.z = (e + 2 < V && residual) ? qrow[e + 2] : 0.f;
      qq.w = (e + 3 < V && residual) ? qrow[e + 3] : 0.f;
    }
  };

  // ---- segment sums of r and p: lane sums of 32 terms added pairwise in
  // fp32, then a float-float warp sum ----
  const int sg = c * kAccWarps + warp;
  float invS;
  if (sg < NS) {
    float4 xv[8], qv[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) load4(sg * kSegTokens + 128 * i + 4 * lane, xv[i], qv[i]);
    invS = ff_div_to_f(1.0f, rs.S);  // while the loads are in flight
    float gr[8], gp[8];
    auto terms = [&](float t) {
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        float rr[4], pz[4];
        draw_terms(xv[i].x, qv[i].x, residual, rs.m, t, invS, rr[0], pz[0]);
        draw_terms(xv[i].y, qv[i].y, residual, rs.m, t, invS, rr[1], pz[1]);
        draw_terms(xv[i].z, qv[i].z, residual, rs.m, t, invS, rr[2], pz[2]);
        draw_terms(xv[i].w, qv[i].w, residual, rs.m, t, invS, rr[3], pz[3]);
        gr[i] = sum4(rr[0], rr[1], rr[2], rr[3]);
        gp[i] = sum4(pz[0], pz[1], pz[2], pz[3]);
      }
    };
    if (tau == 1.0f) terms(1.0f);
    else terms(tau);
    const ff Sr = warp_sum_ff(ff_of(__fadd_rn(__fadd_rn(__fadd_rn(gr[0], gr[1]), __fadd_rn(gr[2], gr[3])),
                                              __fadd_rn(__fadd_rn(gr[4], gr[5]), __fadd_rn(gr[6], gr[7])))));
    const ff Sp = warp_sum_ff(ff_of(__fadd_rn(__fadd_rn(__fadd_rn(gp[0], gp[1]), __fadd_rn(gp[2], gp[3])),
                                              __fadd_rn(__fadd_rn(gp[4], gp[5]), __fadd_rn(gp[6], gp[7])))));
    if (lane == 0) parts[sg] = DrawPart{Sr, Sp};
  } else {
    invS = ff_div_to_f(1.0f, rs.S);
  }

  // ---- the last CTA of the sequence draws the token ----
  __syncthreads();  // every part of this CTA is written
  if (tid == 0) {   // release this CTA's parts, acquire the others'
    s_flag = atom_add_acq_rel_gpu(p.draw_tickets + b, 1u) == static_cast<unsigned>(p.C2 - 1);
    s_owner = INT_MAX;
    s_token = INT_MAX;
  }
  __syncthreads();
  if (!s_flag) return;

  // ---- the segment: thread t owns segments [t per, (t + 1) per), one each up
  // to V = 262144 ----
  const int per = (NS + kAccThreads - 1) / kAccThreads, first = tid * per, end = min(NS, first + per);
  auto part = [&](int at) { return __ldcg(reinterpret_cast<const float4 *>(parts + at)); };
  const float4 v0 = first < end ? part(first) : make_float4(0.f, 0.f, 0.f, 0.f);
  bool use_p = false;
  auto mass = [&](int at) {
    const float4 v = at == first ? v0 : part(at);
    return use_p ? ff{v.z, v.w} : ff{v.x, v.y};
  };
  ff sum, ex, next, total;
  auto scan_segments = [&]() {
    sum = ff_of(0.f);
#pragma unroll 1
    for (int at = first; at < end; ++at) sum = ff_add(sum, mass(at));
    ex = block_scan2(sum, s_scan, &total, &next);
  };
  scan_segments();
  if (!ff_pos(total)) {  // residual with no mass (rounding only): the target's row
    use_p = true;
    scan_segments();
  }
  const ff target = ff_mul(total, u_k);
  // u S at or past the total (rounding), or u outside [0, 1): the last token with
  // mass of all
  const bool take_last = !ff_lt(target, total) || ff_lt(target, ff_of(0.f));
  // the thread's first segment whose running sum passes the target (its last
  // one with mass if rounding leaves none), and the sum before it.  The prefixes
  // are rounded one by one and may step back by a rounding behind a segment of
  // next to no mass, so that two threads' intervals hold a target: the first
  // thread owns it.
  auto walk = [&]() {
    ff run = ex;
#pragma unroll 1
    for (int at = first; at < end; ++at) {
      const ff m = mass(at);
      if (!ff_pos(m)) continue;
      s_seg[warp] = at;
      s_base[warp] = run;
      run = ff_add(run, m);
      if (!take_last && ff_lt(target, run)) break;
    }
    atomicMin(&s_owner, warp);
  };
  const bool here = ff_pos(sum) && (take_last || !ff_lt(target, ex));
  const unsigned holders = __ballot_sync(0xffffffffu, !take_last && here && ff_lt(target, next));
  if (holders && lane == __ffs(holders) - 1) walk();
  __syncthreads();
  if (s_owner == INT_MAX) {  // take_last, or rounding put the target between two threads' intervals
    __syncthreads();
    if (here) atomicMax(&s_flag, tid + 1);  // the last thread with mass up to the target; 1 from the ticket
    __syncthreads();
    if (here && s_flag == tid + 1) walk();
    __syncthreads();
  }
  const int owner = s_owner, cc = owner == INT_MAX ? -1 : s_seg[owner];
  int token = -1;
  if (cc >= 0) {  // uniform over the block
    // the segment in ascending token order: thread t owns tokens 4t .. 4t+3
    // (terms recomputed exactly as in the segment sums)
    const int e = cc * kSegTokens + 4 * tid;
    float4 xv, qv;
    load4(e, xv, qv);
    const float xs[4] = {xv.x, xv.y, xv.z, xv.w};
    const float qs[4] = {qv.x, qv.y, qv.z, qv.w};
    float t[4];
    int last = -1;  // the thread's last token with mass
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      float rr, pz;
      draw_terms(xs[u], qs[u], residual, rs.m, tau, invS, rr, pz);
      t[u] = use_p ? pz : rr;
      last = t[u] > 0.f ? e + u : last;
    }
    if (!take_last) {
      ff all;
      ff cum = ff_add(s_base[owner], block_scan2(ff_add(two_sum(t[0], t[1]), two_sum(t[2], t[3])), s_scan, &all));
      int at = INT_MAX;
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        cum = ff_add(cum, ff_of(t[u]));
        if (at == INT_MAX && t[u] > 0.f && ff_lt(target, cum)) at = e + u;
      }
      at = __reduce_min_sync(0xffffffffu, at);
      if (lane == 0 && at != INT_MAX) atomicMin(&s_token, at);
      __syncthreads();
      token = s_token;
    }
    if (take_last || token == INT_MAX) {
      // rounding put the target past the running sum: the last token with mass
      __syncthreads();  // s_token has been read
      if (tid == 0) s_token = -1;
      __syncthreads();
      last = __reduce_max_sync(0xffffffffu, last);
      if (lane == 0) atomicMax(&s_token, last);
      __syncthreads();
      token = s_token;
    }
  }
  if (tid == 0) {
    p.out_tokens[(size_t)b * (k + 1) + j] = token;
    p.draw_tickets[b] = 0u;
    p.seqs[b].j1 = 0;  // every CTA of the sequence has read it
  }
}

__global__ void __launch_bounds__(kAccThreads, 3)
accept_draw_kernel(const __grid_constant__ AccParams p) {
  // The previous kernel (the decision kernel of this call) lets this grid
  // start only after it has itself waited for the kernel before the call, so
  // the call's inputs (temperature, uniforms) are in place already; j and
  // the row statistics are waited for.
  grid_launch_dependents();
  const int c = blockIdx.x, b = blockIdx.y;
  const int k = p.k;
  const float tau = p.tau[b];
  if (!(tau > 0.0f)) {  // greedy sequences are complete with the decisions
    // The kernel after this one waits for this grid alone, and may use the call's
    // buffers only once the decisions are complete: where no sequence draws, one
    // CTA waits for them.  (Not all: waiting CTAs have to find room beside the
    // previous kernel's.  16 sequences of V = 152064, half of them greedy, 31.7 us,
    // with every CTA waiting 33.4.)
    if (b == 0 && c == 0) {
      int sampled = 0;
      for (int i = threadIdx.x; i < p.B; i += kAccThreads) sampled |= p.tau[i] > 0.0f;
      if (!__syncthreads_or(sampled)) grid_dependency_wait();
    }
    return;
  }
  const float u_k = p.u[(size_t)b * (k + 1) + k];
  grid_dependency_wait();  // j and row j's statistics come from the previous kernel
  const int4 sq = __ldcg(reinterpret_cast<const int4 *>(p.seqs + b));
  const int j = sq.x - 1;
  if (j < 0 || j > k) {  // no decision was written in this call (a timed-out statistics pass)
    if (c == 0 && threadIdx.x == 0) set_status(p.status, SF_DEVICE_TIMEOUT);
    return;
  }
  const RowStat rs = {__int_as_float(sq.y), 0, ff{__int_as_float(sq.z), __int_as_float(sq.w)}};
  draw_residual(p, b, c, j, rs, tau, u_k);
}

// --------------------------------------------------------------------------
// Two-kernel acceptance for vocabularies beyond one cluster (V > 16 x 2048).
//
// accept_chunks_kernel streams the (k+1) x V logits of every sequence once.
// The B (k+1) rows are cut into 1024-token segments ("chunks"), numbered row
// by row, and warp g of NW1 owns chunks [g U / NW1, (g+1) U / NW1) of the U
// in all: a few consecutive chunks, at most two or three rows.  Lane l reads
// tokens 128 i + 4 l .. +3 of a chunk (eight 16-byte loads), and the next
// chunk's loads are in flight while the current one is folded into per-lane
// running state (max, first index, float-float sum of exp((x - max)/tau)).
// At the end of each run of chunks of one row the warp combines its lanes
// and writes one run record; the runs of row R are stored in warp order, so
// that run t of the row is the one of warp chunk_owner(R C1) + t.
//
// The warp that writes a row's last run record (a ticket per row) combines
// the row's runs in run order into its final statistics; the warp that
// finalises a sequence's k + 1 rows (a ticket per sequence) takes the k
// decisions.  accept_draw_kernel, grid (C2, B), then draws the token of row
// j for the sampled sequences.
// --------------------------------------------------------------------------

// The 32 tokens of lane `lane` in chunk c of a row: c*1024 + 128 i + 4 lane + t
// (tokens at or past V read as -inf).
__device__ __forceinline__ void load_chunk(const AccParams &p, int row, int c, int lane,
                                           float4 (&x)[8]) {
  const float *rp = p.logits + (size_t)row * p.V;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int e = c * kSegTokens + 128 * i + 4 * lane;
    if (p.vec4) {
      x[i] = e < p.V ? __ldcg(reinterpret_cast<const float4 *>(rp + e))
                     : make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
    } else {
      x[i].x = e < p.V ? __ldcg(rp + e) : -INFINITY;
      x[i].y = e + 1 < p.V ? __ldcg(rp + e + 1) : -INFINITY;
      x[i].z = e + 2 < p.V ? __ldcg(rp + e + 2) : -INFINITY;
      x[i].w = e + 3 < p.V ? __ldcg(rp + e + 3) : -INFINITY;
    }
  }
}

// State of one warp over its current run (consecutive chunks of one row).
// Each lane keeps the max of its own tokens so far, the first index holding
// it and the float-float sum of exp((x - max)/tau) over them; the warp
// combines the lanes once, at the end of the run.
struct RunState {
  int row, c, len;
  int g0, n_runs;    // the row's first warp and its number of runs
  float tau, scale;  // scale = log2(e) / tau, rounded once
  bool greedy;
  float lm;          // lane max
  int li;            // its first index
  ff lS;             // lane sum, relative to lm
};

__device__ __forceinline__ void run_begin(const AccParams &p, RunState &st, int row, int c, int U) {
  st.row = row;
  st.c = c;
  st.len = 0;
  st.g0 = chunk_owner(row * p.C1, U, p.NW1);
  st.n_runs = chunk_owner(row * p.C1 + p.C1 - 1, U, p.NW1) - st.g0 + 1;
  st.tau = p.tau[row / (p.k + 1)];
  st.greedy = !(st.tau > 0.0f);
  st.scale = st.greedy ? 0.f : __fdiv_rn(1.44269504088896341f, st.tau);
  st.lm = -INFINITY;
  st.li = INT_MAX;
  st.lS = ff_of(0.f);
}

// Folds chunk st.c (its tokens in x) into the lane state.
__device__ __forceinline__ void run_chunk(RunState &st, int lane, const float4 (&x)[8]) {
  float cm = -INFINITY;
#pragma unroll
  for (int i = 0; i < 8; ++i) cm = fmaxf(cm, fmaxf(fmaxf(x[i].x, x[i].y), fmaxf(x[i].z, x[i].w)));
  if (st.len == 0 || cm > st.lm) {
    // new lane max (or the run's first chunk): its first index in this chunk,
    // and the sum so far moved to the new reference
    int fi = INT_MAX;
#pragma unroll
    for (int i = 7; i >= 0; --i) {  // descending, so the first match wins
      const int e = st.c * kSegTokens + 128 * i + 4 * lane;
      fi = x[i].w == cm ? e + 3 : fi;
      fi = x[i].z == cm ? e + 2 : fi;
      fi = x[i].y == cm ? e + 1 : fi;
      fi = x[i].x == cm ? e : fi;
    }
    if (ff_pos(st.lS)) st.lS = ff_mul(st.lS, exp_diff_accurate(st.lm, cm, st.tau));
    st.lm = cm;
    st.li = fi;
  }
  if (!st.greedy && st.lm != -INFINITY) {
    // 2^((x - lm) log2(e)/tau): the difference and the product each rounded
    // once per token (a term's relative error grows with |x - lm| x 1e-7
    // with no common bias), 2^ by the hardware approximation; the 32 terms
    // are added pairwise in fp32 before one float-float add
    float t[8];
#pragma unroll
    for (int i = 0; i < 8; ++i)
      t[i] = sum4(ex2_approx(__fmul_rn(__fsub_rn(x[i].x, st.lm), st.scale)),
                  ex2_approx(__fmul_rn(__fsub_rn(x[i].y, st.lm), st.scale)),
                  ex2_approx(__fmul_rn(__fsub_rn(x[i].z, st.lm), st.scale)),
                  ex2_approx(__fmul_rn(__fsub_rn(x[i].w, st.lm), st.scale)));
    st.lS = ff_add(st.lS, ff_of(__fadd_rn(__fadd_rn(__fadd_rn(t[0], t[1]), __fadd_rn(t[2], t[3])),
                                          __fadd_rn(__fadd_rn(t[4], t[5]), __fadd_rn(t[6], t[7])))));
  }
  ++st.len;
}

// The decisions of sequence b by one warp, from the final row statistics in
// global memory and the drafts' entries; leaves j and row j's statistics to
// the draw kernel.
__device__ __forceinline__ void decide_warp(const AccParams &p, int b, float tau, const DraftEntry &e) {
  const int lane = threadIdx.x & 31, k = p.k;
  float rm = 0.f;
  int rarg = -1;
  ff rS = ff_of(0.f);
  if (lane <= k) {
    const float4 v = __ldcg(reinterpret_cast<const float4 *>(p.rows + (size_t)b * (k + 1) + lane));
    rm = v.x;
    rarg = __float_as_int(v.y);
    rS = ff{v.z, v.w};
  }
  const Decision d = decide_core(p, b, tau, rm, rarg, rS, e.tok, e.u, e.lx, e.qx, true);
  if (lane == 0 && tau > 0.0f) p.seqs[b] = SeqState{d.j + 1, d.m, d.S};
}

// A run record whose row ticket is taken: the row, its number of runs and
// (lane 0) the ticket's value before this warp's add.
struct PendingTicket {
  int row;
  int n_runs;       // runs of the row
  float tau;        // its temperature
  uint32_t ticket;  // lane 0: the row ticket before this warp's add
};

// Ends the warp's run: combines the lanes, writes the run's record and
// takes the row's ticket (lane 0; one atomic per run; nobody waits).
__device__ __forceinline__ PendingTicket run_end(const AccParams &p, const RunState &st, int lane,
                                                 int gw) {
  float wm = st.lm;
  int wi = st.li;
  warp_argmax(wm, wi);
  ff S = ff_of(0.f);
  if (!st.greedy && wm != -INFINITY) {
    ff mine = ff_of(0.f);
    if (ff_pos(st.lS)) mine = ff_mul(st.lS, exp_diff_accurate(st.lm, wm, st.tau));
    S = warp_sum_ff(mine);
  }
  PendingTicket pt{st.row, st.n_runs, st.tau, 0u};
  if (lane == 0) {
    p.runs[(size_t)st.row * p.C1 + (gw - st.g0)] = RowStat{wm, wi, S};  // run gw - g0 of its row
    // the release covers the record; the acquire, the other runs' records
    pt.ticket = atom_add_acq_rel_gpu(p.row_tickets + pt.row, 1u);
  }
  return pt;
}

// Looks at a taken row ticket: the warp that wrote the row's last record
// combines the row's runs in run order into its final statistics, and the
// warp that finalises a sequence's k + 1 rows takes its decisions.
__device__ __forceinline__ void resolve_ticket(const AccParams &p, const PendingTicket &pt, int lane) {
  const bool last = __shfl_sync(0xffffffffu, pt.ticket == static_cast<uint32_t>(pt.n_runs - 1), 0);
  if (!last) return;
  __syncwarp();
  const int b = pt.row / (p.k + 1);
  const DraftEntry e = load_draft(p, b);  // in flight with the records (used by the last row's warp)
  const RowStat rs = combine_records<4>(reinterpret_cast<const float4 *>(p.runs + (size_t)pt.row * p.C1), pt.n_runs,
                                        pt.tau, !(pt.tau > 0.0f));
  uint32_t last_row = 0;
  if (lane == 0) {
    p.rows[pt.row] = rs;
    p.row_tickets[pt.row] = 0u;  // zero again for the next call
    last_row = atom_add_acq_rel_gpu(p.seq_tickets + b, 1u) == static_cast<uint32_t>(p.k);
  }
  if (!__shfl_sync(0xffffffffu, last_row, 0)) return;
  __syncwarp();
  decide_warp(p, b, pt.tau, e);
  if (lane == 0) p.seq_tickets[b] = 0u;
}

// Chunk ring of the bulk-copy path: kChunkStages 4 KB stages per warp (the
// chunks a warp has requested ahead of the one it reduces) and one mbarrier
// per stage.  Two CTAs per SM keep 192 KB of logits in flight per SM.
constexpr int kChunkStages = 3;
constexpr int kChunkRingBytes = kAccWarps * kChunkStages * kSegTokens * 4;
constexpr int kChunkSmemBytes = kChunkRingBytes + kAccWarps * kChunkStages * 8;

// kBulk (rows 16-byte aligned, V % 4 == 0): each warp's lane 0 requests its
// chunks into the warp's ring with 1-D bulk copies, kChunkStages ahead, and
// the warp reduces them from shared memory; otherwise two register buffers
// (chunk u + 1 loads while chunk u is reduced).
template <bool kBulk>
__global__ void __launch_bounds__(kAccThreads, 2)
accept_chunks_kernel(const __grid_constant__ AccParams p) {
  extern __shared__ __align__(128) uint8_t s_ring[];
  // Every input may come from the previous kernel on the stream: wait for
  // it before reading anything, and only then let the finishing kernel be
  // scheduled (so that it too starts after that kernel completed).
  grid_dependency_wait();
  grid_launch_dependents();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int gw = blockIdx.x * kAccWarps + warp;
  const int CPR = p.C1;
  const int U = p.B * (p.k + 1) * CPR;  // < 2^31: the host checks V * (k + 1) and B
  const ChunkRange range = chunk_range(gw, U, p.NW1);
  const int u0 = range.u0, u1 = range.u1;
  if (u0 >= u1) return;  // a warp that fills up the last CTA
  RunState st;
  run_begin(p, st, u0 / CPR, u0 % CPR, U);
  // the next chunk: the row boundary ends the run and looks at its ticket
  auto advance = [&](int u) {
    int nrow = st.row, nc = st.c + 1;
    if (nc == CPR) { nc = 0; ++nrow; }
    if (nc == 0 || u + 1 == u1) {
      const PendingTicket now = run_end(p, st, lane, gw);
      resolve_ticket(p, now, lane);
      if (u + 1 < u1) run_begin(p, st, nrow, 0, U);
    } else {
      st.c = nc;
    }
  };
  if constexpr (kBulk) {
    const float4 *ring = reinterpret_cast<const float4 *>(s_ring + warp * kChunkStages * kSegTokens * 4);
    const uint32_t ring_s = smem_addr(ring);
    const uint32_t bar0 = smem_addr(s_ring + kChunkRingBytes) + static_cast<uint32_t>(warp * kChunkStages * 8);
    if (lane == 0) {
#pragma unroll 1
      for (int s = 0; s < kChunkStages; ++s) mbar_init(bar0 + 8u * s, 1);
      fence_mbar_init();
    }
    __syncwarp();
    // lane 0: chunk u (row u / CPR, tokens from (u % CPR) * 1024) into stage s
    auto request = [&](int u, int s) {
      const int row = u / CPR, c = u - row * CPR;
      const int n = min(kSegTokens, p.V - c * kSegTokens);
      const uint32_t bytes = static_cast<uint32_t>(n) * 4u;
      mbar_arrive_expect_tx(bar0 + 8u * s, bytes);
      bulk_copy_g2s(ring_s + static_cast<uint32_t>(s * kSegTokens * 4),
                    p.logits + (size_t)row * p.V + (size_t)c * kSegTokens, bytes, bar0 + 8u * s);
    };
    if (lane == 0) {
#pragma unroll 1
      for (int s = 0; s < kChunkStages && u0 + s < u1; ++s) request(u0 + s, s);
    }
    int issued = min(kChunkStages, u1 - u0);
#pragma unroll 1
    for (int u = u0; u < u1; ++u) {
      const int i = u - u0, s = i % kChunkStages;
      const bool ok = mbar_wait_bounded(bar0 + 8u * s, static_cast<uint32_t>(i / kChunkStages) & 1u);
      if (!__all_sync(0xffffffffu, ok)) {
        // a copy never completed (not expected): flag it, wait (bounded)
        // for the other requested stages, and stop this warp
        if (lane == 0) {
          set_status(p.status, SF_DEVICE_TIMEOUT);
#pragma unroll 1
          for (int x = i + 1; x < issued; ++x)
            (void)mbar_wait_bounded(bar0 + 8u * (x % kChunkStages), static_cast<uint32_t>(x / kChunkStages) & 1u);
        }
        return;
      }
      float4 x[8];
#pragma unroll
      for (int t = 0; t < 8; ++t) x[t] = ring[s * (kSegTokens / 4) + 32 * t + lane];
      if ((st.c + 1) * kSegTokens > p.V) {
        // the row's last chunk: tokens at or past V were not copied
#pragma unroll
        for (int t = 0; t < 8; ++t) {
          const int e = st.c * kSegTokens + 128 * t + 4 * lane;
          if (e >= p.V) x[t].x = -INFINITY;
          if (e + 1 >= p.V) x[t].y = -INFINITY;
          if (e + 2 >= p.V) x[t].z = -INFINITY;
          if (e + 3 >= p.V) x[t].w = -INFINITY;
        }
      }
      run_chunk(st, lane, x);
      // the stage's reads are complete (their values are consumed): the
      // next request may overwrite it
      __syncwarp();
      if (issued < u1 - u0 && i + kChunkStages == issued) {
        if (lane == 0) {
          fence_proxy_async_smem();
          request(u0 + issued, s);
        }
        ++issued;
      }
      advance(u);
    }
  } else {
    // two register buffers: chunk u + 1 is loading while chunk u is reduced
    float4 xa[8], xb[8];
    load_chunk(p, st.row, st.c, lane, xa);
    auto step = [&](int u, const float4 (&cur)[8], float4 (&nxt)[8]) {
      int nrow = st.row, nc = st.c + 1;
      if (nc == CPR) { nc = 0; ++nrow; }
      if (u + 1 < u1) load_chunk(p, nrow, nc, lane, nxt);
      run_chunk(st, lane, cur);
      advance(u);
    };
    for (int u = u0; u < u1; u += 2) {
      step(u, xa, xb);
      if (u + 1 < u1) step(u + 1, xb, xa);
    }
  }
}

// --------------------------------------------------------------------------
// host side
// --------------------------------------------------------------------------
struct AccPlan {
  int C1, C2;  // segments per row, draw CTAs per row
};

struct AccLayout {
  size_t draw_tickets, row_tickets, seq_tickets, runs, rows, seqs, parts, total;
};

static int plan_accept(int V, AccPlan *plan) {
  plan->C1 = (V + kSegTokens - 1) / kSegTokens;
  plan->C2 = (plan->C1 + kAccWarps - 1) / kAccWarps;
  return SF_OK;
}

static AccLayout acc_layout(int B, int k, const AccPlan &pl) {
  AccLayout l;
  const size_t R = (size_t)B * (k + 1);
  size_t off = 256;
  l.draw_tickets = off; off = round_up(off + 4 * (size_t)B, 256);
  l.row_tickets = off; off = round_up(off + 4 * R, 256);
  l.seq_tickets = off; off = round_up(off + 4 * (size_t)B, 256);
  l.runs = off; off = round_up(off + sizeof(RowStat) * R * pl.C1, 256);
  l.rows = off; off = round_up(off + sizeof(RowStat) * R, 256);
  l.seqs = off; off = round_up(off + sizeof(SeqState) * (size_t)B, 256);
  l.parts = off; off = round_up(off + sizeof(DrawPart) * (size_t)B * pl.C1, 256);
  l.total = off;
  return l;
}

// Cluster size and slice of the single-kernel path: up to 16 CTAs per
// sequence, slices of at most kClusterMaxSlice tokens (a multiple of 4);
// false when V needs more (the two-kernel path spreads those rows over
// many more CTAs).
static bool cluster_plan(int V, int *cs, int *slice) {
  int c = (V + kClusterMaxSlice - 1) / kClusterMaxSlice;
  if (c > kClusterMax) c = kClusterMax;
  if (c < 1) c = 1;
  int sl = (V + c - 1) / c;
  sl = (sl + 3) / 4 * 4;
  if (sl > kClusterMaxSlice) return false;
  *cs = c;
  *slice = sl;
  return true;
}

// The largest dynamic shared memory of a launch: k = 16 rows of a full slice,
// with as many draft rows ahead as fit.
constexpr int kClusterMostSmem = 200 * 1024;
static_assert(kClusterMostSmem >= (SF_MAX_DRAFT + 1) * kClusterMaxSlice * 4, "the rows themselves fit");

using ClusterKernelFn = void (*)(const AccParams, int, int, int, int);

static ClusterKernelFn cluster_kernel(bool exact) {
  return exact ? accept_cluster_kernel<true> : accept_cluster_kernel<false>;
}

// How many clusters of cs CTAs with `smem` bytes of dynamic shared memory each
// are resident at once on the current device (*resident; 0: none can be).  Asked
// of the runtime once per device, size and KB; the kernel's attributes are set
// before the first answer.
static int cluster_resident(int cs, size_t smem, bool exact, int *resident) {
  static std::mutex mu;
  static std::map<std::tuple<int, bool, int, int>, int> known;  // at most 16 x 201 per device and variant
  DeviceInfo dev;
  int st = current_device(&dev);
  if (st != SF_OK) return st;
  const int kb = static_cast<int>((smem + 1023) / 1024);
  std::lock_guard<std::mutex> lock(mu);
  const auto key = std::make_tuple(dev.ordinal, exact, cs, kb);
  const auto it = known.find(key);
  if (it != known.end()) {
    *resident = it->second;
    return SF_OK;
  }
  const ClusterKernelFn fn = cluster_kernel(exact);
  cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kClusterMostSmem);
  if (e != cudaSuccess)
    return fail(SF_ERR_CUDA, "cudaFuncSetAttribute (accept cluster): %s", cudaGetErrorString(e));
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = cs;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(cs, 1);
  cfg.blockDim = dim3(kAccThreads);
  cfg.dynamicSmemBytes = static_cast<size_t>(kb) * 1024;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  int n = 0;
  e = cudaOccupancyMaxActiveClusters(&n, fn, &cfg);
  if (e != cudaSuccess) {  // not usable: clear the error
    (void)cudaGetLastError();
    n = 0;
  }
  known[key] = n;
  *resident = n;
  return SF_OK;
}

// Whether a cluster of cs CTAs can be resident with the most shared memory that a
// launch asks for (*ok false: use the two-kernel path).
static int cluster_setup(int cs, bool exact, bool *ok) {
  int n = 0;
  const int st = cluster_resident(cs, kClusterMostSmem, exact, &n);
  *ok = st == SF_OK && n > 0;
  return st;
}

// Raises the bulk-copy chunk kernel's dynamic shared memory limit once per
// device.
static int chunks_setup(int device) {
  static std::mutex mu;
  static bool done[64] = {};
  if (device < 0 || device >= 64) return fail(SF_ERR_UNSUPPORTED, "device ordinal %d", device);
  std::lock_guard<std::mutex> lock(mu);
  if (!done[device]) {
    const cudaError_t e = cudaFuncSetAttribute(accept_chunks_kernel<true>,
                                               cudaFuncAttributeMaxDynamicSharedMemorySize, kChunkSmemBytes);
    if (e != cudaSuccess)
      return fail(SF_ERR_CUDA, "cudaFuncSetAttribute (accept chunks): %s", cudaGetErrorString(e));
    done[device] = true;
  }
  return SF_OK;
}

// How the rows of a launch of clusters of cs CTAs lie in shared memory: *bufs of
// them at a time, and whether the draft rows follow (*ahead: fetched ahead of the
// decisions).
// Every row, and then the draft rows, as long as the batch's clusters are all
// resident so; else kClusterFewBufs rows at a time: more clusters per SM are worth
// a second round of copies (B = 16, k = 8, V = 32000: 33 us with all nine rows, 26
// with five; draft rows ahead in two waves of clusters: B = 8, k = 8, V = 32000
// 27.2 us, without them 16.7).
static int cluster_rows(int B, int k, int V, int cs, int slice, bool vec4, bool exact, int *bufs, bool *ahead) {
  int n = 0;
  int st = cluster_resident(cs, cluster_smem(k, slice, k + 1, false), exact, &n);
  if (st != SF_OK) return st;
  *bufs = B <= n || k + 1 < kClusterFewBufs ? k + 1 : kClusterFewBufs;
  const size_t both = cluster_smem(k, slice, k + 1, true);
  *ahead = vec4 && *bufs == k + 1 && 4LL * B * k * V <= kAheadBytes && both <= static_cast<size_t>(kClusterMostSmem);
  if (!*ahead) return SF_OK;
  st = cluster_resident(cs, both, exact, &n);
  *ahead = B <= n;
  return st;
}

static int check_accept_shapes(int B, int k, int V) {
  if (B < 1 || B > SF_MAX_BATCH) return fail(SF_ERR_INVALID_ARG, "B=%d outside [1, %d]", B, SF_MAX_BATCH);
  if (k < 1 || k > SF_MAX_DRAFT) return fail(SF_ERR_INVALID_ARG, "k=%d outside [1, %d]", k, SF_MAX_DRAFT);
  if (V < 2 || (long long)V * (k + 1) >= (1LL << 31))
    return fail(SF_ERR_INVALID_ARG, "V=%d outside [2, 2^31/(k+1))", V);
  return SF_OK;
}

// sf_accept; exact_sums: see accept_cluster_kernel (the two-kernel path has none).
static int launch_accept(const float *target_logits, const float *draft_probs, const int32_t *draft_tokens,
                         const float *uniforms, const float *temperature, int B, int k, int V, int32_t *num_accepted,
                         int32_t *out_tokens, float *accept_ratio, void *workspace, size_t workspace_bytes,
                         bool exact_sums, cudaStream_t stream) {
  int st = check_accept_shapes(B, k, V);
  if (st != SF_OK) return st;
  if (!target_logits || !draft_probs || !draft_tokens || !uniforms || !temperature ||
      !num_accepted || !out_tokens)
    return fail(SF_ERR_INVALID_ARG, "a required pointer is NULL");
  if (!aligned(target_logits, 4) || !aligned(draft_probs, 4) || !aligned(draft_tokens, 4) ||
      !aligned(uniforms, 4) || !aligned(temperature, 4) || !aligned(num_accepted, 4) ||
      !aligned(out_tokens, 4) || (accept_ratio && !aligned(accept_ratio, 4)))
    return fail(SF_ERR_INVALID_ARG, "buffers must be 4-byte aligned");
  if (!workspace || !aligned(workspace, 256))
    return fail(SF_ERR_WORKSPACE, "workspace must be non-NULL and 256-byte aligned");
  AccPlan plan;
  st = plan_accept(V, &plan);
  if (st != SF_OK) return st;
  const AccLayout lay = acc_layout(B, k, plan);
  if (workspace_bytes < lay.total)
    return fail(SF_ERR_WORKSPACE, "workspace has %zu bytes, needs %zu", workspace_bytes, lay.total);

  uint8_t *ws = static_cast<uint8_t *>(workspace);
  AccParams prm;
  prm.logits = target_logits;
  prm.q = draft_probs;
  prm.tokens = draft_tokens;
  prm.u = uniforms;
  prm.tau = temperature;
  prm.num_accepted = num_accepted;
  prm.out_tokens = out_tokens;
  prm.ratio = accept_ratio;
  prm.status = reinterpret_cast<uint32_t *>(ws);
  prm.draw_tickets = reinterpret_cast<uint32_t *>(ws + lay.draw_tickets);
  prm.row_tickets = reinterpret_cast<uint32_t *>(ws + lay.row_tickets);
  prm.seq_tickets = reinterpret_cast<uint32_t *>(ws + lay.seq_tickets);
  prm.runs = reinterpret_cast<RowStat *>(ws + lay.runs);
  prm.rows = reinterpret_cast<RowStat *>(ws + lay.rows);
  prm.seqs = reinterpret_cast<SeqState *>(ws + lay.seqs);
  prm.parts = reinterpret_cast<DrawPart *>(ws + lay.parts);
  prm.B = B;
  prm.k = k;
  prm.V = V;
  prm.C1 = plan.C1;
  prm.C2 = plan.C2;
  prm.NW1 = 0;
  prm.vec4 = (V % 4 == 0) && aligned(target_logits, 16) && aligned(draft_probs, 16);

  // One cluster per sequence when a row fits 16 slices: a single launch
  int cs = 0, slice = 0;
  bool cluster_ok = false;
  if (cluster_plan(V, &cs, &slice)) {
    st = cluster_setup(cs, exact_sums, &cluster_ok);
    if (st != SF_OK) return st;
  }
  if (cluster_ok) {
    cudaLaunchAttribute cattr[2];
    cattr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    cattr[0].val.programmaticStreamSerializationAllowed = 1;
    cattr[1].id = cudaLaunchAttributeClusterDimension;
    cattr[1].val.clusterDim.x = cs;
    cattr[1].val.clusterDim.y = 1;
    cattr[1].val.clusterDim.z = 1;
    cudaLaunchConfig_t ccfg = {};
    ccfg.gridDim = dim3(cs, B);
    ccfg.blockDim = dim3(kAccThreads);
    int bufs = 0;
    bool ahead = false;
    st = cluster_rows(B, k, V, cs, slice, prm.vec4 != 0, exact_sums, &bufs, &ahead);
    if (st != SF_OK) return st;
    ccfg.dynamicSmemBytes = cluster_smem(k, slice, bufs, ahead);
    ccfg.stream = stream;
    ccfg.attrs = cattr;
    ccfg.numAttrs = 2;
    cudaError_t ce = cudaLaunchKernelEx(&ccfg, cluster_kernel(exact_sums), prm, cs, slice, bufs, ahead ? 1 : 0);
    if (ce != cudaSuccess) return fail(SF_ERR_CUDA, "accept cluster launch: %s", cudaGetErrorString(ce));
    return SF_OK;
  }

  // Both kernels are launched with programmatic stream serialisation: each
  // may be scheduled while the previous kernel on the stream drains and
  // waits for it (griddepcontrol.wait) before writing or reading its results.
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  DeviceInfo dev;
  st = current_device(&dev);
  if (st != SF_OK) return st;
  // at most two CTAs per SM
  prm.NW1 = chunk_warps((long long)B * (k + 1) * plan.C1, 2LL * dev.sm_count * kAccWarps);
  const int ctas = (prm.NW1 + kAccWarps - 1) / kAccWarps;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>(ctas));
  cfg.blockDim = dim3(kAccThreads);
  cfg.dynamicSmemBytes = prm.vec4 ? kChunkSmemBytes : 0;
  cfg.stream = stream;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if (prm.vec4) {
    st = chunks_setup(dev.ordinal);
    if (st != SF_OK) return st;
  }
  cudaError_t e = prm.vec4 ? cudaLaunchKernelEx(&cfg, accept_chunks_kernel<true>, prm)
                           : cudaLaunchKernelEx(&cfg, accept_chunks_kernel<false>, prm);
  if (e != cudaSuccess) return fail(SF_ERR_CUDA, "accept chunks launch: %s", cudaGetErrorString(e));
  cfg.gridDim = dim3(plan.C2, B);
  cfg.dynamicSmemBytes = 0;
  e = cudaLaunchKernelEx(&cfg, accept_draw_kernel, prm);
  if (e != cudaSuccess) return fail(SF_ERR_CUDA, "accept draw launch: %s", cudaGetErrorString(e));
  return SF_OK;
}

}  // namespace sf

extern "C" {

size_t sf_accept_workspace_size(int B, int k, int V) {
  if (sf::check_accept_shapes(B, k, V) != SF_OK) return 0;
  sf::AccPlan plan;
  if (sf::plan_accept(V, &plan) != SF_OK) return 0;
  return sf::acc_layout(B, k, plan).total;
}

int sf_accept_kernel_launches(int B, int k, int V) {
  using namespace sf;
  if (check_accept_shapes(B, k, V) != SF_OK) return 0;
  int cs = 0, slice = 0;
  bool cluster_ok = false;
  if (cluster_plan(V, &cs, &slice) && cluster_setup(cs, false, &cluster_ok) != SF_OK) return 0;
  return cluster_ok ? 1 : 2;
}

int sf_accept(const float *target_logits, const float *draft_probs,
              const int32_t *draft_tokens, const float *uniforms, const float *temperature,
              int B, int k, int V, int32_t *num_accepted, int32_t *out_tokens,
              float *accept_ratio, void *workspace, size_t workspace_bytes,
              cudaStream_t stream) {
  using namespace sf;
  clear_error();
  return launch_accept(target_logits, draft_probs, draft_tokens, uniforms, temperature, B, k, V, num_accepted,
                       out_tokens, accept_ratio, workspace, workspace_bytes, false, stream);
}

size_t sf_verify_lm_head_accept_workspace_size(int B, int k, int V) {
  using namespace sf;
  if (check_accept_shapes(B, k, V) != SF_OK || B * (k + 1) > SF_MAX_DRAFT_ROWS) return 0;
  AccPlan plan;
  if (plan_accept(V, &plan) != SF_OK) return 0;
  DeviceInfo dev;
  if (current_device(&dev) != SF_OK) return 0;
  const size_t G = static_cast<size_t>(projection_groups(V, dev.sm_count));
  return acc_layout(B, k, plan).total + round_up(sizeof(SampStat) * B * (k + 1) * G, 256);
}

int sf_verify_lm_head_accept(const void *hidden, const void *weight, const float *draft_probs,
                             const int32_t *draft_tokens, const float *uniforms,
                             const float *temperature, int B, int k, int V, int d, float *logits,
                             int32_t *num_accepted, int32_t *out_tokens, float *accept_ratio,
                             void *workspace, size_t workspace_bytes, cudaStream_t stream) {
  using namespace sf;
  clear_error();
  int st = check_accept_shapes(B, k, V);
  if (st != SF_OK) return st;
  if (B * (k + 1) > SF_MAX_DRAFT_ROWS)
    return fail(SF_ERR_INVALID_ARG, "B*(k+1)=%d above %d rows", B * (k + 1), SF_MAX_DRAFT_ROWS);
  if (!draft_probs || !draft_tokens || !uniforms || !temperature || !num_accepted || !out_tokens)
    return fail(SF_ERR_INVALID_ARG, "a required pointer is NULL");
  if (!aligned(draft_probs, 4) || !aligned(draft_tokens, 4) || !aligned(uniforms, 4) ||
      !aligned(temperature, 4) || !aligned(num_accepted, 4) || !aligned(out_tokens, 4) ||
      (accept_ratio && !aligned(accept_ratio, 4)))
    return fail(SF_ERR_INVALID_ARG, "buffers must be 4-byte aligned");
  if (!workspace || !aligned(workspace, 256))
    return fail(SF_ERR_WORKSPACE, "workspace must be non-NULL and 256-byte aligned");
  AccPlan plan;
  st = plan_accept(V, &plan);
  if (st != SF_OK) return st;
  DeviceInfo dev;
  st = current_device(&dev);
  if (st != SF_OK) return st;
  const AccLayout lay = acc_layout(B, k, plan);
  const int R = B * (k + 1);
  const size_t G = static_cast<size_t>(projection_groups(V, dev.sm_count));
  const size_t need = lay.total + round_up(sizeof(SampStat) * R * G, 256);
  if (workspace_bytes < need)
    return fail(SF_ERR_WORKSPACE, "workspace has %zu bytes, needs %zu", workspace_bytes, need);

  uint8_t *ws = static_cast<uint8_t *>(workspace);
  const bool vec4 = (V % 4 == 0) && aligned(logits, 16) && aligned(draft_probs, 16);
  int Gl = 0;
  // Where sf_accept is one cluster launch with the draft rows fetched ahead, the
  // projection can write the logits alone and the cluster sums the rows at the
  // statistics' precision, in place of the statistics, the decisions and the
  // draw.  A cluster takes its rows one after another, 0.7-1.1 us each; the
  // statistics cost more with every 16 rows and at temperatures other than 1.  So
  // one draft, many sequences or few rows go to the cluster, long rows of more
  // sequences than clusters run at a time don't.  Whole calls (us at
  // temperature 1 and 0.7, statistics -> cluster), on its side of each line:
  //   k = 1, B = 4        V = 2000 15.6 -> 15.0, 20.5 -> 17.2; 32000 25.1 -> 23.8, 29.9 -> 26.7
  //   k = 8, B = 12       V = 2000 27.2 -> 25.1, 32.2 -> 32.8; 16000 30.4 -> 27.0, 35.9 -> 34.5
  //   k = 3, B = 64       V = 8000 45.8 -> 31.0, 51.2 -> 35.2
  //   k = 3, B = 1        V = 2000 17.2 -> 16.6, 20.6 -> 20.2; 32000 25.1 -> 22.1, 31.2 -> 25.0
  //   k = 2, B = 4        V = 8000 17.8 -> 16.2, 22.4 -> 18.8
  //   k = 5, B = 1        V = 16000 19.6 -> 18.6, 24.5 -> 23.9; 32000 25.2 -> 23.9, 31.1 -> 28.8
  // and beyond it:
  //   k = 1, B = 32       V = 32000 30.3 -> 32.3, 34.6 -> 36.3
  //   k = 16, B = 12      V = 8000 39.3 -> 39.1, 44.7 -> 45.8
  //   k = 8, B = 8        V = 2000 23.5 -> 24.4, 28.3 -> 32.0; 32000 32.6 -> 32.7, 38.6 -> 39.0
  //   k = 3, B = 4        V = 2000 16.3 -> 17.3, 19.9 -> 20.8; 32000 25.1 -> 25.8, 29.4 -> 30.0
  //   k = 2, B = 4        V = 16000 19.4 -> 22.0, 24.4 -> 24.2
  //   k = 5, B = 1        V = 8000 18.0 -> 18.6, 21.8 -> 23.3
  //   k = 5, B = 2        V = 2000 15.9 -> 18.5, 20.5 -> 23.9; 32000 25.3 -> 25.9, 30.9 -> 31.4
  // (d = 1024).  Not fetched ahead it is longer (B = 2, k = 16, V = 32000, d = 4096 58.1 ->
  // 61.0 before the finer sums).
  const bool few = (B <= 2 && k <= 3) || (k == 2 && V <= 8192) || (B == 1 && k <= 5 && V > 12288);
  const bool many = (k == 1 || (k <= 8 && B >= 12)) && (V <= 16384 || B <= 16);
  int cs = 0, slice = 0, bufs = 0;
  bool cluster_ok = false, ahead = false;
  if ((few || many) && cluster_plan(V, &cs, &slice)) {
    st = cluster_setup(cs, true, &cluster_ok);
    if (st == SF_OK && cluster_ok) st = cluster_rows(B, k, V, cs, slice, vec4, true, &bufs, &ahead);
    if (st != SF_OK) return st;
  }
  if (cluster_ok && ahead) {
    st = launch_projection_stats(hidden, weight, R, d, V, logits, temperature, k + 1, nullptr,
                                 reinterpret_cast<uint32_t *>(ws), &Gl, stream);
    if (st != SF_OK) return st;
    return launch_accept(logits, draft_probs, draft_tokens, uniforms, temperature, B, k, V, num_accepted, out_tokens,
                         accept_ratio, workspace, workspace_bytes, true, stream);
  }
  SampStat *stats = reinterpret_cast<SampStat *>(ws + lay.total);
  // target logits and their per-CTA row statistics; row b*(k+1)+i uses tau_b
  st = launch_projection_stats(hidden, weight, R, d, V, logits, temperature, k + 1, stats,
                               reinterpret_cast<uint32_t *>(ws), &Gl, stream);
  if (st != SF_OK) return st;

  AccParams prm;
  prm.logits = logits;
  prm.q = draft_probs;
  prm.tokens = draft_tokens;
  prm.u = uniforms;
  prm.tau = temperature;
  prm.num_accepted = num_accepted;
  prm.out_tokens = out_tokens;
  prm.ratio = accept_ratio;
  prm.status = reinterpret_cast<uint32_t *>(ws);
  prm.row_tickets = reinterpret_cast<uint32_t *>(ws + lay.row_tickets);
  prm.seq_tickets = reinterpret_cast<uint32_t *>(ws + lay.seq_tickets);
  prm.draw_tickets = reinterpret_cast<uint32_t *>(ws + lay.draw_tickets);
  prm.runs = reinterpret_cast<RowStat *>(ws + lay.runs);
  prm.rows = reinterpret_cast<RowStat *>(ws + lay.rows);
  prm.seqs = reinterpret_cast<SeqState *>(ws + lay.seqs);
  prm.parts = reinterpret_cast<DrawPart *>(ws + lay.parts);
  prm.B = B;
  prm.k = k;
  prm.V = V;
  prm.C1 = plan.C1;
  prm.C2 = plan.C2;
  prm.NW1 = 0;
  prm.vec4 = vec4;

  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(B);
  cfg.blockDim = dim3(32 * (k + 1));
  cfg.stream = stream;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  cudaError_t e = cudaLaunchKernelEx(&cfg, accept_decide_kernel, prm,
                                     static_cast<const SampStat *>(stats), Gl);
  if (e != cudaSuccess) return fail(SF_ERR_CUDA, "accept decide launch: %s", cudaGetErrorString(e));
  cfg.gridDim = dim3(plan.C2, B);
  cfg.blockDim = dim3(kAccThreads);
  e = cudaLaunchKernelEx(&cfg, accept_draw_kernel, prm);
  if (e != cudaSuccess) return fail(SF_ERR_CUDA, "accept draw launch: %s", cudaGetErrorString(e));
  return SF_OK;
}

}  // extern "C"
