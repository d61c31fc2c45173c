// draft_tail.cu -- the draft-distribution tail of Algorithm 1 on sm_103a.
//
// The semi-autoregressive draft head ends with the frozen LM head (Sec. 3.3,
// Algorithm 1): each of the K draft positions' hidden states is projected to
// vocabulary logits, P'_i = softmax(logits_i / tau) is the draft distribution
// q that the verification rule divides by, and T'_i is drawn from it,
// independently per position.  The draw is an inverse CDF in ascending token
// order (the smallest token x with u_i * S < C(x)); tau <= 0 is greedy (the
// first argmax, a one-hot P').
//
// GB300 design.  The projection streams the whole V x hidden bf16 LM head
// (262 MB for LLaVA's 32000 x 4096, 1.09 GB for QwenVL's 152064 x 3584) for
// a few dozen rows, so it is bound by HBM and everything else hides under
// that stream:
//  * lm_head_kernel: one CTA per SM, each owning an equal contiguous range
//    of vocabulary rows (floor or ceil of V / G), cut into 256-row tiles; a
//    range's last tile is loaded with a box of exactly its remaining height
//    (two extra tensor maps), so every SM streams the same number of weight
//    bytes.  Warp 9 streams 256 x 64 weight boxes and
//    the matching 64-column box of the hidden states (rows padded to NP, a
//    multiple of 16, by the copy's zero fill) into a deep ring; warp 8 issues
//    logits^T = W H^T as tcgen05 MMAs of M = 128 (a half tile of the
//    vocabulary), N = NP (draft rows), K = 16, accumulating in tensor memory,
//    double-buffered per tile where that fits; warps 0-7 (four per half) read
//    a finished tile back (one vocabulary row per lane), store the fp32 logits
//    coalesced along the vocabulary and, for the fused path, reduce each
//    draft row over the tile to (max, first argmax, float-float sum of
//    exp((x - max)/tau)), merged across the CTA's tiles.
//    Tiles of 256 rows, not 128 (but see launch_lm_head): the hidden-state box
//    is re-read from L2 for every tile, and a CTA of V = 32000 (210 rows) has
//    one tile and one exposed epilogue instead of two.  Measured with 128 and 256 rows:
//    5 rows x 32000 x 4096 50.8 -> 39.8 us (6.6 TB/s), 36 x 152064 x 3584
//    171.0 -> 161.7, 128 x 152064 x 3584 195.7 -> 184 us.
//    Weight copies run before griddepcontrol.wait (the weights are constant);
//    the hidden states are copied after it.
//  * sample_stats_kernel (sf_sample only): the same per-chunk statistics
//    from given logits, 2048 tokens per CTA.
//  * sample_finish_kernel: grid (CTAs per row, rows).  Every CTA of a row
//    combines the row's chunk statistics in the same fixed order (so all get
//    bit-identical max, sum and crossing chunk), writes probabilities for its
//    span of tokens, and the CTA whose span holds the crossing chunk's first
//    token scans that chunk in ascending order for the token.
// Arithmetic: per-token terms are fp32 (exp of a float-float argument, see
// ff_math.cuh); sums, prefixes and the crossing test are float-float in a
// fixed order, so results are deterministic.  The chunk sums are taken
// relative to each chunk's own maximum and rescaled by exp((m_c - m)/tau) when
// combined; the scan inside the crossing chunk uses terms relative to the
// row maximum, so the two differ by rounding only, and where rounding puts
// the target past the chunk's own terms the chunk's last positive token is
// taken.
#include <climits>
#include <cmath>
#include <map>
#include <mutex>
#include <tuple>

#include "ff_math.cuh"
#include "sf_device.cuh"
#include "sf_host.h"

namespace sf {

constexpr int kLmThreads = 320;
constexpr int kLmHalf = 128;                           // vocabulary rows per MMA (M), threads per epilogue group
constexpr int kLmEpiThreads = 2 * kLmHalf;             // one group per half tile
constexpr int kLmMmaWarp = 8;
constexpr int kLmProducerWarp = 9;
constexpr int kLmTileV = 2 * kLmHalf;                  // vocabulary rows per tile: two MMAs share a hidden-state box
constexpr int kLmChunkK = 64;                          // hidden columns per ring slot
constexpr int kLmMaxStages = 32;
constexpr int kLmEpiWarps = kLmEpiThreads / 32;
constexpr int kLmColGroup = 16;                        // draft rows per epilogue step
constexpr int kLmTStride = 34;                         // floats per transposed row (2 mod 32 banks)
constexpr int kLmTBufFloats = kLmColGroup * kLmTStride;  // per epilogue warp
constexpr int kSampleUnit = 2048;                      // tokens per statistics chunk (sf_sample)
constexpr int kSampleSpan = 1024;                      // least tokens per finishing CTA (4 per thread)
constexpr int kFinishCtasPerSm = 5;                    // resident finishing CTAs (registers)
constexpr int kMaxStatChunks = 4096;                   // statistics chunks per row

struct LmParams {
  float *logits;     // [R][V]
  const float *tau;  // temperature of row r: tau[r / tau_div]; read only with stats
  SampStat *stats;   // [R][G], or null for the plain projection
  uint32_t *status;
  int R, V, NP;
  int G;             // CTAs; CTA c owns vocabulary rows [c*V/G, (c+1)*V/G)
  int ha, hb;        // box heights of the two last-tile weight maps
  int KC;            // hidden chunks of 64
  int tile;          // vocabulary rows per tile: kLmTileV or kLmHalf
  int halves;        // 128-row halves of a tile in use (1: tiles or ranges of at most 128 rows)
  int nbuf;          // accumulator buffers in tensor memory (2, or 1)
  int stages;
  uint32_t w_bytes;      // weight box of the tallest tile
  uint32_t stage_bytes;  // weight box + NP * 128 bytes of hidden states
  uint32_t tmem_cols;
  uint32_t idesc;
  int w_after_wait;  // copy the weight rows only after griddepcontrol.wait
  int w_keep;        // weight rows are re-read next: L2 evict_last instead of evict_first
  int tau_div;       // rows per temperature entry (1: one per row)
  int ks;            // hidden-dimension splits: CTA (g, s) sums chunks [s*KC/ks, (s+1)*KC/ks)
  long long part_stride;  // floats between the ks partial outputs (split s adds s * part_stride)
};

struct SampleParams {
  const float *logits;    // [R][V]
  SampStat *stats;        // [R][Cn]
  const float *u;         // [R]
  const float *tau;       // [R]
  float *probs;           // [R][V]
  int32_t *tokens;        // [R]
  int R, V;
  int Cn;                 // statistics chunks per row
  int unit, T;            // chunk c covers [e(c), e(c+1)), e(c) = min(V, unit * (c*T/Cn))
  int span;               // tokens per finishing CTA (a multiple of 4)
  int vec4;               // rows 16-byte aligned and V % 4 == 0
};

// ---------------------------------------------------------------------------
// LM-head projection (tcgen05)
// ---------------------------------------------------------------------------
struct LmSmem {
  static size_t bytes(int stages, uint32_t stage_bytes, int NP) {
    // ring | transposed values and running statistics of every epilogue warp |
    // temperatures | barriers | misc.  An MMA reads 128 rows from its half's
    // first row, whatever the box's height: what lies behind the last slot
    // covers the rest of a tile, so that those reads stay inside the allocation.
    const size_t behind = kLmEpiWarps * 4 * kLmTBufFloats +
                          static_cast<size_t>(NP) * (kLmEpiWarps * sizeof(SampStat) + 4) +
                          8 * (2 * stages + 5) + 64;
    const size_t tile = kLmTileV * kLmChunkK * 2;
    return 1024 + static_cast<size_t>(stages) * stage_bytes +
           (behind + stage_bytes > tile ? behind : tile - stage_bytes);
  }
};

// exp((x - m) / tau) for one token; a token at -inf (masked) has weight 0.
__device__ __forceinline__ float term_of(float x, float m, float tau) {
  return x == -INFINITY ? 0.f : exp_diff_accurate(x, m, tau);
}

// Folds one tile's (max, argmax, sum) of a row into the CTA's running
// statistics; tiles arrive in ascending order, so on equal maxima the
// earlier index stays.
__device__ __forceinline__ void stat_merge(SampStat &run, float m, int arg, ff s, float tau,
                                           bool greedy) {
  if (better(m, arg, run.m, run.arg)) {
    if (!greedy)
      run.S = ff_add(run.m == -INFINITY ? run.S : ff_mul(run.S, exp_diff_accurate(run.m, m, tau)), s);
    run.m = m;
    run.arg = arg;
  } else if (!greedy) {
    run.S = ff_add(run.S, ff_mul(s, term_of(m, run.m, tau)));
  }
}

// One epilogue step of a warp: 16 draft rows (TMEM columns from `taddr`) of
// its 32 vocabulary rows vbase .. vbase + 31 (one per lane).  The fp32 logits go
// straight to global memory, coalesced along the vocabulary.  For the
// statistics (wrun: the warp's running statistics of these draft rows) the
// warp transposes the values through its own shared memory tb, so that two
// lanes hold a draft row, 16 values each: the maximum, its first index and the
// float-float sum of their terms as trees, so that a lane's exponentials
// overlap; warps never wait for one another.
__device__ __forceinline__ void lm_epilogue_step(uint32_t taddr, float *logits, int V, int vbase, bool vin,
                                                 int cols_left, float *tb, const float *tau_row,
                                                 SampStat *wrun) {
  const int lane = threadIdx.x & 31;
  uint32_t x[16];
  tmem_ld_32x32b_x16(taddr, x);
  if (vin) {
    float *dst = logits + vbase + lane;
#pragma unroll
    for (int j = 0; j < 16; ++j)
      if (j < cols_left) dst[static_cast<size_t>(j) * V] = __uint_as_float(x[j]);
  }
  if (!wrun) return;
  __syncwarp();  // the previous step's reads are done
#pragma unroll
  for (int j = 0; j < 16; ++j) tb[j * kLmTStride + lane] = vin ? __uint_as_float(x[j]) : -INFINITY;
  __syncwarp();
  const int part = lane & 1, r = lane >> 1;
  const float *col = tb + r * kLmTStride + part;
  float xv[16];
#pragma unroll
  for (int e = 0; e < 16; ++e) xv[e] = col[2 * e];
  float mx[8];
#pragma unroll
  for (int e = 0; e < 8; ++e) mx[e] = fmaxf(xv[e], xv[e + 8]);
#pragma unroll
  for (int w = 4; w >= 1; w >>= 1) {
#pragma unroll
    for (int e = 0; e < w; ++e) mx[e] = fmaxf(mx[e], mx[e + w]);
  }
  float bv = fmaxf(mx[0], -INFINITY);  // NaN values only: -inf
  unsigned hits = 0u;
#pragma unroll
  for (int e = 0; e < 16; ++e) hits |= xv[e] == bv ? 1u << e : 0u;
  int bi = hits ? vbase + part + 2 * (__ffs(hits) - 1) : INT_MAX;  // first index of the maximum
  {
    const float ov = __shfl_xor_sync(0xffffffffu, bv, 1);
    const int oi = __shfl_xor_sync(0xffffffffu, bi, 1);
    if (better(ov, oi, bv, bi)) {
      bv = ov;
      bi = oi;
    }
  }
  const float tau = tau_row[r];
  const bool greedy = !(tau > 0.f);
  ff s = ff_of(0.f);
  if (!greedy) {
    // terms exp((x - bv) / tau), the argument carried to float-float
    const float ref = bv == -INFINITY ? 0.f : bv;  // all masked: every term is 0
    if (tau == 1.f) {  // one branch for all: the divisions are skipped together
#pragma unroll
      for (int e = 0; e < 16; ++e) xv[e] = term_of(xv[e], ref, 1.f);
    } else if (tau >= kRecipTauMin && tau <= kRecipTauMax) {
      const float inv = __fdiv_rn(1.f, tau);
#pragma unroll
      for (int e = 0; e < 16; ++e) xv[e] = exp_diff_recip(xv[e], ref, tau, inv);
    } else {
#pragma unroll
      for (int e = 0; e < 16; ++e) xv[e] = term_of(xv[e], ref, tau);
    }
    ff t[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) t[e] = two_sum(xv[e], xv[e + 8]);
#pragma unroll
    for (int w = 4; w >= 1; w >>= 1) {
#pragma unroll
      for (int e = 0; e < w; ++e) t[e] = ff_add(t[e], t[e + w]);
    }
    s = t[0];
  }
  s = ff_add(s, shfl_xor_ff(s, 1));
  if (part == 0) stat_merge(*(wrun + r), bv, bi, s, tau, greedy);
}

__global__ void __launch_bounds__(kLmThreads, 1)
lm_head_kernel(const __grid_constant__ CUtensorMap tmap_w, const __grid_constant__ CUtensorMap tmap_wa,
               const __grid_constant__ CUtensorMap tmap_wb, const __grid_constant__ CUtensorMap tmap_h,
               const __grid_constant__ LmParams p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t *smem = reinterpret_cast<uint8_t *>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  const int S = p.stages;
  const uint32_t ring = smem_addr(smem);
  float *tbuf = reinterpret_cast<float *>(smem + static_cast<size_t>(S) * p.stage_bytes);
  SampStat *run = reinterpret_cast<SampStat *>(tbuf + kLmEpiWarps * kLmTBufFloats);
  float *s_tau = reinterpret_cast<float *>(run + kLmEpiWarps * p.NP);
  uint64_t *bar_mem = reinterpret_cast<uint64_t *>(s_tau + p.NP);
  int *s_misc = reinterpret_cast<int *>(bar_mem + 2 * S + 5);
  // s_misc: [0] TMEM base, [1] abort word, [2] chunks issued, [3] chunks consumed
  volatile int *s_abort = s_misc + 1;
  const uint32_t bars = smem_addr(bar_mem);
  const int FULL = 0, EMPTY = S, DFULL = 2 * S, DEMPTY = 2 * S + 2, FIN = 2 * S + 4;
  auto bar = [&](int i) -> uint32_t { return bars + 8u * static_cast<uint32_t>(i); };

  const int tid = threadIdx.x, warp = uniform_warp_id(), lane = tid & 31;
  const int grp = static_cast<int>(blockIdx.x) % p.G, split = static_cast<int>(blockIdx.x) / p.G;
  const int v0 = static_cast<int>(static_cast<long long>(grp) * p.V / p.G);
  const int v1 = static_cast<int>(static_cast<long long>(grp + 1) * p.V / p.G);
  const int n_tiles = (v1 - v0 + p.tile - 1) / p.tile;
  const int last_h = v1 - v0 - (n_tiles - 1) * p.tile;  // rows of the last tile
  const int kc0 = split * p.KC / p.ks;                      // this CTA's hidden chunks
  const int nkc = (split + 1) * p.KC / p.ks - kc0;
  float *const logits = p.logits + static_cast<long long>(split) * p.part_stride;
  const uint32_t total = static_cast<uint32_t>(n_tiles) * static_cast<uint32_t>(nkc);
  // weight map and box height of tile i
  auto tile_map = [&](int i, uint32_t &bytes) -> const CUtensorMap * {
    const int h = i == n_tiles - 1 ? last_h : p.tile;
    bytes = static_cast<uint32_t>(h) * (kLmChunkK * 2) + static_cast<uint32_t>(p.NP) * (kLmChunkK * 2);
    return h == p.tile ? &tmap_w : (h == p.ha ? &tmap_wa : &tmap_wb);
  };

  grid_launch_dependents();
  if (tid == 0) {
    for (int s = 0; s < S; ++s) {
      mbar_init(bar(FULL + s), 1);
      mbar_init(bar(EMPTY + s), 1);
    }
    for (int x = 0; x < 2; ++x) {
      mbar_init(bar(DFULL + x), 1);
      mbar_init(bar(DEMPTY + x), static_cast<uint32_t>(p.halves * kLmHalf));
    }
    mbar_init(bar(FIN), 1);
    fence_mbar_init();
    prefetch_tensormap(&tmap_w);
    prefetch_tensormap(&tmap_wa);
    prefetch_tensormap(&tmap_wb);
    prefetch_tensormap(&tmap_h);
    s_misc[1] = 0;
    s_misc[2] = 0;
    s_misc[3] = 0;
  }
  __syncthreads();  // barrier initialisation visible to every role
  // Tensor memory is allocated only once the previous kernel on the stream
  // has completed: a predecessor that is still waiting for its own
  // predecessor may not have allocated yet, and holding TMEM here while it
  // waits for columns could deadlock the pair.  The producer warp does not
  // need TMEM and starts its weight copies meanwhile.
  uint32_t tmem = 0;
  if (warp != kLmProducerWarp) {
    if (warp == kLmMmaWarp) {
      grid_dependency_wait();
      tmem_alloc(smem_addr(s_misc), p.tmem_cols);
      tmem_relinquish_alloc_permit();
      tc_fence_before_sync();
    }
    named_bar_sync(2, kLmEpiThreads + 32);
    tc_fence_after_sync();
    tmem = static_cast<uint32_t>(s_misc[0]);
  }

  if (warp == kLmProducerWarp) {
    // The whole warp runs the loop and an elected lane issues, so that the
    // copies' operands are warp-uniform (see smem_desc_sw128).
    const uint64_t pol_w = p.w_keep ? l2_policy_evict_last() : l2_policy_evict_first();
    const uint64_t pol_h = l2_policy_evict_last();
    const int prime = total < static_cast<uint32_t>(S) ? static_cast<int>(total) : S;
    int i = 0, kc = 0;  // tile and hidden chunk of the next slot
    auto next = [&]() {
      if (++kc == nkc) {
        kc = 0;
        ++i;
      }
    };
    // the first ring fill: weights before the dependency wait (unless
    // they may come from the previous kernel), hidden states after it
    if (p.w_after_wait) grid_dependency_wait();
    for (int q = 0; q < prime; ++q, next()) {
      uint32_t bytes;
      const CUtensorMap *mw = tile_map(i, bytes);
      if (elect_one()) {
        mbar_arrive_expect_tx(bar(FULL + q), bytes);
        tma_load_2d(ring + static_cast<uint32_t>(q) * p.stage_bytes, mw, (kc0 + kc) * kLmChunkK, v0 + i * p.tile,
                    bar(FULL + q), pol_w);
      }
      __syncwarp();
    }
    if (!p.w_after_wait) grid_dependency_wait();
    for (int q = 0, hc = 0; q < prime; ++q) {
      if (elect_one())
        tma_load_2d(ring + static_cast<uint32_t>(q) * p.stage_bytes + p.w_bytes, &tmap_h, (kc0 + hc) * kLmChunkK, 0,
                    bar(FULL + q), pol_h);
      __syncwarp();
      if (++hc == nkc) hc = 0;
    }
    uint32_t q = static_cast<uint32_t>(prime), lap = 0;  // earlier passes over the ring
    int slot = 0;
    for (; q < total; ++q, next()) {
      const bool w = mbar_wait_or_abort(bar(EMPTY + slot), lap & 1u, s_abort);
      if (!__all_sync(0xffffffffu, w)) break;
      const uint32_t dst = ring + static_cast<uint32_t>(slot) * p.stage_bytes;
      uint32_t bytes;
      const CUtensorMap *mw = tile_map(i, bytes);
      if (elect_one()) {
        mbar_arrive_expect_tx(bar(FULL + slot), bytes);
        tma_load_2d(dst, mw, (kc0 + kc) * kLmChunkK, v0 + i * p.tile, bar(FULL + slot), pol_w);
        tma_load_2d(dst + p.w_bytes, &tmap_h, (kc0 + kc) * kLmChunkK, 0, bar(FULL + slot), pol_h);
      }
      __syncwarp();
      if (++slot == S) {
        slot = 0;
        ++lap;
      }
    }
    if (lane == 0) s_misc[2] = static_cast<int>(q);
    __syncwarp();
  } else if (warp == kLmMmaWarp) {
    // ------------------------------------------------------------------
    // MMA issue: per 64-column chunk four K steps (16 columns, +32 bytes along
    // the 128-byte swizzled rows) for each 128-row half of the tile, the halves
    // sharing the hidden-state box; the slot is released by a commit.  Rows
    // beyond a short tile's box hold stale data; their accumulator rows are
    // never stored.
    // ------------------------------------------------------------------
    uint32_t q = 0, lap = 0;
    int slot = 0;
    bool ok = true;
    for (int i = 0; i < n_tiles && ok; ++i) {
      const int buf = i % p.nbuf;
      const int halves = (i == n_tiles - 1 ? last_h : p.tile) > kLmHalf ? 2 : 1;
      if (i >= p.nbuf) {
        int w = 1;
        if (lane == 0) w = mbar_wait_or_abort(bar(DEMPTY + buf), (i / p.nbuf - 1) & 1, s_abort);
        if (!__shfl_sync(0xffffffffu, w, 0)) break;
      }
      tc_fence_after_sync();
      const uint32_t d = tmem + static_cast<uint32_t>(buf * p.halves * p.NP);
      for (int kc = 0; kc < nkc; ++kc, ++q) {
        const bool w = mbar_wait_or_abort(bar(FULL + slot), lap & 1u, s_abort);
        if (!__all_sync(0xffffffffu, w)) {
          ok = false;
          break;
        }
        tc_fence_after_sync();
        if (lane == 0) s_misc[3] = static_cast<int>(q + 1);
        const uint32_t wa = ring + static_cast<uint32_t>(slot) * p.stage_bytes;
        const uint64_t a0 = smem_desc_sw128(wa, 16, 1024), b0 = smem_desc_sw128(wa + p.w_bytes, 16, 1024);
        const uint32_t acc = kc > 0 ? 1u : 0u;
        if (elect_one()) {
#pragma unroll
          for (int kk = 0; kk < kLmChunkK / 16; ++kk) tc_mma_ss(d, a0 + 2 * kk, b0 + 2 * kk, p.idesc, kk > 0 ? 1u : acc);
          if (halves > 1) {
#pragma unroll
            for (int kk = 0; kk < kLmChunkK / 16; ++kk)
              tc_mma_ss(d + static_cast<uint32_t>(p.NP), a0 + (kLmHalf * kLmChunkK * 2 >> 4) + 2 * kk, b0 + 2 * kk,
                        p.idesc, kk > 0 ? 1u : acc);
          }
          tc_commit(bar(EMPTY + slot));
        }
        __syncwarp();
        if (++slot == S) {
          slot = 0;
          ++lap;
        }
      }
      if (!ok) break;
      if (elect_one()) tc_commit(bar(DFULL + buf));
      __syncwarp();
    }
    if (elect_one()) tc_commit(bar(FIN));
    __syncwarp();
    (void)mbar_wait_bounded(bar(FIN), 0);
  } else {
    // ------------------------------------------------------------------
    // epilogue: warps 0-3 take the tile's first 128 vocabulary rows, warps
    // 4-7 the others; 16 draft rows per step.  The last tile's epilogue is
    // exposed: at 128 draft rows the statistics added 30 us with a 128-thread
    // transpose and chains of float-float adds on four warps.
    // ------------------------------------------------------------------
    const bool stats = p.stats != nullptr;
    const int hf = warp >> 2;  // half of the tile
    grid_dependency_wait();    // outputs and temperatures follow the previous kernel
    if (stats) {
      for (int c = tid; c < p.NP; c += kLmEpiThreads) s_tau[c] = c < p.R ? p.tau[c / p.tau_div] : 1.f;
      for (int c = tid; c < kLmEpiWarps * p.NP; c += kLmEpiThreads) run[c] = SampStat{-INFINITY, INT_MAX, ff_of(0.f)};
      named_bar_sync(1, kLmEpiThreads);
    }
    const uint32_t lane_base = tmem + (static_cast<uint32_t>(32 * (warp & 3)) << 16);
    float *tb = tbuf + warp * kLmTBufFloats;
    SampStat *wrun = stats ? run + warp * p.NP : nullptr;
    for (int i = 0; i < n_tiles && hf < p.halves; ++i) {
      const int buf = i % p.nbuf;
      const bool ok = mbar_wait_or_abort(bar(DFULL + buf), (i / p.nbuf) & 1, s_abort);
      if (!__all_sync(0xffffffffu, ok)) break;
      tc_fence_after_sync();
      const int vbase = v0 + i * p.tile + 32 * warp;  // the warp's vocabulary rows
      const bool vin = vbase + lane < v1;
      const uint32_t acc = lane_base + static_cast<uint32_t>((buf * p.halves + hf) * p.NP);
#pragma unroll 1
      for (int c0 = 0; c0 < p.NP && vbase < v1; c0 += kLmColGroup)
        lm_epilogue_step(acc + static_cast<uint32_t>(c0), logits + static_cast<size_t>(c0) * p.V, p.V, vbase, vin,
                         p.R - c0, tb, s_tau + c0, stats ? wrun + c0 : nullptr);
      tc_fence_before_sync();
      mbar_arrive(bar(DEMPTY + buf));
    }
    if (stats) {
      named_bar_sync(1, kLmEpiThreads);
      // the eight warps' statistics of a draft row, a lane for each: rescaled at
      // once, by float-float factors (a warp's 32 rows are few of a chunk, and the
      // errors of as many plain factors showed in the probabilities), and summed
      // as a tree
      for (int i0 = 32 * warp; i0 < kLmEpiWarps * p.R; i0 += kLmEpiThreads) {
        const int c = min((i0 + lane) / kLmEpiWarps, p.R - 1), w = lane % kLmEpiWarps;
        const SampStat o = run[w * p.NP + c];
        SampStat st = o;
#pragma unroll
        for (int n = kLmEpiWarps / 2; n >= 1; n >>= 1) {
          const float om = __shfl_xor_sync(0xffffffffu, st.m, n);
          const int oa = __shfl_xor_sync(0xffffffffu, st.arg, n);
          if (better(om, oa, st.m, st.arg)) {
            st.m = om;
            st.arg = oa;
          }
        }
        if (s_tau[c] > 0.f && o.m != -INFINITY && o.m != st.m) st.S = ff_mul(o.S, exp_diff_ff(o.m, st.m, s_tau[c]));
        st.S = warp_sum_ff<kLmEpiWarps>(st.S);
        if (w == 0 && i0 + lane < kLmEpiWarps * p.R) p.stats[static_cast<size_t>(c) * p.G + grp] = st;
      }
    }
  }

  // ---- teardown ----
  __syncthreads();
  if (*s_abort) {
    if (tid == 0) set_status(p.status, SF_DEVICE_TIMEOUT);
    if (warp == kLmProducerWarp && lane == 0) {
      // copies issued but never consumed: wait (bounded) until they land
      for (uint32_t x = static_cast<uint32_t>(s_misc[3]); x < static_cast<uint32_t>(s_misc[2]); ++x)
        (void)mbar_wait_bounded(bar(FULL + x % S), (x / S) & 1u);
    }
    __syncthreads();
  }
  if (warp == kLmMmaWarp) {
    tc_fence_after_sync();
    tmem_dealloc(tmem, p.tmem_cols);
  }
}

// ---------------------------------------------------------------------------
// sampling
// ---------------------------------------------------------------------------
__device__ __forceinline__ int chunk_start(const SampleParams &p, int c) {
  const long long e = static_cast<long long>(p.unit) * (static_cast<long long>(c) * p.T / p.Cn);
  return e < p.V ? static_cast<int>(e) : p.V;
}

// Statistics of one kSampleUnit chunk of one row (sf_sample): grid (Cn, R).
__global__ void __launch_bounds__(kFfThreads) sample_stats_kernel(const __grid_constant__ SampleParams p) {
  __shared__ ff s_d[32];
  __shared__ float s_v[32];
  __shared__ int s_i[32];
  grid_dependency_wait();
  grid_launch_dependents();
  const int c = blockIdx.x, r = blockIdx.y, tid = threadIdx.x;
  const float *row = p.logits + static_cast<size_t>(r) * p.V;
  const int e0 = c * kSampleUnit;
  const float tau = p.tau[r];
  const bool greedy = !(tau > 0.f);
  constexpr int kPer = kSampleUnit / kFfThreads;  // 8 tokens per thread, 4 consecutive
  float x[kPer];
#pragma unroll
  for (int h = 0; h < kPer / 4; ++h) {
    const int i0 = e0 + h * 4 * kFfThreads + 4 * tid;
    if (p.vec4 && i0 + 3 < p.V) {
      const float4 f = *reinterpret_cast<const float4 *>(row + i0);
      x[4 * h] = f.x;
      x[4 * h + 1] = f.y;
      x[4 * h + 2] = f.z;
      x[4 * h + 3] = f.w;
    } else {
#pragma unroll
      for (int j = 0; j < 4; ++j) x[4 * h + j] = i0 + j < p.V ? row[i0 + j] : -INFINITY;
    }
  }
  float bv = -INFINITY;
  int bi = INT_MAX;
#pragma unroll
  for (int h = 0; h < kPer / 4; ++h)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int idx = e0 + h * 4 * kFfThreads + 4 * tid + j;
      if (idx < p.V && better(x[4 * h + j], idx, bv, bi)) {
        bv = x[4 * h + j];
        bi = idx;
      }
    }
  block_argmax(bv, bi, s_v, s_i);
  ff s = ff_of(0.f);
  if (!greedy) {
#pragma unroll
    for (int e = 0; e < kPer; ++e) s = ff_add(s, ff_of(term_of(x[e], bv, tau)));
    s = block_sum(s, s_d);
  }
  if (tid == 0) p.stats[static_cast<size_t>(r) * p.Cn + c] = SampStat{bv, bi, s};
}

// Combines a row's chunk statistics, writes P' for this CTA's span of
// tokens and, in the CTA holding the crossing chunk's first
// token, draws T'.  grid (ceil(V / span), R); dynamic shared memory
// holds the row's Cn statistics.
//
// Nothing is written before the combination, while the first logits are in
// flight.  With many CTAs per SM (the other CTAs' work hides it) or few chunks,
// warp 0 combines alone, with shuffles and one barrier in all (a block-wide
// combine of ten barriers: 10 us in a wave of CTAs before its first store).
// With kBlock a thread takes each chunk, with one barrier for the maximum, two
// for the scan and one for the crossing chunk: with one or two CTAs per SM and
// the projection's 152 chunks 2.4 us instead of 5.5 (five chunks to a lane, in
// code that runs cold).
template <bool kStream, bool kBlock>
__global__ void __launch_bounds__(kFfThreads, kBlock ? 4 : kFinishCtasPerSm)
sample_finish_kernel(const __grid_constant__ SampleParams p) {
  extern __shared__ SampStat s_st[];
  __shared__ ff s_scan[kFfWarps];
  __shared__ float s_m, s_inv, s_wm[kFfWarps];
  __shared__ int s_arg, s_cross, s_crossed, s_tok, s_last, s_wi[kFfWarps];
  __shared__ ff s_base, s_target, s_bases[kBlock ? kFfThreads : 1];
  constexpr int kBatch = 4;
  constexpr unsigned kAll = 0xffffffffu;
  grid_dependency_wait();  // the statistics and logits come from the previous kernels
  grid_launch_dependents();
  const int r = blockIdx.y, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const float4 rec = kBlock && tid < p.Cn  // this thread's chunk
                         ? __ldcg(reinterpret_cast<const float4 *>(p.stats + static_cast<size_t>(r) * p.Cn) + tid)
                         : make_float4(-INFINITY, __int_as_float(INT_MAX), 0.f, 0.f);
  const float *row = p.logits + static_cast<size_t>(r) * p.V;
  float *prow = p.probs + static_cast<size_t>(r) * p.V;
  const float tau = p.tau[r];
  const bool greedy = !(tau > 0.f);
  const int x0 = blockIdx.x * p.span;
  const int x1 = min(p.V, x0 + p.span);
  auto load4 = [&](int x) {
    const float4 *at = reinterpret_cast<const float4 *>(row + x);
    return kStream ? __ldcg(at) : __ldcs(at);
  };
  float4 f[kBatch];  // the vector path's first tokens
  if (p.vec4 && !greedy) {
#pragma unroll
    for (int j = 0; j < kBatch; ++j) {
      const int x = x0 + 4 * tid + j * 4 * kFfThreads;
      if (x < x1) f[j] = load4(x);
    }
  }
  float m, invS = 0.f;
  int arg, cs = -1;
  ff target;
  bool crossed = false;
  if constexpr (kBlock) {
    const float u = p.u[r];
    // row maximum and its first index
    m = rec.x;
    arg = __float_as_int(rec.y);
    warp_argmax(m, arg);
    if (lane == 0) {
      s_wm[warp] = m;
      s_wi[warp] = arg;
    }
    if (tid == 0) {
      s_cross = INT_MAX;
      s_tok = INT_MAX;
      s_last = -1;
    }
    __syncthreads();
    m = lane < kFfWarps ? s_wm[lane] : -INFINITY;
    arg = lane < kFfWarps ? s_wi[lane] : INT_MAX;
    warp_argmax(m, arg);
    if (!greedy) {
      // chunk masses relative to m, and their prefix over the threads
      const ff mass = rec.x == -INFINITY ? ff_of(0.f) : ff_mul(ff{rec.z, rec.w}, exp_diff_ff(rec.x, m, tau));
      ff total, next;
      const ff ex = block_scan2(mass, s_scan, &total, &next);
      invS = ff_div_to_f(1.f, total);
      target = ff_mul(total, u);
      crossed = ff_lt(target, total);  // not for u >= 1 or NaN: then the last chunk with mass
      // u < 0: the first chunk, as by one warp
      const bool here = ff_lt(target, ff_of(0.f)) ? tid == 0 : ff_pos(mass) && (!crossed || !ff_lt(target, ex));
      // (rounded prefixes may step back behind a chunk of next to no mass, so that
      // two chunks hold the target: the first one)
      if (crossed && here && ff_lt(target, next)) {
        s_bases[tid] = ex;
        atomicMin(&s_cross, tid);
      }
      __syncthreads();
      if (s_cross == INT_MAX) {  // nothing crossed, or rounding put the target between two chunks' intervals
        if (here) atomicMax(&s_last, tid);
        __syncthreads();
        const int owner = s_last;
        __syncthreads();
        if (tid == owner) {
          s_cross = tid;
          s_bases[tid] = ex;
        }
        if (tid == 0) s_last = -1;
        __syncthreads();
      }
      cs = s_cross < INT_MAX ? s_cross : -1;
    }
  } else {
    if (tid < 32) {
      const SampStat *st = p.stats + static_cast<size_t>(r) * p.Cn;
#pragma unroll 4
      for (int c = lane; c < p.Cn; c += 32) s_st[c] = st[c];
      __syncwarp();
      // lane l owns chunks [c_lo, c_hi), in order
      const int c_lo = lane * p.Cn / 32, c_hi = (lane + 1) * p.Cn / 32;
      // row maximum and its first index
      m = -INFINITY;
      arg = INT_MAX;
      for (int c = c_lo; c < c_hi; ++c)
        if (better(s_st[c].m, s_st[c].arg, m, arg)) {
          m = s_st[c].m;
          arg = s_st[c].arg;
        }
      warp_argmax(m, arg);
      if (!greedy) {
        // chunk masses relative to m, and their prefix over the lanes: excl of a
        // lane is, bit for bit, incl of the lane before
        ff incl = ff_of(0.f);
        for (int c = c_lo; c < c_hi; ++c) {
          const ff w = s_st[c].m == -INFINITY ? ff_of(0.f) : ff_mul(s_st[c].S, exp_diff_ff(s_st[c].m, m, tau));
          s_st[c].S = w;
          incl = ff_add(incl, w);
        }
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const ff n = shfl_up_ff(incl, o);
          if (lane >= o) incl = ff_add(n, incl);
        }
        const ff prev = shfl_up_ff(incl, 1);
        const ff total = ff{__shfl_sync(kAll, incl.hi, 31), __shfl_sync(kAll, incl.lo, 31)};
        target = ff_mul(total, p.u[r]);
        // the first chunk whose inclusive prefix exceeds the target
        ff cum = lane > 0 ? prev : ff_of(0.f);
        ff base = cum;
        int cand = INT_MAX, lastpos = -1;
        for (int c = c_lo; c < c_hi; ++c) {
          const ff w = s_st[c].S;
          const ff nxt = ff_add(cum, w);
          if (ff_pos(w)) lastpos = c;
          if (cand == INT_MAX && ff_lt(target, nxt)) {
            cand = c;
            base = cum;
          }
          cum = nxt;
        }
        const unsigned any = __ballot_sync(kAll, cand != INT_MAX);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) lastpos = max(lastpos, __shfl_xor_sync(kAll, lastpos, o));
        if (lane == (any ? __ffs(any) - 1 : 0)) {
          s_crossed = any != 0u;
          s_cross = any ? cand : lastpos;  // no crossing (u >= 1 or NaN): last positive chunk
          s_base = base;
          s_target = target;
          s_inv = ff_div_to_f(1.f, total);
        }
      }
      if (lane == 0) {
        s_m = m;
        s_arg = arg;
        s_tok = INT_MAX;
        s_last = -1;
      }
    }
    __syncthreads();
    m = s_m;
    arg = s_arg;
    if (!greedy) {
      target = s_target;
      crossed = s_crossed != 0;
      cs = s_cross;
      invS = s_inv;
    }
  }
  if (greedy) {
    // one-hot P', T' = the first argmax
    for (int x = x0 + tid; x < x1; x += kFfThreads) prow[x] = x == arg ? 1.f : 0.f;
    if (tid == 0 && arg >= x0 && arg < x1) p.tokens[r] = arg;
    return;
  }

  // P' for this CTA's span.  Rows are 16-byte aligned and the span a
  // multiple of 4 in the vector path, so a float4 is either wholly inside
  // the span or wholly outside; each thread issues the next kBatch loads
  // before the arithmetic and stores of the current ones.
  if (p.vec4) {
    constexpr int kStep = 4 * kFfThreads * kBatch;
    for (int base = x0 + 4 * tid; base < x1; base += kStep) {
      float4 g[kBatch];
#pragma unroll
      for (int j = 0; j < kBatch; ++j) {
        const int x = base + kStep + j * 4 * kFfThreads;
        if (x < x1) g[j] = load4(x);
      }
#pragma unroll
      for (int j = 0; j < kBatch; ++j) {
        const int x = base + j * 4 * kFfThreads;
        if (x < x1) {
          float4 o;
          if (tau == 1.f) {  // constant, so that the divisions are branched over once
            o.x = __fmul_rn(term_of(f[j].x, m, 1.f), invS);
            o.y = __fmul_rn(term_of(f[j].y, m, 1.f), invS);
            o.z = __fmul_rn(term_of(f[j].z, m, 1.f), invS);
            o.w = __fmul_rn(term_of(f[j].w, m, 1.f), invS);
          } else {
            o.x = __fmul_rn(term_of(f[j].x, m, tau), invS);
            o.y = __fmul_rn(term_of(f[j].y, m, tau), invS);
            o.z = __fmul_rn(term_of(f[j].z, m, tau), invS);
            o.w = __fmul_rn(term_of(f[j].w, m, tau), invS);
          }
          if constexpr (kStream) __stcs(reinterpret_cast<float4 *>(prow + x), o);
          else *reinterpret_cast<float4 *>(prow + x) = o;
        }
        f[j] = g[j];
      }
    }
  } else {
    for (int x = x0 + tid; x < x1; x += kFfThreads)
      prow[x] = __fmul_rn(term_of(row[x], m, tau), invS);
  }

  if (cs < 0) return;  // no positive chunk: unreachable for finite logits
  const int e0 = chunk_start(p, cs), e1 = chunk_start(p, cs + 1);
  if (e0 < x0 || e0 >= x1) return;

  // scan the chunk in ascending order, 4 consecutive tokens per thread
  ff base = kBlock ? s_bases[cs] : s_base;
  int lastpos = -1;
  for (int s0 = e0; s0 < e1; s0 += 4 * kFfThreads) {
    float t[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int x = s0 + 4 * tid + j;
      t[j] = x < e1 ? term_of(row[x], m, tau) : 0.f;
      if (t[j] > 0.f) lastpos = x;
    }
    ff tot;
    const ff ex = block_scan2(ff_add(two_sum(t[0], t[1]), two_sum(t[2], t[3])), s_scan, &tot);
    if (crossed) {
      ff cum = ff_add(base, ex);
      int at = INT_MAX;  // the thread's first token past the target
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        cum = ff_add(cum, ff_of(t[j]));
        if (at == INT_MAX && ff_lt(target, cum)) at = s0 + 4 * tid + j;
      }
      at = __reduce_min_sync(kAll, at);
      if (at != INT_MAX && (tid & 31) == 0) atomicMin(&s_tok, at);
    }
    __syncthreads();
    if (s_tok != INT_MAX) {
      if (tid == 0) p.tokens[r] = s_tok;
      return;
    }
    base = ff_add(base, tot);
  }
  // nothing crossed (rounding, u >= 1 or NaN): the chunk's last token with mass
  lastpos = __reduce_max_sync(kAll, lastpos);
  if (lastpos >= 0 && (tid & 31) == 0) atomicMax(&s_last, lastpos);
  __syncthreads();
  if (tid == 0) p.tokens[r] = s_last;
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
static int np_of(int R) { return (R + 15) / 16 * 16; }

// As many slots as fit: the weight stream needs ~200 KB in flight per SM
// (152064 x 3584, 128 draft rows: 183 us with four 48 KB slots, 196 with three).
static int lm_stages(const DeviceInfo &dev, uint32_t stage_bytes, int NP) {
  int s = kLmMaxStages;
  while (s > 2 && LmSmem::bytes(s, stage_bytes, NP) > static_cast<size_t>(dev.max_smem_optin)) --s;
  return s;
}

static int lm_setup(const DeviceInfo &dev) {
  static std::mutex mu;
  static bool done[64] = {};
  if (dev.ordinal < 0 || dev.ordinal >= 64) return fail(SF_ERR_UNSUPPORTED, "device ordinal %d", dev.ordinal);
  std::lock_guard<std::mutex> lock(mu);
  if (done[dev.ordinal]) return SF_OK;
  cudaError_t e = cudaFuncSetAttribute(lm_head_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       dev.max_smem_optin);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(sample_finish_kernel<false, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             kMaxStatChunks * static_cast<int>(sizeof(SampStat)));
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(sample_finish_kernel<true, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             kMaxStatChunks * static_cast<int>(sizeof(SampStat)));
  if (e != cudaSuccess) return fail(SF_ERR_CUDA, "cudaFuncSetAttribute (draft tail): %s", cudaGetErrorString(e));
  done[dev.ordinal] = true;
  return SF_OK;
}

// Tensor maps of the weights {hidden, V} (box 64 x tile, 64 x ha, 64 x hb) and
// hidden states {hidden, R} (box 64 x NP), cached by (base, rows, hidden, box
// rows).
static int lm_tensor_map(CUtensorMap *out, const void *base, uint64_t rows, int hidden, uint32_t box_rows) {
  static std::mutex mu;
  static std::map<std::tuple<const void *, uint64_t, int, uint32_t>, CUtensorMap> maps;
  const auto key = std::make_tuple(base, rows, hidden, box_rows);
  {
    std::lock_guard<std::mutex> lock(mu);
    auto it = maps.find(key);
    if (it != maps.end()) {
      *out = it->second;
      return SF_OK;
    }
  }
  const uint64_t dims[2] = {static_cast<uint64_t>(hidden), rows};
  const uint64_t strides[1] = {static_cast<uint64_t>(hidden) * 2};
  const uint32_t box[2] = {static_cast<uint32_t>(kLmChunkK), box_rows};
  const int st = encode_tensor_map_bf16(out, base, 2, dims, strides, box);
  if (st != SF_OK) return st;
  std::lock_guard<std::mutex> lock(mu);
  if (maps.size() >= 4096) maps.clear();
  maps.emplace(key, *out);
  return SF_OK;
}

static int check_lm_args(const void *hidden, const void *weight, int R, int hidden_size, int V,
                         const float *logits) {
  if (R < 1 || R > SF_MAX_DRAFT_ROWS)
    return fail(SF_ERR_INVALID_ARG, "R=%d outside [1, %d]", R, SF_MAX_DRAFT_ROWS);
  if (hidden_size < 8 || hidden_size % 8 != 0 || hidden_size > (1 << 20))
    return fail(SF_ERR_INVALID_ARG, "hidden_size=%d must be a multiple of 8 in [8, 2^20]", hidden_size);
  if (V < 1 || V > SF_MAX_VOCAB) return fail(SF_ERR_INVALID_ARG, "V=%d outside [1, %d]", V, SF_MAX_VOCAB);
  if (!hidden || !weight || !logits) return fail(SF_ERR_INVALID_ARG, "a required pointer is NULL");
  if (!aligned(hidden, 16) || !aligned(weight, 16))
    return fail(SF_ERR_INVALID_ARG, "hidden and weight must be 16-byte aligned");
  if (!aligned(logits, 4)) return fail(SF_ERR_INVALID_ARG, "logits must be 4-byte aligned");
  return SF_OK;
}

static int check_sample_args(int R, int V, const float *uniforms, const float *temperature,
                             const float *probs, const int32_t *tokens) {
  if (R < 1 || R > 65535) return fail(SF_ERR_INVALID_ARG, "R=%d outside [1, 65535]", R);
  if (V < 1 || V > SF_MAX_VOCAB) return fail(SF_ERR_INVALID_ARG, "V=%d outside [1, %d]", V, SF_MAX_VOCAB);
  if (!uniforms || !temperature || !probs || !tokens)
    return fail(SF_ERR_INVALID_ARG, "a required pointer is NULL");
  if (!aligned(uniforms, 4) || !aligned(temperature, 4) || !aligned(probs, 4) || !aligned(tokens, 4))
    return fail(SF_ERR_INVALID_ARG, "buffers must be 4-byte aligned");
  return SF_OK;
}

static size_t stats_bytes(int R, int V, int sm_count) {
  const size_t cn = static_cast<size_t>((V + kSampleUnit - 1) / kSampleUnit);
  const size_t cn_max = cn > static_cast<size_t>(sm_count) ? cn : static_cast<size_t>(sm_count);
  return 256 + round_up(static_cast<size_t>(R) * cn_max * sizeof(SampStat), 256);
}

static cudaLaunchConfig_t pdl_config(dim3 grid, dim3 block, size_t smem, cudaStream_t stream,
                                     cudaLaunchAttribute *attr) {
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cfg;
}

// Launches the projection; with `stats` the epilogue also writes the per-CTA
// sampling statistics [R][G] and *G_out receives G.
static int launch_lm_head(const void *hidden, const void *weight, int R, int hidden_size, int V,
                          float *logits, const float *temperature, SampStat *stats, uint32_t *status,
                          int *G_out, cudaStream_t stream, bool w_after_wait = false,
                          bool w_keep = false, int ks = 1, int tau_div = 1) {
  DeviceInfo dev;
  int st = current_device(&dev);
  if (st != SF_OK) return st;
  if (dev.cc_major != 10) return fail(SF_ERR_UNSUPPORTED, "the LM-head kernel needs an sm_10x GPU");
  st = lm_setup(dev);
  if (st != SF_OK) return st;
  const int NP = np_of(R);
  LmParams prm;
  prm.logits = logits;
  prm.tau = temperature;
  prm.stats = stats;
  prm.status = status;
  prm.R = R;
  prm.V = V;
  prm.NP = NP;
  prm.G = projection_groups(V, dev.sm_count);
  const int q = V / prm.G;  // every CTA owns q or q + 1 rows
  const int most = q + (V % prm.G ? 1 : 0);
  // 128-row tiles where two 256-row accumulators don't fit tensor memory (more
  // than 128 draft rows) and a CTA has more than two such tiles: each tile's
  // statistics then stand between its MMAs and the next tile's, with 128 rows they
  // overlap.  144 draft rows x 128000 x 4096 275.1 -> 228.2 us, 256 x 152064 x 3584 411.1
  // -> 360.4; with fewer tiles the 256-row epilogue by eight warps is shorter (160 x
  // 60000 x 1024 81.3, 99.3 us with 128 rows).  The logits alone take 256 rows at
  // every size (256 x 152064 x 3584 245.6, 257.8 us).
  prm.tile = stats && 4 * NP > 512 && most > 2 * kLmTileV ? kLmHalf : kLmTileV;
  const int tallest = most < prm.tile ? most : prm.tile;
  prm.halves = tallest > kLmHalf ? 2 : 1;
  prm.w_bytes = static_cast<uint32_t>((tallest + 7) / 8 * 8) * (kLmChunkK * 2);
  prm.ha = (q - 1) % prm.tile + 1;
  prm.hb = q % prm.tile + 1;
  prm.KC = (hidden_size + kLmChunkK - 1) / kLmChunkK;
  prm.stage_bytes = prm.w_bytes + static_cast<uint32_t>(NP) * 128u;
  prm.stages = lm_stages(dev, prm.stage_bytes, NP);
  const uint32_t acc = static_cast<uint32_t>(prm.halves * NP);  // columns of one tile's accumulators
  prm.nbuf = 2 * acc <= 512 ? 2 : 1;
  uint32_t cols = 32;
  while (cols < static_cast<uint32_t>(prm.nbuf) * acc) cols <<= 1;
  prm.tmem_cols = cols;
  prm.idesc = idesc_bf16_f32(128, NP, 0, 0);
  prm.w_after_wait = w_after_wait ? 1 : 0;
  prm.w_keep = w_keep ? 1 : 0;
  prm.ks = ks < 1 ? 1 : (ks > prm.KC ? prm.KC : ks);
  prm.tau_div = tau_div < 1 ? 1 : tau_div;
  prm.part_stride = static_cast<long long>(R) * V;
  if (stats && prm.ks != 1) return fail(SF_ERR_INVALID_ARG, "statistics need an unsplit projection");
  const size_t smem = LmSmem::bytes(prm.stages, prm.stage_bytes, NP);
  if (smem > static_cast<size_t>(dev.max_smem_optin))
    return fail(SF_ERR_UNSUPPORTED, "LM-head ring needs %zu bytes of shared memory", smem);
  CUtensorMap tw, twa, twb, th;
  st = lm_tensor_map(&tw, weight, static_cast<uint64_t>(V), hidden_size, static_cast<uint32_t>(prm.tile));
  if (st == SF_OK)
    st = lm_tensor_map(&twa, weight, static_cast<uint64_t>(V), hidden_size, static_cast<uint32_t>(prm.ha));
  if (st == SF_OK)
    st = lm_tensor_map(&twb, weight, static_cast<uint64_t>(V), hidden_size, static_cast<uint32_t>(prm.hb));
  if (st != SF_OK) return st;
  st = lm_tensor_map(&th, hidden, static_cast<uint64_t>(R), hidden_size, static_cast<uint32_t>(NP));
  if (st != SF_OK) return st;
  cudaLaunchAttribute attr[1];
  cudaLaunchConfig_t cfg = pdl_config(dim3(prm.G * prm.ks), dim3(kLmThreads), smem, stream, attr);
  cudaError_t e = cudaLaunchKernelEx(&cfg, lm_head_kernel, tw, twa, twb, th, prm);
  if (e != cudaSuccess) return fail(SF_ERR_CUDA, "LM-head launch: %s", cudaGetErrorString(e));
  if (G_out) *G_out = prm.G;
  return SF_OK;
}

// Span per finishing CTA, a multiple of kSampleSpan.  With vector accesses at most
// two CTAs per SM as long as that leaves spans of at most 4 kSampleSpan: the kernel
// is then a chain of latencies, to which every CTA adds its combination (sampling alone, 128 x 8000
// 11.7 us with 256 CTAs, 14.7 with 512; 5 x 152064 10.7 with 250, 13.0 with 745; the
// projection and sampling of 5 x 152064 x 3584 169.9, 172.3).  Larger ones take as
// many CTAs as fit the GPU at once: the kernel is then bound by its bytes (64 x
// 32000 15.3 us with 512, 16.4 with 256), and a second, nearly empty wave cost 128
// rows of 152064 tokens a third of the kernel.  So do all sizes with scalar
// accesses, of which a thread has one in flight (projection and sampling of 32 rows
// of 33333 tokens, hidden 1024 25.3 us, 26.6 with two CTAs per SM).
static int finish_span(int R, int V, int sm_count, bool vec4) {
  auto span_of = [&](int per_sm) {
    const long long spans = static_cast<long long>(per_sm) * sm_count / R;
    const long long n = spans > 1 ? spans : 1;
    return ((V + n - 1) / n + kSampleSpan - 1) / kSampleSpan * kSampleSpan;
  };
  long long span = span_of(2);
  if (!vec4 || span > 4 * kSampleSpan) span = span_of(kFinishCtasPerSm);
  return static_cast<int>(span < V ? span : (V + 3) / 4 * 4);
}

// From this size on, logits (just written) and probabilities together no
// longer stay in the 129 MB L2 beside the weights passing through it: the
// probabilities are then stored as streaming data, so that they don't push
// out the logits that are still to be read (projection and sampling of 128 rows
// of 152064 tokens 231.2 -> 225.6 us, 96 rows 216.2 -> 211.0, 64 rows 200.6 -> 199.4).
// Smaller ones stay in L2, where the acceptance reads them (48 rows, 58 MB:
// 192 us against 193 streaming).
constexpr long long kStreamBytes = 64LL << 20;

static int launch_finish(SampleParams prm, cudaStream_t stream) {
  cudaLaunchAttribute attr[1];
  DeviceInfo dev;
  const int st = current_device(&dev);
  if (st != SF_OK) return st;
  prm.span = finish_span(prm.R, prm.V, dev.sm_count, prm.vec4 != 0);
  const int spans = (prm.V + prm.span - 1) / prm.span;
  // Projection and sampling of 5 rows, 32000 x 4096 (160 CTAs, 152 chunks) 52.1 ->
  // 49.8 us, 9 rows, 32000 x 2048 (288 CTAs) 31.0 -> 29.2; beyond two CTAs per SM the
  // block-wide combination is even (128 rows, 152064 x 3584, 5 CTAs per SM: 73.3 ->
  // 73.6 us for the sampling), and up to 32 chunks it has little to share out
  // (sampling alone, 128 x 8000, 4 chunks: 11.7 -> 11.8).
  const bool block = prm.Cn > 32 && prm.Cn <= kFfThreads &&
                     static_cast<long long>(spans) * prm.R <= 2LL * dev.sm_count;
  cudaLaunchConfig_t cfg = pdl_config(dim3(spans, prm.R), dim3(kFfThreads),
                                      block ? 0 : static_cast<size_t>(prm.Cn) * sizeof(SampStat), stream, attr);
  const bool streaming = 8LL * prm.R * prm.V >= kStreamBytes;
  auto *kernel = block       ? (streaming ? sample_finish_kernel<true, true> : sample_finish_kernel<false, true>)
                 : streaming ? sample_finish_kernel<true, false>
                             : sample_finish_kernel<false, false>;
  cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, prm);
  if (e != cudaSuccess) return fail(SF_ERR_CUDA, "sampling launch: %s", cudaGetErrorString(e));
  return SF_OK;
}

int launch_projection_stats(const void *hidden, const void *weight, int R, int hidden_size, int V,
                            float *logits, const float *temperature, int rows_per_temperature,
                            SampStat *stats, uint32_t *status, int *G_out, cudaStream_t stream) {
  const int st = check_lm_args(hidden, weight, R, hidden_size, V, logits);
  if (st != SF_OK) return st;
  return launch_lm_head(hidden, weight, R, hidden_size, V, logits, temperature, stats, status, G_out,
                        stream, false, false, 1, rows_per_temperature);
}

int projection_groups(int V, int sm_count) {
  const int g = (V + kLmHalf - 1) / kLmHalf;
  return g < sm_count ? g : sm_count;
}

int projection_splits(int V, int hidden_size, int sm_count) {
  const int G = projection_groups(V, sm_count);
  const int KC = (hidden_size + kLmChunkK - 1) / kLmChunkK;
  int ks = sm_count / G;
  if (ks > KC) ks = KC;
  return ks < 1 ? 1 : ks;
}

int launch_projection(const void *rows_r, const void *rows_v, int R, int hidden_size, int V,
                      float *out, uint32_t *status, bool inputs_after_wait, bool keep_v_rows,
                      int splits, cudaStream_t stream) {
  const int st = check_lm_args(rows_r, rows_v, R, hidden_size, V, out);
  if (st != SF_OK) return st;
  return launch_lm_head(rows_r, rows_v, R, hidden_size, V, out, nullptr, nullptr, status, nullptr,
                        stream, inputs_after_wait, keep_v_rows, splits);
}

}  // namespace sf

extern "C" {

size_t sf_draft_tail_workspace_size(int R, int V) {
  using namespace sf;
  if (R < 1 || R > 65535 || V < 1 || V > SF_MAX_VOCAB) return 0;
  DeviceInfo dev;
  if (current_device(&dev) != SF_OK) return 0;
  return stats_bytes(R, V, dev.sm_count);
}

int sf_lm_head(const void *hidden, const void *weight, int R, int hidden_size, int V, float *logits,
               void *workspace, size_t workspace_bytes, cudaStream_t stream) {
  using namespace sf;
  clear_error();
  int st = check_lm_args(hidden, weight, R, hidden_size, V, logits);
  if (st != SF_OK) return st;
  if (!workspace || !aligned(workspace, 256) || workspace_bytes < 256)
    return fail(SF_ERR_WORKSPACE, "workspace must be non-NULL, 256-byte aligned and >= 256 bytes");
  return launch_lm_head(hidden, weight, R, hidden_size, V, logits, nullptr, nullptr,
                        static_cast<uint32_t *>(workspace), nullptr, stream);
}

int sf_sample(const float *logits, const float *uniforms, const float *temperature, int R, int V,
              float *probs, int32_t *tokens, void *workspace, size_t workspace_bytes,
              cudaStream_t stream) {
  using namespace sf;
  clear_error();
  int st = check_sample_args(R, V, uniforms, temperature, probs, tokens);
  if (st != SF_OK) return st;
  if (!logits || !aligned(logits, 4)) return fail(SF_ERR_INVALID_ARG, "logits NULL or misaligned");
  DeviceInfo dev;
  st = current_device(&dev);
  if (st != SF_OK) return st;
  st = lm_setup(dev);
  if (st != SF_OK) return st;
  if (!workspace || !aligned(workspace, 256))
    return fail(SF_ERR_WORKSPACE, "workspace must be non-NULL and 256-byte aligned");
  const size_t need = stats_bytes(R, V, dev.sm_count);
  if (workspace_bytes < need)
    return fail(SF_ERR_WORKSPACE, "workspace has %zu bytes, needs %zu", workspace_bytes, need);
  SampleParams prm;
  prm.logits = logits;
  prm.stats = reinterpret_cast<SampStat *>(static_cast<uint8_t *>(workspace) + 256);
  prm.u = uniforms;
  prm.tau = temperature;
  prm.probs = probs;
  prm.tokens = tokens;
  prm.R = R;
  prm.V = V;
  prm.Cn = (V + kSampleUnit - 1) / kSampleUnit;
  prm.unit = kSampleUnit;
  prm.T = prm.Cn;
  prm.vec4 = (V % 4 == 0) && aligned(logits, 16) && aligned(probs, 16);
  cudaLaunchAttribute attr[1];
  cudaLaunchConfig_t cfg = pdl_config(dim3(prm.Cn, R), dim3(kFfThreads), 0, stream, attr);
  cudaError_t e = cudaLaunchKernelEx(&cfg, sample_stats_kernel, prm);
  if (e != cudaSuccess) return fail(SF_ERR_CUDA, "sampling statistics launch: %s", cudaGetErrorString(e));
  return launch_finish(prm, stream);
}

int sf_draft_sample(const void *hidden, const void *weight, const float *uniforms,
                    const float *temperature, int R, int hidden_size, int V, float *logits,
                    float *probs, int32_t *tokens, void *workspace, size_t workspace_bytes,
                    cudaStream_t stream) {
  using namespace sf;
  clear_error();
  int st = check_lm_args(hidden, weight, R, hidden_size, V, logits);
  if (st != SF_OK) return st;
  st = check_sample_args(R, V, uniforms, temperature, probs, tokens);
  if (st != SF_OK) return st;
  DeviceInfo dev;
  st = current_device(&dev);
  if (st != SF_OK) return st;
  if (!workspace || !aligned(workspace, 256))
    return fail(SF_ERR_WORKSPACE, "workspace must be non-NULL and 256-byte aligned");
  const size_t need = stats_bytes(R, V, dev.sm_count);
  if (workspace_bytes < need)
    return fail(SF_ERR_WORKSPACE, "workspace has %zu bytes, needs %zu", workspace_bytes, need);
  SampleParams prm;
  prm.stats = reinterpret_cast<SampStat *>(static_cast<uint8_t *>(workspace) + 256);
  int G = 0;
  st = launch_lm_head(hidden, weight, R, hidden_size, V, logits, temperature, prm.stats,
                      static_cast<uint32_t *>(workspace), &G, stream);
  if (st != SF_OK) return st;
  prm.logits = logits;
  prm.u = uniforms;
  prm.tau = temperature;
  prm.probs = probs;
  prm.tokens = tokens;
  prm.R = R;
  prm.V = V;
  prm.Cn = G;  // chunk c = CTA c's rows [c*V/G, (c+1)*V/G)
  prm.unit = 1;
  prm.T = V;
  prm.vec4 = (V % 4 == 0) && aligned(logits, 16) && aligned(probs, 16);
  return launch_finish(prm, stream);
}

}  // extern "C"
