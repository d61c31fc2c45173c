// visual_compress.cu -- visual token compression of the draft model
// (Sec. 3.2, Eq. 3; Algorithm 1) on sm_103a:
//
//     F^_V = softmax(Q F_V^T) F_V
//
// per image or frame, with the learnable query set Q (C x d) shared by all
// frames, F_V (N x d) acting as both keys and values, the softmax over the
// frame's N tokens and no score scale (Eq. 3 writes none).  The sizes are
// the paper's: N = 576 -> C = 64 for LLaVA images, 324 -> 36 for QwenVL, at
// the hidden size d of the target (4096, 3584).
//
// GB300 design.  The work is 4 C N d flops per frame over 2 N d bytes of
// features: 2 C = 128 flop/byte for LLaVA, below the bf16 tensor ridge
// (~286), so the floor is reading the features once at HBM speed, and only
// tensor cores keep the arithmetic under that.  Three launches:
//  1. scores S = Q F_V^T for all frames at once ([C][F*N] fp32) with the
//     tcgen05 projection kernel of draft_tail.cu (queries as the N side, the
//     F*N feature rows streamed as the M side), the hidden dimension split
//     into ks ranges when F*N has too few 128-row tiles to fill the GPU
//     (each split writes partial sums); it copies the features after the
//     dependency wait and leaves them in L2 (evict_last) for 3.;
//  2. compress_softmax_kernel: a warp, or a block where there are several
//     partials, per (frame, query) sums the ks partials in a fixed order;
//     one warp takes the row max, and writes the unnormalised weights
//     exp(s - max) rounded to bf16 into P [C][F][Np] (Np = N rounded up to
//     64, zeros past N) and the sum of the rounded weights into l [F][C];
//  3. compress_apply_kernel, up to two CTAs per SM, each with some of a frame's
//     groups of 128 columns: the transposed product O^T = F_V^T P^T as a
//     pipelined tcgen05 GEMM with M = 128 feature columns (A = the frame's
//     features, MN-major), N = C padded to 16 (B = P, K-major) and K = 16
//     tokens, two accumulators in tensor memory.
// Measured per call (graph of calls over three inputs), against a CTA per 128
// columns and one softmax warp per query: 5 x 576 x 4096, C 64: 23.6 -> 16.4 us;
// 128 x 144 x 3584, C 16: 55.9 -> 46.6; 1 x 576 x 4096, C 64: 36.9 -> 14.5.
// A single launch with a cluster per frame, the scores exchanged through
// distributed shared memory, was slower (31.7 and 48.9 us): a CTA's 147 KB of
// partial scores and 74 KB of weights move at ~13 bytes per clock.  Computing
// the weights in the third kernel instead of the second: 46.1 us for the video
// shape, 66.6 for the images.
// N is at most 768 and C at most 128.  Every wait is bounded
// (SF_DEVICE_TIMEOUT).
#include <cmath>
#include <mutex>

#include "sf_device.cuh"
#include "sf_host.h"

namespace sf {

constexpr int kVcThreads = 320;
constexpr int kVcEpiThreads = 256;  // two warps per lane quarter of tensor memory
constexpr int kVcMmaWarp = 8;
constexpr int kVcProducerWarp = 9;
constexpr int kVcCols = 128;        // feature columns per group (MMA M)
constexpr int kVcTokens = 64;       // tokens per box of weights (128 bytes)
constexpr int kVcMaxTokens = 768;   // N
constexpr int kVcMaxQueries = 128;  // C
constexpr int kVcMaxStages = 8;
constexpr int kVcSoftmaxWarpThreads = 64;  // softmax CTA where a warp takes a query

struct VcSoftmaxParams {
  const float *scores;  // [ks][C][F*N]
  __nv_bfloat16 *P;     // [C][F*Np]
  float *l;             // [F][C]
  long long part_stride;  // C*F*N
  int ks, F, N, C, Np;
};

struct VcParams {
  const float *l;       // [F][C]
  __nv_bfloat16 *out;   // [F][C][d]
  uint32_t *status;
  int F, N, C, Cp, d, Np;
  int groups, per_frame;  // d / 128 column groups, split over per_frame CTAs
  int T, slots;           // tokens per ring slot (a multiple of 16), slots per group
  int stages;
  uint32_t stage_bytes;   // 2 x T x 128 bytes of features, then T / 64 boxes of weights
  uint32_t tmem_cols;
};

static size_t vc_smem_bytes(int stages, uint32_t stage_bytes, int C) {
  return 1024 + static_cast<size_t>(stages) * stage_bytes + 8 * (2 * stages + 5) + 64 + 4 * C;
}

// One query of one frame: the partial scores summed in split order, then the
// unnormalised weights exp(s - max) rounded to bf16, zeros past N, and their
// sum l.  Threads: kT share the partials' loads and sums, then the query's first
// warp goes on alone, lane t with tokens 64 i + 2 t and the next.  l is added as
// 32 chains (chain t: tokens t, t + 32, ...) and a tree over them.  Neither order
// depends on kT.
// Bound by memory round trips, so kFly partials of every token of a thread are in
// flight at once (loads of one partial behind the sums of the one before: 17.6
// us alone for 5 x 576 x 4096, C 64).  grid (F, queries / those of a CTA).
template <int kT>
__global__ void __launch_bounds__(kT > 32 ? kT : kVcSoftmaxWarpThreads)
compress_softmax_kernel(const __grid_constant__ VcSoftmaxParams p) {
  constexpr int kPairs = kVcMaxTokens / 64;                // token pairs per lane of the first warp
  constexpr int kOwn = kVcMaxTokens / kT;                  // tokens whose partials a thread adds
  constexpr int kFly = 72 / kOwn;                          // partials in flight
  constexpr int kQueries = kT > 32 ? 1 : kVcSoftmaxWarpThreads / kT;  // per CTA
  constexpr unsigned kAll = 0xffffffffu;
  __shared__ float2 s_x[kT > 32 ? kVcMaxTokens / 2 : 1];
  grid_dependency_wait();  // the partial scores come from the projection
  grid_launch_dependents();
  const int f = blockIdx.x, c = blockIdx.y * kQueries + threadIdx.x / kT;
  const int t = threadIdx.x % kT, lane = threadIdx.x & 31;
  if (c >= p.C) return;
  const float *row = p.scores + static_cast<long long>(c) * p.F * p.N + static_cast<long long>(f) * p.N;
  auto token = [&](int i) { return kT > 32 ? t + kT * i : 64 * (i / 2) + 2 * t + i % 2; };
  float x[2 * kPairs];
#pragma unroll
  for (int i = 0; i < kOwn; ++i) x[i] = token(i) < p.N ? row[token(i)] : -INFINITY;
#pragma unroll 1
  for (int s0 = 1; s0 < p.ks; s0 += kFly) {
    float v[kFly][kOwn];
#pragma unroll
    for (int u = 0; u < kFly; ++u) {
      const float *part = row + (s0 + u) * p.part_stride;
#pragma unroll
      for (int i = 0; i < kOwn; ++i)
        v[u][i] = s0 + u < p.ks && token(i) < p.N ? part[token(i)] : 0.f;
    }
#pragma unroll
    for (int u = 0; u < kFly; ++u) {
#pragma unroll
      for (int i = 0; i < kOwn; ++i) x[i] += v[u][i];
    }
  }
  if constexpr (kT > 32) {
#pragma unroll
    for (int i = 0; i < kOwn; ++i) reinterpret_cast<float *>(s_x)[token(i)] = x[i];
    __syncthreads();
    if (t >= 32) return;
#pragma unroll
    for (int i = 0; i < kPairs; ++i) {
      const float2 pair = s_x[32 * i + lane];
      x[2 * i] = pair.x;
      x[2 * i + 1] = pair.y;
    }
  }
  float m = -INFINITY;
#pragma unroll
  for (int i = 0; i < 2 * kPairs; ++i) m = fmaxf(m, x[i]);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(kAll, m, o));
  constexpr float kLog2e = 1.4426950408889634f;
  const float mb = m * kLog2e;
  uint32_t *prow = reinterpret_cast<uint32_t *>(p.P + static_cast<long long>(c) * p.F * p.Np +
                                                static_cast<long long>(f) * p.Np);
  float l = 0.f;
#pragma unroll
  for (int i = 0; i < kPairs; ++i) {
    const int n = 64 * i + 2 * lane;
    if (64 * i < p.Np) {
      const __nv_bfloat162 w = __floats2bfloat162_rn(n < p.N ? fast_exp2(fmaf(x[2 * i], kLog2e, -mb)) : 0.f,
                                                     n + 1 < p.N ? fast_exp2(fmaf(x[2 * i + 1], kLog2e, -mb)) : 0.f);
      const uint32_t bits = *reinterpret_cast<const uint32_t *>(&w);
      prow[32 * i + lane] = bits;
      // chain `lane`: tokens 64 i + lane and 64 i + 32 + lane
      const uint32_t w0 = __shfl_sync(kAll, bits, lane >> 1), w1 = __shfl_sync(kAll, bits, 16 + (lane >> 1));
      l += __uint_as_float(lane & 1 ? w0 & 0xffff0000u : w0 << 16);
      l += __uint_as_float(lane & 1 ? w1 & 0xffff0000u : w1 << 16);
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) l += __shfl_xor_sync(kAll, l, o);
  if (lane == 0) p.l[f * p.C + c] = l;
}

// O^T = F_V^T P^T of a frame: CTA (part, f) takes its share of the frame's
// groups of 128 columns, M = 128 columns, N = C padded to 16, K = 16 tokens.
// Warp 9 streams the features (MN-major A) and the weights (K-major B) of T
// tokens per ring slot, warp 8 issues the MMAs into one of two accumulators,
// warps 0-7 divide by l and store bf16.  One CTA per 128 columns and copies
// issued from a one-lane branch (~500 cycles each, three per slot) took 10.4 us
// for 5 x 576 x 4096 and 28.8 us for 128 x 144 x 3584 alone.
__global__ void __launch_bounds__(kVcThreads)
compress_apply_kernel(const __grid_constant__ CUtensorMap tmap_f, const __grid_constant__ CUtensorMap tmap_p,
                      const __grid_constant__ VcParams p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t *smem = reinterpret_cast<uint8_t *>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  const int S = p.stages;
  const uint32_t ring = smem_addr(smem);
  uint64_t *bar_mem = reinterpret_cast<uint64_t *>(smem + static_cast<size_t>(S) * p.stage_bytes);
  int *s_misc = reinterpret_cast<int *>(bar_mem + 2 * S + 5);  // [0] TMEM, [1] abort, [2] issued, [3] consumed
  float *s_inv = reinterpret_cast<float *>(s_misc + 16);       // 1 / l of the frame's queries
  volatile int *s_abort = s_misc + 1;
  const uint32_t bars = smem_addr(bar_mem);
  const int FULL = 0, EMPTY = S, OFULL = 2 * S, OEMPTY = 2 * S + 2, FIN = 2 * S + 4;
  auto bar = [&](int i) -> uint32_t { return bars + 8u * static_cast<uint32_t>(i); };

  const int f = blockIdx.y;
  const int tid = threadIdx.x, warp = uniform_warp_id(), lane = tid & 31;
  // this CTA's column groups, taken last first: the scores read the columns
  // in ascending order, so the last ones are the likeliest to be in L2 still
  const int part = blockIdx.x;
  const int g0 = part * p.groups / p.per_frame, g1 = (part + 1) * p.groups / p.per_frame;

  grid_launch_dependents();
  if (tid == 0) {
    for (int i = 0; i < S; ++i) {
      mbar_init(bar(FULL + i), 1);
      mbar_init(bar(EMPTY + i), 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(bar(OFULL + i), 1);
      mbar_init(bar(OEMPTY + i), kVcEpiThreads);
    }
    mbar_init(bar(FIN), 1);
    fence_mbar_init();
    prefetch_tensormap(&tmap_f);
    prefetch_tensormap(&tmap_p);
    s_misc[1] = 0;
    s_misc[2] = 0;
    s_misc[3] = 0;
  }
  __syncthreads();  // barrier initialisation visible to every role
  // Tensor memory only once the previous kernel on the stream has completed
  // (a predecessor still waiting for its own predecessor may not have
  // allocated yet; holding TMEM here could deadlock the pair).
  uint32_t tmem = 0;
  if (warp != kVcProducerWarp) {
    if (warp == kVcMmaWarp) {
      grid_dependency_wait();
      tmem_alloc(smem_addr(s_misc), p.tmem_cols);
      tmem_relinquish_alloc_permit();
      tc_fence_before_sync();
    }
    named_bar_sync(3, kVcEpiThreads + 32);
    tc_fence_after_sync();
    tmem = static_cast<uint32_t>(s_misc[0]);
  }

  const uint32_t half = static_cast<uint32_t>(p.T) * 128u;       // 64 columns of a slot's tokens
  const uint32_t pbox = static_cast<uint32_t>(p.Cp) * 128u;      // the weights of 64 tokens
  const int pboxes = (p.T + kVcTokens - 1) / kVcTokens;
  if (warp == kVcProducerWarp) {
    // the whole warp runs the loop and an elected lane issues, so that the
    // copies' operands are warp-uniform (see smem_desc_sw128)
    grid_dependency_wait();  // P comes from the softmax kernel
    const uint64_t pol_f = l2_policy_evict_first(), pol_p = l2_policy_evict_last();
    int slot = 0, q = 0;
    uint32_t lap = 0;  // earlier passes over the ring
    bool ok = true;
    for (int g = g1 - 1; g >= g0 && ok; --g)
      for (int t = 0; t < p.slots; ++t, ++q) {
        bool w = true;
        if (lap > 0) w = mbar_wait_or_abort(bar(EMPTY + slot), (lap - 1) & 1u, s_abort);
        if (!(ok = __all_sync(0xffffffffu, w))) break;
        const uint32_t dst = ring + static_cast<uint32_t>(slot) * p.stage_bytes, fb = bar(FULL + slot);
        if (elect_one()) {
          mbar_arrive_expect_tx(fb, p.stage_bytes);
          // the slot's tokens of columns [128 g, +64) and [128 g + 64, +64);
          // tokens past the frame are zero-filled
          tma_load_3d(dst, &tmap_f, g * kVcCols, t * p.T, f, fb, pol_f);
          tma_load_3d(dst + half, &tmap_f, g * kVcCols + 64, t * p.T, f, fb, pol_f);
          // their weights for every query (rows >= C are zero-filled)
          tma_load_2d(dst + 2 * half, &tmap_p, f * p.Np + t * p.T, 0, fb, pol_p);
          if (pboxes > 1) tma_load_2d(dst + 2 * half + pbox, &tmap_p, f * p.Np + t * p.T + kVcTokens, 0, fb, pol_p);
        }
        __syncwarp();
        if (++slot == S) {
          slot = 0;
          ++lap;
        }
      }
    if (lane == 0) s_misc[2] = q;
    __syncwarp();
  } else if (warp == kVcMmaWarp) {
    const uint32_t idesc = idesc_bf16_f32(128, p.Cp, 1, 0);  // A MN-major, B K-major
    int slot = 0, q = 0;
    uint32_t lap = 0;
    bool ok = true;
    for (int g = g1 - 1, i = 0; g >= g0 && ok; --g, ++i) {
      const int buf = i & 1;
      if (i >= 2) {
        const bool w = mbar_wait_or_abort(bar(OEMPTY + buf), (i / 2 - 1) & 1, s_abort);
        if (!(ok = __all_sync(0xffffffffu, w))) break;
        tc_fence_after_sync();
      }
      const uint32_t d = tmem + static_cast<uint32_t>(buf * p.Cp);
      for (int t = 0; t < p.slots; ++t) {
        const bool w = mbar_wait_or_abort(bar(FULL + slot), lap & 1u, s_abort);
        if (!(ok = __all_sync(0xffffffffu, w))) break;
        tc_fence_after_sync();
        if (lane == 0) s_misc[3] = ++q;
        const uint32_t base = ring + static_cast<uint32_t>(slot) * p.stage_bytes;
        // A: 16 tokens = two 8-row atoms (2 KB) into each 64-column half, the
        // halves (M) `half` apart.  B: 16 tokens = 32 bytes along the 128-byte
        // swizzled rows of P, 8-row groups 1 KB apart.
        const uint64_t a0 = smem_desc_sw128(base, half, 1024), b0 = smem_desc_sw128(base + 2 * half, 16, 1024);
        const uint64_t b1 = b0 + (pbox >> 4);
        const int steps = p.T / 16;
        const uint32_t acc = t > 0 ? 1u : 0u;
        if (elect_one()) {
#pragma unroll
          for (int k = 0; k < 4; ++k)
            if (k < steps) tc_mma_ss(d, a0 + 128 * k, b0 + 2 * k, idesc, k > 0 ? 1u : acc);
          if (steps > 4) {
#pragma unroll
            for (int k = 4; k < 8; ++k)
              if (k < steps) tc_mma_ss(d, a0 + 128 * k, b1 + 2 * (k - 4), idesc, 1u);
          }
          tc_commit(bar(EMPTY + slot));
        }
        __syncwarp();
        if (++slot == S) {
          slot = 0;
          ++lap;
        }
      }
      if (ok && elect_one()) tc_commit(bar(OFULL + buf));
      __syncwarp();
    }
    if (elect_one()) tc_commit(bar(FIN));
    __syncwarp();
    (void)mbar_wait_bounded(bar(FIN), 0);  // every MMA issued has completed
  } else {
    // ------------------------------------------------------------------
    // epilogue: lane = feature column of the group, TMEM columns = queries;
    // the two warps of a lane quarter take 16 queries in turn
    // ------------------------------------------------------------------
    grid_dependency_wait();  // l comes from the softmax kernel
    for (int c = tid; c < p.C; c += kVcEpiThreads) {
      const float l = p.l[f * p.C + c];
      s_inv[c] = l > 0.f ? 1.f / l : 0.f;
    }
    named_bar_sync(1, kVcEpiThreads);
    const int quarter = warp & 3;
    const uint32_t lane_base = tmem + (static_cast<uint32_t>(32 * quarter) << 16);
    for (int g = g1 - 1, i = 0; g >= g0; --g, ++i) {
      const int buf = i & 1;
      const bool ok = mbar_wait_or_abort(bar(OFULL + buf), (i / 2) & 1, s_abort);
      if (!__all_sync(0xffffffffu, ok)) break;
      tc_fence_after_sync();
      __nv_bfloat16 *dst =
          p.out + static_cast<size_t>(f) * p.C * p.d + g * kVcCols + 32 * quarter + lane;
#pragma unroll 1
      for (int c0 = 16 * (warp >> 2); c0 < p.C; c0 += 32) {
        uint32_t v[16];
        tmem_ld_32x32b_x16(lane_base + static_cast<uint32_t>(buf * p.Cp + c0), v);
#pragma unroll
        for (int j = 0; j < 16; ++j)
          if (c0 + j < p.C)
            dst[static_cast<size_t>(c0 + j) * p.d] = __float2bfloat16_rn(__uint_as_float(v[j]) * s_inv[c0 + j]);
      }
      tc_fence_before_sync();
      mbar_arrive(bar(OEMPTY + buf));
    }
    tc_fence_before_sync();
  }

  // ---- teardown ----
  __syncthreads();
  if (*s_abort) {
    if (tid == 0) set_status(p.status, SF_DEVICE_TIMEOUT);
    if (warp == kVcProducerWarp && lane == 0)
      for (int k = s_misc[3]; k < s_misc[2]; ++k) (void)mbar_wait_bounded(bar(FULL + k % S), (k / S) & 1);
    __syncthreads();
  }
  if (warp == kVcMmaWarp) {
    tc_fence_after_sync();
    tmem_dealloc(tmem, p.tmem_cols);
  }
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
static int vc_setup(const DeviceInfo &dev) {
  static std::mutex mu;
  static bool done[64] = {};
  if (dev.ordinal < 0 || dev.ordinal >= 64) return fail(SF_ERR_UNSUPPORTED, "device ordinal %d", dev.ordinal);
  std::lock_guard<std::mutex> lock(mu);
  if (done[dev.ordinal]) return SF_OK;
  cudaError_t e = cudaFuncSetAttribute(compress_apply_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       dev.max_smem_optin);
  if (e != cudaSuccess) return fail(SF_ERR_CUDA, "cudaFuncSetAttribute (compressor): %s", cudaGetErrorString(e));
  done[dev.ordinal] = true;
  return SF_OK;
}

struct VcLayout {
  int ks;
  size_t scores, P, l, total;
};

static VcLayout vc_layout(int F, int N, int C, int d, int sm_count) {
  VcLayout L;
  L.ks = projection_splits(F * N, d, sm_count);
  const int Np = (N + kVcTokens - 1) / kVcTokens * kVcTokens;
  size_t off = 256;
  L.scores = off;
  off = round_up(off + static_cast<size_t>(L.ks) * C * F * N * sizeof(float), 256);
  L.P = off;
  off = round_up(off + static_cast<size_t>(C) * F * Np * 2, 256);
  L.l = off;
  off = round_up(off + static_cast<size_t>(F) * C * sizeof(float), 256);
  L.total = off;
  return L;
}

static int check_vc(const void *queries, const void *features, int F, int N, int C, int d, const void *out) {
  if (F < 1 || F > 65535) return fail(SF_ERR_INVALID_ARG, "F=%d outside [1, 65535]", F);
  if (N < 1 || N > kVcMaxTokens) return fail(SF_ERR_INVALID_ARG, "N=%d outside [1, %d]", N, kVcMaxTokens);
  if (C < 1 || C > kVcMaxQueries) return fail(SF_ERR_INVALID_ARG, "C=%d outside [1, %d]", C, kVcMaxQueries);
  if (d < kVcCols || d % kVcCols != 0 || d > (1 << 20))
    return fail(SF_ERR_INVALID_ARG, "d=%d must be a multiple of 128 in [128, 2^20]", d);
  if (static_cast<long long>(F) * N > SF_MAX_VOCAB)
    return fail(SF_ERR_INVALID_ARG, "F*N=%lld above %d", static_cast<long long>(F) * N, SF_MAX_VOCAB);
  if (!queries || !features || !out) return fail(SF_ERR_INVALID_ARG, "a required pointer is NULL");
  if (!aligned(queries, 16) || !aligned(features, 16) || !aligned(out, 16))
    return fail(SF_ERR_INVALID_ARG, "queries, features and out must be 16-byte aligned");
  return SF_OK;
}

}  // namespace sf

extern "C" {

size_t sf_visual_compress_workspace_size(int F, int N, int C, int d) {
  using namespace sf;
  if (F < 1 || N < 1 || C < 1 || N > kVcMaxTokens || C > kVcMaxQueries || d < kVcCols) return 0;
  DeviceInfo dev;
  if (current_device(&dev) != SF_OK) return 0;
  return vc_layout(F, N, C, d, dev.sm_count).total;
}

int sf_visual_compress(const void *queries, const void *features, int F, int N, int C, int d,
                       void *out, void *workspace, size_t workspace_bytes, cudaStream_t stream) {
  using namespace sf;
  clear_error();
  int st = check_vc(queries, features, F, N, C, d, out);
  if (st != SF_OK) return st;
  DeviceInfo dev;
  st = current_device(&dev);
  if (st != SF_OK) return st;
  if (dev.cc_major != 10) return fail(SF_ERR_UNSUPPORTED, "the compressor needs an sm_10x GPU");
  if (!workspace || !aligned(workspace, 256))
    return fail(SF_ERR_WORKSPACE, "workspace must be non-NULL and 256-byte aligned");
  const VcLayout L = vc_layout(F, N, C, d, dev.sm_count);
  if (workspace_bytes < L.total)
    return fail(SF_ERR_WORKSPACE, "workspace has %zu bytes, needs %zu", workspace_bytes, L.total);
  st = vc_setup(dev);
  if (st != SF_OK) return st;

  uint8_t *ws = static_cast<uint8_t *>(workspace);
  uint32_t *status = reinterpret_cast<uint32_t *>(ws);
  float *scores = reinterpret_cast<float *>(ws + L.scores);
  __nv_bfloat16 *P = reinterpret_cast<__nv_bfloat16 *>(ws + L.P);
  float *lsum = reinterpret_cast<float *>(ws + L.l);
  const int Np = (N + kVcTokens - 1) / kVcTokens * kVcTokens;

  // 1. partial scores S_s = Q F_V^T over hidden range s, all frames: [ks][C][F*N]
  st = launch_projection(queries, features, C, d, F * N, scores, status, true, true, L.ks, stream);
  if (st != SF_OK) return st;

  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.stream = stream;
  cfg.attrs = attr;
  cfg.numAttrs = 1;

  // 2. weights P = bf16(exp(S - max)) and their sums l
  VcSoftmaxParams sp;
  sp.scores = scores;
  sp.P = P;
  sp.l = lsum;
  sp.part_stride = static_cast<long long>(C) * F * N;
  sp.ks = L.ks;
  sp.F = F;
  sp.N = N;
  sp.C = C;
  sp.Np = Np;
  // Threads per query: the fewest that have all partials in flight at once
  // (kFly + 1: 4, 13 or 25), or 256.  Whole calls: 5 x
  // 576 x 4096, C 64 (6 partials) 128 threads 16.4 us, 256 17.2; 1 x 576 x 4096
  // (30) 14.5, 15.0 with 128.  Few partials: 128 threads as long as the CTAs fit the
  // GPU at once (8 x 576 x 4096, C 64, 4 partials: 20.0, 20.7 with a warp per query),
  // else the warp (310 x 20 x 768, C 3: 15.4, 16.1 with 128 threads).
  const bool one_wave = static_cast<long long>(F) * C <= 5LL * dev.sm_count;
  const int threads = L.ks <= 1 || (L.ks <= 4 && !one_wave) ? 32 : (L.ks <= 13 ? 128 : 256);
  const int per_cta = threads == 32 ? kVcSoftmaxWarpThreads / 32 : 1;  // queries
  cfg.gridDim = dim3(F, (C + per_cta - 1) / per_cta);
  cfg.blockDim = dim3(per_cta * threads);
  cfg.dynamicSmemBytes = 0;
  void (*softmax)(const VcSoftmaxParams) = threads == 32    ? compress_softmax_kernel<32>
                                           : threads == 128 ? compress_softmax_kernel<128>
                                                            : compress_softmax_kernel<256>;
  cudaError_t e = cudaLaunchKernelEx(&cfg, softmax, sp);
  if (e != cudaSuccess) return fail(SF_ERR_CUDA, "compressor softmax launch: %s", cudaGetErrorString(e));

  // 3. O^T = F_V^T P^T per (128 columns, frame), divided by l
  VcParams prm;
  prm.l = lsum;
  prm.out = static_cast<__nv_bfloat16 *>(out);
  prm.status = status;
  prm.F = F;
  prm.N = N;
  prm.C = C;
  prm.Cp = (C + 15) / 16 * 16;
  prm.d = d;
  prm.Np = Np;
  prm.groups = d / kVcCols;
  // CTAs per frame: at most two per SM, each with as many column groups as that
  // leaves (one prologue for all of them), or one group each.  128 frames x
  // 3584: 2 per frame 46.8 us for the whole call, 1 55.1, 3 50.9, 28 53.5
  prm.per_frame = 2 * dev.sm_count / F;
  if (prm.per_frame < 1) prm.per_frame = 1;
  if (prm.per_frame > prm.groups) prm.per_frame = prm.groups;
  // tokens per slot: the whole frame where it is short, else 64 (one box of
  // weights)
  const int n16 = (N + 15) / 16 * 16;
  prm.T = n16 <= 96 ? n16 : kVcTokens;
  prm.slots = (n16 + prm.T - 1) / prm.T;
  const uint32_t boxes = static_cast<uint32_t>((prm.T + kVcTokens - 1) / kVcTokens);
  prm.stage_bytes = static_cast<uint32_t>(prm.T) * 256u + boxes * static_cast<uint32_t>(prm.Cp) * 128u;
  // a ring no deeper than the CTA's slots, and small enough for two CTAs per
  // SM (prologue, softmax wait and epilogue of one under the other's stream)
  const int slots = prm.slots * ((prm.groups + prm.per_frame - 1) / prm.per_frame);
  prm.stages = slots < kVcMaxStages ? slots : kVcMaxStages;
  while (prm.stages > 2 && vc_smem_bytes(prm.stages, prm.stage_bytes, C) > static_cast<size_t>(dev.max_smem_optin) / 2 - 1024)
    --prm.stages;
  uint32_t cols = 32;
  while (cols < 2u * static_cast<uint32_t>(prm.Cp)) cols <<= 1;
  prm.tmem_cols = cols;
  CUtensorMap tmap_f, tmap_p;
  {
    // frames as the third dimension: tokens past a frame's last are zero-filled
    const uint64_t row = static_cast<uint64_t>(d) * 2;
    const uint64_t dims[3] = {static_cast<uint64_t>(d), static_cast<uint64_t>(N), static_cast<uint64_t>(F)};
    const uint64_t strides[2] = {row, row * static_cast<uint64_t>(N)};
    const uint32_t box[3] = {64, static_cast<uint32_t>(prm.T), 1};
    st = encode_tensor_map_bf16(&tmap_f, features, 3, dims, strides, box);
    if (st != SF_OK) return st;
  }
  {
    const uint64_t dims[2] = {static_cast<uint64_t>(F) * Np, static_cast<uint64_t>(C)};
    const uint64_t strides[1] = {static_cast<uint64_t>(F) * Np * 2};
    const uint32_t box[2] = {static_cast<uint32_t>(kVcTokens), static_cast<uint32_t>(prm.Cp)};
    st = encode_tensor_map_bf16(&tmap_p, P, 2, dims, strides, box);
    if (st != SF_OK) return st;
  }
  cfg.gridDim = dim3(prm.per_frame, F);
  cfg.blockDim = dim3(kVcThreads);
  cfg.dynamicSmemBytes = vc_smem_bytes(prm.stages, prm.stage_bytes, C);
  e = cudaLaunchKernelEx(&cfg, compress_apply_kernel, tmap_f, tmap_p, prm);
  if (e != cudaSuccess) return fail(SF_ERR_CUDA, "compressor launch: %s", cudaGetErrorString(e));
  return SF_OK;
}

}  // extern "C"
