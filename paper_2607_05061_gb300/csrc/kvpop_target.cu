// Future-attention target for training the scorer (Sec. 3.4, App. D, App. F.1-F.2).
//
// Kernel 1, the transposed attention pass (App. D.2): for every key t of KV
// head h and every query head g of its group,
//   log mbar_t^(g) = LSE over d in [t + w, S - 1] (and d <= t + w + L with a
//                    lookahead L) of  q_d^(g) . k_t / sqrt(d_k) - LSE_d^(g),
// where LSE_d is the dense causal normaliser (exact target) or the sparse one
// returned by the prompt attention (App. D.3).  Keys play the queries: a CTA
// holds 128 keys of one (sequence, KV head) as the A operand in registers and
// streams the query rows of each head g past them in blocks of 64 (B operand,
// 16-byte cp.async into a swizzled double buffer) with the per-column LSE_d in
// shared memory; only a running max and sum are kept per (key, head) -- the
// value output of the pass is never formed.  bf16 on m16n8k16 tensor-core
// MMAs, fp32 on CUDA cores (64 keys x 128 queries per block, target_f32_kernel).
//
// bf16 with d = 128 runs on the 5th-generation tensor cores (lse_t5_kernel), which also
// serves the dense causal normalisers of App. D.1.
//
// Kernel 2 aggregates per KV head (Eq. 2, App. F.1-F.2):
//   r_t = log(eps + Agg_g mbar_t^(g) / N_t),  N_t = max(1, S - (t + w)),
// N_t clipped to L + 1 with a lookahead, Agg = max or mean; without count
// normalisation N_t = 1.
#include <cuda.h>

#include <algorithm>
#include <cstdlib>

#include "kvpop_mma.cuh"
#include "kvpop_ptx.cuh"
#include "kvpop_tc05.cuh"

namespace kvpop {
namespace {

constexpr float kLog2e = 1.4426950408889634f;
constexpr float kLn2f = 0.69314718055994530942f;

struct TargetArgs {
  const void* Q;             // [n][H*G][S][d]
  const void* K;             // [n][H][S][d]
  const float* lse;          // [n][H*G][S] natural log
  const int32_t* len;        // [n] or nullptr
  float* logm;               // [n][H*G][S] out
  int H, G, S, w, la;
  float kscale;              // log2(e) / sqrt(d)
  int32_t* err;              // first-error word or nullptr
};

__device__ __forceinline__ int row_len(const TargetArgs& a, int seq) {
  return a.len ? max(0, min(a.len[seq], a.S)) : a.S;
}

// last query position that may attend to key t (-1 if none)
__device__ __forceinline__ int future_hi(int t, int L, int w, int la) {
  const int hi = la > 0 ? min(L - 1, t + w + la) : L - 1;
  return t + w <= hi ? hi : -1;
}

// ---------------------------------------------------------------- fp32 kernel
// One CTA: 64 keys of one (sequence, KV head) against one query head, the queries streamed in
// blocks of 128 through a cp.async double buffer.  A thread holds 4 keys x 8 queries (keys
// ty + 16 i, queries tx + 16 j), so 4 dimensions cost 12 16-byte shared loads for 128 FMAs;
// rows are padded by 4 floats, which makes those loads conflict-free.  Each thread keeps the
// running (max, sum) of its own columns and the 16 threads of a key merge once at the end.
// Bound by FP32 FMA.  16 (pair, head) rows of 2039 tokens, d = 64: 171 us, against
// 10982 us with one warp per (key, head), where each lane walked a query row of its own and
// every load touched 32 lines.
constexpr int TF_NT = 256;
constexpr int TF_BK = 64;
constexpr int TF_BQ = 128;

template <int HD>
struct TfP {
  static constexpr int RS = HD + 4;              // padded row
  static constexpr int OFF_Q = TF_BK * RS;       // floats: K tile, then two query blocks
  static constexpr int OFF_L = OFF_Q + 2 * TF_BQ * RS;
  static constexpr size_t SMEM = (size_t)(OFF_L + 2 * TF_BQ) * 4;
};

template <int HD>
__global__ void __launch_bounds__(TF_NT) target_f32_kernel(TargetArgs a) {
  using P = TfP<HD>;
  extern __shared__ __align__(16) float sm_tf[];
  float* Ks = sm_tf;
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const int pair = blockIdx.y, seq = pair / a.H, h = pair - seq * a.H;
  const int S = a.S, L = row_len(a, seq), w = a.w, la = a.la;
  const int t0 = blockIdx.x * TF_BK;
  if (t0 >= L) return;
  const int t1 = min(t0 + TF_BK - 1, L - 1);
  const size_t qrow = (size_t)seq * a.H * a.G + (size_t)h * a.G + blockIdx.z;
  float* out = a.logm + qrow * S;
  const int d_lo = t0 + w;
  const int d_hi = la > 0 ? min(L - 1, t1 + w + la) : L - 1;
  if (d_lo > d_hi) {                             // no key of the tile has a future query
    if (tid <= t1 - t0) out[t0 + tid] = -INFINITY;
    return;
  }
  const float* Kp = static_cast<const float*>(a.K) + ((size_t)pair * S + t0) * HD;
  const float* Qg = static_cast<const float*>(a.Q) + qrow * S * HD;
  const float* lse = a.lse + qrow * S;
  const int nblk = (d_hi - d_lo + TF_BQ) / TF_BQ;
  auto issue = [&](int b, int st) {
    const int d0 = d_lo + b * TF_BQ;
    const uint32_t dst = smem_u32(sm_tf + P::OFF_Q + st * TF_BQ * P::RS);
    for (int i = tid; i < TF_BQ * (HD / 4); i += TF_NT) {
      const int r = i / (HD / 4), c = i - r * (HD / 4);
      const bool ok = d0 + r <= d_hi;
      cp_async16(dst + (r * P::RS + 4 * c) * 4, Qg + (size_t)(ok ? d0 + r : d0) * HD + 4 * c, ok ? 16 : 0);
    }
    if (tid < TF_BQ)
      sm_tf[P::OFF_L + st * TF_BQ + tid] = d0 + tid <= d_hi ? lse[d0 + tid] * kLog2e : 0.f;
  };
  issue(0, 0);
  cp_commit();
  for (int i = tid; i < TF_BK * (HD / 4); i += TF_NT) {
    const int r = i / (HD / 4), c = i - r * (HD / 4);
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (t0 + r <= t1) v = *reinterpret_cast<const float4*>(Kp + (size_t)r * HD + 4 * c);
    v.x *= a.kscale; v.y *= a.kscale; v.z *= a.kscale; v.w *= a.kscale;
    *reinterpret_cast<float4*>(Ks + r * P::RS + 4 * c) = v;
  }
  float m[4], l[4];
  int hi[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    m[i] = -INFINITY;
    l[i] = 0.f;
    const int t = t0 + ty + 16 * i;
    hi[i] = t <= t1 ? future_hi(t, L, w, la) : -1;
  }
  for (int b = 0; b < nblk; ++b) {
    const int st = b & 1, d0 = d_lo + b * TF_BQ;
    if (b + 1 < nblk) issue(b + 1, st ^ 1);
    cp_commit();
    cp_wait<1>();
    __syncthreads();
    const float* Qs = sm_tf + P::OFF_Q + st * TF_BQ * P::RS;
    float acc[4][8];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 8; ++j) acc[i][j] = 0.f;
#pragma unroll 4
    for (int c = 0; c < HD; c += 4) {
      float4 kf[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) kf[i] = *reinterpret_cast<const float4*>(Ks + (ty + 16 * i) * P::RS + c);
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const float4 q = *reinterpret_cast<const float4*>(Qs + (tx + 16 * j) * P::RS + c);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          acc[i][j] = fmaf(kf[i].x, q.x, acc[i][j]);
          acc[i][j] = fmaf(kf[i].y, q.y, acc[i][j]);
          acc[i][j] = fmaf(kf[i].z, q.z, acc[i][j]);
          acc[i][j] = fmaf(kf[i].w, q.w, acc[i][j]);
        }
      }
    }
    float nl[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) nl[j] = sm_tf[P::OFF_L + st * TF_BQ + tx + 16 * j];
    const bool masked = d0 < t1 + w || d0 + TF_BQ - 1 > d_hi || (la > 0 && d0 + TF_BQ - 1 > t0 + w + la);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int t = t0 + ty + 16 * i;
      float mx = m[i];
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        float v = acc[i][j] - nl[j];
        if (masked) {
          const int d = d0 + tx + 16 * j;
          if (d < t + w || d > hi[i]) v = -INFINITY;
        }
        acc[i][j] = v;
        mx = fmaxf(mx, v);
      }
      const float u = mx == -INFINITY ? 0.f : mx;
      float sum = 0.f;
#pragma unroll
      for (int j = 0; j < 8; ++j) sum += exp2f(acc[i][j] - u);
      l[i] = l[i] * exp2f(m[i] - u) + sum;
      m[i] = mx;
    }
    __syncthreads();
  }
  cp_wait<0>();
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    float M = m[i];
#pragma unroll
    for (int o = 1; o < 16; o <<= 1) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, o));
    float s = M == -INFINITY ? 0.f : l[i] * exp2f(m[i] - M);
#pragma unroll
    for (int o = 1; o < 16; o <<= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    const int t = t0 + ty + 16 * i;
    if (tx == 0 && t <= t1) out[t] = s > 0.f ? (M + log2f(s)) * kLn2f : -INFINITY;
  }
}

template <int HD>
cudaError_t launch_target_f32(const TargetArgs& a, int n_pairs, cudaStream_t stream) {
  cudaError_t e = raise_smem_limit(target_f32_kernel<HD>, TfP<HD>::SMEM);
  if (e != cudaSuccess) return e;
  target_f32_kernel<HD><<<dim3((a.S + TF_BK - 1) / TF_BK, n_pairs, a.G), TF_NT, TfP<HD>::SMEM, stream>>>(a);
  return cudaGetLastError();
}

// ---------------------------------------------------------------- tensor-core kernel
template <int HD>
struct TgP {
  static constexpr int NW = 8;
  static constexpr int THREADS = NW * 32;
  static constexpr int ROWS = 16 * NW;             // keys per CTA
  static constexpr int BN = 64;                    // queries per block
  static constexpr int NKS = HD / 16;
  static constexpr int NNT = BN / 8;
  static constexpr int CH = HD / 8;
  static constexpr int ROWB = HD * 2;
  static constexpr int QB = BN * ROWB;
  static constexpr int STAGES = 2;
  static constexpr int OFF_LSE = STAGES * QB;
  static constexpr int SMEM = OFF_LSE + STAGES * BN * 4;
  static_assert(ROWS * ROWB <= STAGES * QB, "the key tile is staged in the query buffers");
};

template <int HD>
__global__ void __launch_bounds__(TgP<HD>::THREADS, 1) target_tc_kernel(TargetArgs a) {
  using P = TgP<HD>;
  extern __shared__ __align__(1024) unsigned char smem_tg[];
  float* lseS = reinterpret_cast<float*>(smem_tg + P::OFF_LSE);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int pair = blockIdx.y, seq = pair / a.H, h = pair - seq * a.H;
  const int G = a.G, S = a.S, L = row_len(a, seq), w = a.w, la = a.la;
  const int t0 = blockIdx.x * P::ROWS;
  if (t0 >= L) return;
  const int t1 = min(t0 + P::ROWS - 1, L - 1);
  const size_t qrow0 = (size_t)seq * a.H * G + (size_t)h * G;
  const int d_lo = t0 + w;
  const int d_hi = la > 0 ? min(L - 1, t1 + w + la) : L - 1;
  const int ra = 16 * warp + (lane >> 2), rb = ra + 8;
  const int ta = t0 + ra, tb = t0 + rb;
  if (d_lo > d_hi) {                               // no key of the tile has a future query
    for (int i = tid; i < (t1 - t0 + 1) * G; i += P::THREADS) {
      const int tl = i / G, g = i - tl * G;
      a.logm[(qrow0 + g) * S + t0 + tl] = -INFINITY;
    }
    return;
  }
  const int nblk = (d_hi - d_lo + P::BN) / P::BN;
  const int total = G * nblk;
  const uint32_t sbase = (uint32_t)__cvta_generic_to_shared(smem_tg);
  const bf16* Kp = static_cast<const bf16*>(a.K) + (size_t)pair * S * HD;

  // key tile -> query buffers (rows past the sequence zero-filled) -> A fragments
  for (int i = tid; i < P::ROWS * P::CH; i += P::THREADS) {
    const int r = i / P::CH, c = i - r * P::CH;
    const bool ok = t0 + r <= t1;
    cp_async16(sbase + swz(r, c, P::ROWB), Kp + (size_t)(ok ? t0 + r : t0) * HD + c * 8, ok ? 16 : 0);
  }
  cp_commit();
  cp_wait<0>();
  __syncthreads();
  uint32_t kf[P::NKS][4];
#pragma unroll
  for (int ks = 0; ks < P::NKS; ++ks) {
    const int r = 16 * warp + ((lane >> 3) & 1) * 8 + (lane & 7);
    const int c = 2 * ks + (lane >> 4);
    ldsm_x4(sbase + swz(r, c, P::ROWB), kf[ks][0], kf[ks][1], kf[ks][2], kf[ks][3]);
  }
  __syncthreads();

  auto issue = [&](int j, int st) {
    const int g = j / nblk, b = j - g * nblk;
    const int d0 = d_lo + b * P::BN;
    const bf16* Qg = static_cast<const bf16*>(a.Q) + (qrow0 + g) * S * HD;
    const uint32_t dst = sbase + st * P::QB;
    for (int i = tid; i < P::BN * P::CH; i += P::THREADS) {
      const int r = i / P::CH, c = i - r * P::CH;
      const bool ok = d0 + r <= d_hi;
      cp_async16(dst + swz(r, c, P::ROWB), Qg + (size_t)(ok ? d0 + r : d0) * HD + c * 8, ok ? 16 : 0);
    }
    if (tid < P::BN) {
      const float* lse = a.lse + (qrow0 + g) * S;
      if (d0 + tid <= d_hi)
        cp_async4(sbase + P::OFF_LSE + (st * P::BN + tid) * 4, lse + d0 + tid);
      else
        lseS[st * P::BN + tid] = 0.f;
    }
  };

  const int hia = future_hi(ta, L, w, la), hib = future_hi(tb, L, w, la);
  float ma = -INFINITY, mb = -INFINITY, la_ = 0.f, lb_ = 0.f;
  issue(0, 0);
  cp_commit();
  if (total > 1) issue(1, 1);
  cp_commit();
  for (int j = 0; j < total; ++j) {
    const int st = j & 1;
    const int g = j / nblk, b = j - g * nblk;
    const int d0 = d_lo + b * P::BN;
    cp_wait<1>();
    __syncthreads();
    const uint32_t qb = sbase + st * P::QB;
    float sc[P::NNT][4];
#pragma unroll
    for (int n = 0; n < P::NNT; ++n) sc[n][0] = sc[n][1] = sc[n][2] = sc[n][3] = 0.f;
#pragma unroll
    for (int ks = 0; ks < P::NKS; ++ks) {
#pragma unroll
      for (int np = 0; np < P::NNT / 2; ++np) {
        const int r = 8 * (2 * np + (lane >> 4)) + (lane & 7);
        const int c = 2 * ks + ((lane >> 3) & 1);
        uint32_t b0, b1, b2, b3;
        ldsm_x4(qb + swz(r, c, P::ROWB), b0, b1, b2, b3);
        mma_bf16(sc[2 * np], kf[ks][0], kf[ks][1], kf[ks][2], kf[ks][3], b0, b1);
        mma_bf16(sc[2 * np + 1], kf[ks][0], kf[ks][1], kf[ks][2], kf[ks][3], b2, b3);
      }
    }
    // rows need a mask where the block reaches below t + w, past t + w + L, or past the end
    const bool masked = d0 < t1 + w || d0 + P::BN - 1 > d_hi || (la > 0 && d0 + P::BN - 1 > t0 + w + la);
    float mxa = -INFINITY, mxb = -INFINITY;
#pragma unroll
    for (int n = 0; n < P::NNT; ++n) {
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const int col = n * 8 + 2 * (lane & 3) + (c & 1);
        const int d = d0 + col;
        float v = sc[n][c] * a.kscale - lseS[st * P::BN + col] * kLog2e;
        if (masked) {
          const int t = c < 2 ? ta : tb;
          const int hi = c < 2 ? hia : hib;
          if (d < t + w || d > hi) v = -INFINITY;
        }
        sc[n][c] = v;
      }
      mxa = fmaxf(mxa, fmaxf(sc[n][0], sc[n][1]));
      mxb = fmaxf(mxb, fmaxf(sc[n][2], sc[n][3]));
    }
#pragma unroll
    for (int o = 1; o <= 2; o <<= 1) {
      mxa = fmaxf(mxa, __shfl_xor_sync(0xffffffffu, mxa, o));
      mxb = fmaxf(mxb, __shfl_xor_sync(0xffffffffu, mxb, o));
    }
    const float mna = fmaxf(ma, mxa), mnb = fmaxf(mb, mxb);
    const float ua = mna == -INFINITY ? 0.f : mna, ub = mnb == -INFINITY ? 0.f : mnb;
    float sa = 0.f, sb = 0.f;
#pragma unroll
    for (int n = 0; n < P::NNT; ++n) {
      sa += ex2(sc[n][0] - ua) + ex2(sc[n][1] - ua);
      sb += ex2(sc[n][2] - ub) + ex2(sc[n][3] - ub);
    }
    la_ = la_ * ex2(ma - ua) + sa;
    lb_ = lb_ * ex2(mb - ub) + sb;
    ma = mna;
    mb = mnb;
    if (b == nblk - 1) {                           // head g done: write and reset
      float sa2 = la_, sb2 = lb_;
#pragma unroll
      for (int o = 1; o <= 2; o <<= 1) {
        sa2 += __shfl_xor_sync(0xffffffffu, sa2, o);
        sb2 += __shfl_xor_sync(0xffffffffu, sb2, o);
      }
      if ((lane & 3) == 0) {
        float* out = a.logm + (qrow0 + g) * S;
        if (ta <= t1) out[ta] = sa2 > 0.f ? (ma + __log2f(sa2)) * kLn2f : -INFINITY;
        if (tb <= t1) out[tb] = sb2 > 0.f ? (mb + __log2f(sb2)) * kLn2f : -INFINITY;
      }
      ma = mb = -INFINITY;
      la_ = lb_ = 0.f;
    }
    __syncthreads();
    if (j + 2 < total) issue(j + 2, st);
    cp_commit();
  }
  cp_wait<0>();
}

// ---------------------------------------------------------------- tcgen05 kernel (d = 128)
// Log-sum-exp of rows against streamed columns, S = A B^T, in two uses:
//  * FUTURE (transposed pass): rows are 256 keys of one (sequence, KV head); for each query
//    head its rows q >= t0 + w are streamed, with -log2(e) LSE_d added per column;
//  * causal normalisers (App. D.1): rows are the 256 (head, query) pairs of 256 / G queries, the
//    keys 0 .. q1 are streamed once for all of them.
// The rows sit in tensor memory as the MMA's A operand; the streamed operand comes by TMA
// (128-byte swizzle; rows past the sequence read as zeros).  One warp issues the MMAs (M = 128,
// N = 128), the tiles (block, 128-row half) taking three S buffers in turn; 16 softmax warps take
// 32 rows x 64 columns of every block apiece.  A 256 x 128 block needs 1024 clocks of the tensor
// unit (64 per MMA) and 1024 of the exponential unit (32 per clock); the softmax warps' code sets
// the pace, about 1500 clocks (causal) and 2000 (future, which also reads a normaliser per
// column).  What paid: barriers arrived at once per warp, a warp's whole part in registers
// before its exponentials (the S buffer is free at once), the MMA warp's operands kept
// warp-uniform (see elect_one; 945 -> 815 us), and the row operand loaded as whole lines before the
// set-up (798 -> 778 us; 16 x 8 heads of 256 tokens 35.0 -> 26.8, of 1024 158 -> 134).  8 heads x
// 16384 tokens, 4 query heads each: causal 778 us, against 1354 with 64-key blocks in the prompt
// kernel; future 984 us, against 1363 with copies by cp.async, one arrival per thread and the rows
// in shared memory.  Measured and not kept: a cluster of two CTAs sharing the streamed blocks by
// multicast (843 / 1075 us); column halves past the last streamed one left out (2% slower from 1500
// tokens on).
// Blocks: longest tiles first over all pairs (tiles of one pair after the other left the last
// pair's longest tile to the end).
constexpr int T6_HALF = 128;
constexpr int T6_ROWS = 2 * T6_HALF;            // rows per CTA
constexpr int T6_BN = 128;                      // columns per block (MMA N)
constexpr int T6_ST = 6;                        // column-block stages
constexpr int T6_SOFT = 16;                     // warps 0-15 softmax, 16 MMA, 17 copies
constexpr int T6_MMA_WARP = T6_SOFT;
constexpr int T6_THREADS = 32 * (T6_SOFT + 2);
constexpr int T6_QB = T6_BN * 256;              // column block, bytes
constexpr int T6_OFF_LSE = T6_ST * T6_QB;
constexpr int T6_OFF_BAR = T6_OFF_LSE + T6_ST * T6_BN * 4;
constexpr int T6_OFF_TMEM = T6_OFF_BAR + 8 * 32;
constexpr int T6_OFF_PX = T6_OFF_TMEM + 16;      // [query head][2 halves][128 rows][m, l, done, -]
constexpr int T6_MAX_G = 4;                      // query heads per KV head
constexpr int T6_SMEM = T6_OFF_PX + T6_MAX_G * 2 * T6_HALF * 16 + 1024;   // 1024: swizzle atom alignment
constexpr int T6_FULL = 0, T6_EMPTY = T6_ST, T6_SFULL = 2 * T6_ST, T6_PFULL = 2 * T6_ST + 3,
              T6_AFULL = 2 * T6_ST + 6;
// tensor memory: the row tiles of the two halves (64 columns each, two bf16 per word), then
// three S buffers that the tiles (block, half) take in turn
constexpr int T6_TM_S = 128;
enum : int { T6ERR_WAIT = 22 };

struct LseArgs {
  const bf16* A;             // row operand: keys (FUTURE) or queries, [heads][S][128]
  const float* lse;          // FUTURE: [n][H*G][S] natural log
  const int32_t* len;        // [n] or nullptr
  float* out;                // [n][H*G][S]
  int n_pairs, H, S, w, la;
  float scale;               // log2(e) / sqrt(d)
  int32_t* err;
};

__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap* map, int x, int y, int z,
                                            uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z), "r"(bar)
      : "memory");
}

// map: boxes of 64 columns x 128 rows of the streamed operand, [heads][S][128].
template <int G, bool FUTURE>
__global__ void __launch_bounds__(T6_THREADS, 1)
    lse_t5_kernel(const __grid_constant__ CUtensorMap map, LseArgs a) {
  using namespace tc05;
  constexpr int NQ = FUTURE ? T6_ROWS : T6_ROWS / G;      // positions of a tile
  extern __shared__ unsigned char sm6_raw[];
  unsigned char* sm6 = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(sm6_raw) + 1023) & ~(uintptr_t)1023);
  const uint32_t sb = smem_u32(sm6);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int tile = blockIdx.x / a.n_pairs, pair = blockIdx.x - tile * a.n_pairs;
  const int seq = pair / a.H, h0 = pair - seq * a.H;
  const int S = a.S, L = a.len ? max(0, min(a.len[seq], S)) : S, w = a.w, la = a.la;
  // longest first: the future of early keys, the past of late queries
  const int t0 = (FUTURE ? tile : (S + NQ - 1) / NQ - 1 - tile) * NQ;
  if (t0 >= L) return;
  const int t1 = min(t0 + NQ - 1, L - 1);
  const int qrow0 = seq * a.H * G + h0 * G;
  // streamed columns d_lo .. d_hi, once (causal) or per query head (FUTURE)
  const int d_lo = FUTURE ? t0 + w : 0;
  const int d_hi = !FUTURE ? t1 : la > 0 ? min(L - 1, t1 + w + la) : L - 1;
  if (FUTURE && d_lo > d_hi) {                     // no key of the tile has a future query
    for (int i = tid; i < (t1 - t0 + 1) * G; i += T6_THREADS) {
      const int tl = i / G, g = i - tl * G;
      a.out[(size_t)(qrow0 + g) * S + t0 + tl] = -INFINITY;
    }
    return;
  }
  const int nblk = (d_hi - d_lo + T6_BN) / T6_BN;
  const int total = FUTURE ? G * nblk : nblk;
  // Rows of the A operand on their way while barriers and tensor memory are set up: warps 0-3 and
  // 4-7 take 32 rows of a half each, four lanes 64 bytes of a row at a time (see below).
  float4 x[16];                                    // piece lane % 4 of rows 8 (i % 4) + lane / 4
  if (warp < T6_SOFT / 2) {
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      const int rr = warp * 32 + 8 * (i & 3) + (lane >> 2);
      const int tt = t0 + (FUTURE ? rr : rr % NQ);
      const bf16* src = a.A + ((size_t)(FUTURE ? pair : qrow0 + rr / NQ) * S + (tt <= t1 ? tt : t0)) * 128;
      x[i] = __ldg(reinterpret_cast<const float4*>(src) + 4 * (i >> 2) + (lane & 3));
      if (tt > t1) x[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
  }
  auto bar = [&](int i) { return sb + T6_OFF_BAR + 8u * (uint32_t)i; };
  if (tid == 0) {
    for (int i = 0; i < T6_ST; ++i) {
      mbar_init(bar(T6_FULL + i), FUTURE ? 2 : 1);         // the copies, and the normalisers' warp
      mbar_init(bar(T6_EMPTY + i), FUTURE ? 1 + T6_SOFT : 1);   // MMA commit, normalisers read
    }
    for (int i = 0; i < 3; ++i) {
      mbar_init(bar(T6_SFULL + i), 1);
      mbar_init(bar(T6_PFULL + i), T6_SOFT / 2);
    }
    mbar_init(bar(T6_AFULL), T6_SOFT / 2);
    mbar_fence_init();
  }
  static_assert(G <= T6_MAX_G, "one slot per head");
  if (warp == T6_MMA_WARP) tmem_alloc(sb + T6_OFF_TMEM, 512);
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = *reinterpret_cast<volatile uint32_t*>(sm6 + T6_OFF_TMEM);
  if (warp == T6_MMA_WARP + 1) {
    // ---------------------------------------------------------------- copies
    int j = 0;
    for (; j < total; ++j) {
      const int st = j % T6_ST;
      const bool ok = j < T6_ST || mbar_wait(bar(T6_EMPTY + st), ((j / T6_ST) - 1) & 1, a.err, T6ERR_WAIT);
      if (!__all_sync(0xffffffffu, ok)) break;
      const int g = FUTURE ? j / nblk : 0, d0 = d_lo + (j - g * nblk) * T6_BN;
      if (lane == 0) {
        const uint32_t qd = sb + st * T6_QB;
        const int z = FUTURE ? qrow0 + g : pair;
        mbar_arrive_expect_tx(bar(T6_FULL + st), T6_QB);
        tma_load_3d(qd, &map, 0, d0, z, bar(T6_FULL + st));
        tma_load_3d(qd + T6_BN * 128, &map, 64, d0, z, bar(T6_FULL + st));
      }
      if (FUTURE) {
        // the block's normalisers, stored once as -log2(e) LSE_d
        float* nls = reinterpret_cast<float*>(sm6 + T6_OFF_LSE) + st * T6_BN;
        const float* lse = a.lse + (size_t)(qrow0 + g) * S;
        float v[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) v[i] = __ldg(lse + min(d0 + lane + 32 * i, d_hi));
#pragma unroll
        for (int i = 0; i < 4; ++i) nls[lane + 32 * i] = -kLog2e * v[i];
        __syncwarp();
        if (lane == 0) mbar_arrive(bar(T6_FULL + st));
      }
    }
    // every copy has landed before the CTA ends (the waiting roles may have given up)
    if (lane == 0)
      for (int k = max(0, j - T6_ST); k < j; ++k)
        mbar_wait(bar(T6_FULL + k % T6_ST), (k / T6_ST) & 1, a.err, T6ERR_WAIT);
    __syncwarp();
  } else if (warp == T6_MMA_WARP) {
    // ---------------------------------------------------------------- MMA issue
    const uint32_t idS = idesc_bf16(128, T6_BN, 0);
    const bool lead = elect_one();
    const uint64_t bd0 = kmajor_desc(sb, T6_BN, 0);
    bool ok = mbar_wait(bar(T6_AFULL), 0, a.err, T6ERR_WAIT);
    int sbuf = 0;                                   // S buffer of the tile and its use so far
    uint32_t use = 0;
    for (int j = 0; j < total; ++j) {
      const int st = j % T6_ST;
      ok = ok && mbar_wait(bar(T6_FULL + st), (j / T6_ST) & 1, a.err, T6ERR_WAIT);
      if (!__all_sync(0xffffffffu, ok)) break;
      fence_after();
      const uint64_t bd = desc_at(bd0, st * T6_QB);
#pragma unroll
      for (int hh = 0; hh < 2; ++hh) {
        // the warps of the buffer's last tile must have it in registers
        if (use > 0) ok = ok && mbar_wait(bar(T6_PFULL + sbuf), (use - 1) & 1, a.err, T6ERR_WAIT);
        if (!__all_sync(0xffffffffu, ok)) break;
        fence_after();
        if (lead) {
          const uint32_t dS = tmem + T6_TM_S + (uint32_t)sbuf * T6_BN;
#pragma unroll
          for (int ks = 0; ks < 8; ++ks)
            mma_bf16_ts(dS, tmem + hh * 64 + ks * 8, kmajor_step(bd, T6_BN, ks), idS, ks > 0);
          commit(bar(T6_SFULL + sbuf));
          if (hh == 1) commit(bar(T6_EMPTY + st));
        }
        __syncwarp();
        if (++sbuf == 3) {
          sbuf = 0;
          ++use;
        }
      }
    }
    // every MMA has completed (the last stage's release) before the CTA ends
    if (__all_sync(0xffffffffu, ok) && total > 0)
      mbar_wait(bar(T6_EMPTY + (total - 1) % T6_ST), ((total - 1) / T6_ST) & 1, a.err, T6ERR_WAIT);
    __syncwarp();
  } else {
    // ---------------------------------------------------------------- softmax rows
    // warp w: half hh = (w / 4) mod 2 of the CTA's rows, row r = 32 (w mod 4) + lane (the warp's
    // tensor-memory lane quarter), and columns [64 cs, 64 cs + 64) of every block with cs = w / 8:
    // four warps per subpartition share the exponentials of a block.  The two column halves of
    // a row keep their own (max, sum) over a head's blocks and meet at its end in shared memory.
    const int hh = (warp >> 2) & 1, cs = warp >> 3;
    const int r = (warp & 3) * 32 + lane, ra = hh * T6_HALF + r;
    const int t = t0 + (FUTURE ? ra : ra % NQ);            // the row's position
    const int lo = FUTURE ? t + w : 0;                     // columns the row takes: lo .. hi
    const int hi = t > t1 ? -1 : FUTURE ? future_hi(t, L, w, la) : t;
    const uint32_t tl = tmem + ((uint32_t)((warp & 3) * 32) << 16);
    const uint32_t tS = tl + T6_TM_S + 64 * cs;
    const float* nlS = reinterpret_cast<const float*>(sm6 + T6_OFF_LSE) + 64 * cs;   // -log2(e) LSE_d
    float* pxs = reinterpret_cast<float*>(sm6 + T6_OFF_PX);
    const uint64_t cc = f2_pack(a.scale, a.scale);
    if (cs == 0) {
      // The warp's 32 rows into tensor memory as the MMA's A operand (zeros past the tile): the
      // pieces change lanes in the warp's part of the exchange slots (loaded a row per lane, each
      // load would touch 32 lines: 2 us of a CTA).
      auto at = [&](int row, int c) {               // 16-byte piece c of a row's 64 bytes
        return reinterpret_cast<float4*>(pxs) + (c * 2 + hh) * T6_HALF + (warp & 3) * 32 + (row ^ (2 * c));
      };
#pragma unroll
      for (int h = 0; h < 4; ++h) {
        float v[16];
#pragma unroll
        for (int k = 0; k < 4; ++k) *at(8 * k + (lane >> 2), lane & 3) = x[4 * h + k];
        __syncwarp();
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const float4 y = *at(lane, k);
          v[4 * k] = y.x; v[4 * k + 1] = y.y; v[4 * k + 2] = y.z; v[4 * k + 3] = y.w;
        }
        __syncwarp();
        tmem_st16(tl + hh * 64 + h * 16, v);
      }
      // the rows' exchange slots start with no head done (read after S, and so after all of this)
#pragma unroll
      for (int g = 0; g < G; ++g) reinterpret_cast<int*>(pxs)[4 * ((g * 2 + hh) * T6_HALF + r) + 2] = 0;
      tmem_wait_st();
      fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(bar(T6_AFULL));
    }
    float m = -INFINITY, l = 0.f;
    int g = 0, b = 0;
    int sbuf = hh;                                   // S buffer of tile 2 j + hh, its phase
    uint32_t ph = 0;
    for (int j = 0; j < total; ++j) {
      const int st = j % T6_ST;
      const int e0 = d_lo + b * T6_BN + 64 * cs;
      bool ok = mbar_wait(bar(T6_SFULL + sbuf), ph, a.err, T6ERR_WAIT);
      // the stage's normalisers (complete long before S; the wait orders their reads)
      if (FUTURE) ok = ok && mbar_wait(bar(T6_FULL + st), (j / T6_ST) & 1, a.err, T6ERR_WAIT);
      if (!__all_sync(0xffffffffu, ok)) break;
      fence_after();
      float s[2][32];
      tmem_ld32(tS + sbuf * T6_BN, s[0]);
      tmem_ld32(tS + sbuf * T6_BN + 32, s[1]);
      tmem_wait_ld();
      // the warp's part of the S buffer is in registers: the MMA may overwrite it
      fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(bar(T6_PFULL + sbuf));
      sbuf += 2;
      if (sbuf >= 3) {
        sbuf -= 3;
        ph ^= 1;
      }
      // some row of the tile ends (or begins) inside these columns
      const bool masked = FUTURE ? (e0 < t1 + w || e0 + 63 > d_hi || (la > 0 && e0 + 63 > t0 + w + la))
                                 : e0 + 63 > t0;
      if (masked) {                                 // on the raw logits: -inf c2 + n = -inf
#pragma unroll
        for (int c = 0; c < 2; ++c)
#pragma unroll
          for (int i = 0; i < 32; ++i) {
            const int d = e0 + 32 * c + i;
            if (d < lo || d > hi) s[c][i] = -INFINITY;
          }
      }
      // FUTURE: x = s c2 - log2(e) LSE_d is the query's log2 attention probability of the key, so
      // 2^x needs no running maximum unless the key lies outside the query's kept set with a much
      // larger logit: sum with base 0.  Causal: x = s c2 - m with the first part's maximum as
      // the base.  The maximum is taken only when a part's sum leaves [2^-60, 2^60] (overflow,
      // NaN, or every term tiny or masked); causal, [2^-60, 2^8]: an exponent is formed in fp32 and
      // so is off by up to its size times 2^-24.  Mean error from 64 bits of 8 heads x 16384
      // tokens with outlier channels 7.7e-7 (2^60: 7.9e-7; a base moved at 2^8 of one logit, as in
      // the prompt kernel: 7.7e-7), where the first keys' logits lie 32 below the others' 8.0e-7
      // (1.8e-6; 8.0e-7), for 4 us in 798.
      constexpr float kMaxSum = FUTURE ? 0x1p60f : 0x1p8f;
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        const float nb1 = FUTURE || m == -INFINITY ? 0.f : -m;
        const uint64_t nb = f2_pack(nb1, nb1);
        uint64_t ps[4] = {0ull, 0ull, 0ull, 0ull};
        float* sc = s[c];
#pragma unroll
        for (int i4 = 0; i4 < 8; ++i4) {
          uint64_t n0 = nb, n1 = nb;
          if (FUTURE) {
            const float4 v = reinterpret_cast<const float4*>(nlS + st * T6_BN + 32 * c)[i4];
            n0 = f2_pack(v.x, v.y);
            n1 = f2_pack(v.z, v.w);
          }
          f2_unpack(f2_fma(f2_pack(sc[4 * i4], sc[4 * i4 + 1]), cc, n0), sc[4 * i4], sc[4 * i4 + 1]);
          f2_unpack(f2_fma(f2_pack(sc[4 * i4 + 2], sc[4 * i4 + 3]), cc, n1), sc[4 * i4 + 2], sc[4 * i4 + 3]);
          const int k = (2 * i4) & 3;
          ps[k] = f2_add(ps[k], f2_pack(ex2(sc[4 * i4]), ex2(sc[4 * i4 + 1])));
          ps[k + 1] = f2_add(ps[k + 1], f2_pack(ex2(sc[4 * i4 + 2]), ex2(sc[4 * i4 + 3])));
        }
        if (FUTURE && c == 1) {                    // the warp is done with the stage's normalisers
          __syncwarp();
          if (lane == 0) mbar_arrive(bar(T6_EMPTY + st));
        }
        const uint64_t p2 = f2_add(f2_add(ps[0], ps[1]), f2_add(ps[2], ps[3]));
        float q0, q1;
        f2_unpack(p2, q0, q1);
        const float sum = q0 + q1;
        if (sum >= 0x1p-60f && sum <= kMaxSum && (FUTURE || m != -INFINITY)) {
          if (!FUTURE) {
            l += sum;
          } else if (m <= 0.f) {                    // new base 0
            l = (m == 0.f ? l : l * ex2(m)) + sum;
            m = 0.f;
          } else {
            l = fmaf(sum, ex2(-m), l);
          }
          continue;
        }
        // part maximum: 8 chains of three-input maxima
        float pm[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) pm[k] = fmax3(sc[k], sc[8 + k], sc[16 + k]);
#pragma unroll
        for (int k = 0; k < 8; ++k) pm[k] = fmaxf(pm[k], sc[24 + k]);
        // the values in sc are relative to -nb1
        const float mx = fmax3(fmax3(pm[0], pm[1], pm[2]), fmax3(pm[3], pm[4], pm[5]), fmaxf(pm[6], pm[7]));
        const float mn = fmaxf(m, mx - nb1);
        const float base = mn == -INFINITY ? 0.f : mn + nb1;
        float part = 0.f;
#pragma unroll
        for (int i = 0; i < 32; ++i) part += ex2(sc[i] - base);
        l = l * ex2(m - (mn == -INFINITY ? 0.f : mn)) + part;
        m = mn;
      }
      if (++b == nblk) {
        // head g done: the upper column half hands its (max, sum) to the lower, which merges
        // and writes the row's result.  Every head has a slot of its own: the upper half may be
        // heads ahead (it needs the lower one only to have loaded its logits).  (The mask changes
        // no index; with the range known the loop's code is 3% faster: 1016 -> 984 us.)
        volatile float* px = pxs + (((size_t)(g & (T6_MAX_G - 1)) * 2 + hh) * T6_HALF + r) * 4;
        volatile int* done = reinterpret_cast<volatile int*>(px) + 2;
        if (cs == 1) {
          px[0] = m;
          px[1] = l;
          __threadfence_block();
          *done = 1;
        } else {
          bool ready = *done != 0;
          if (!ready) {
            const unsigned long long tw = globaltimer();
            while (!(ready = *done != 0))
              if (globaltimer() - tw > kWaitLimitNs) { atomicCAS(a.err, 0, T6ERR_WAIT); break; }
          }
          __threadfence_block();
          const float m1 = px[0], l1 = px[1];
          const float M = fmaxf(m, m1);
          float Lr = 0.f;
          if (M != -INFINITY)
            Lr = (m == -INFINITY ? 0.f : l * ex2(m - M)) + (m1 == -INFINITY ? 0.f : l1 * ex2(m1 - M));
          const int head = FUTURE ? g : ra / NQ;
          if (t <= t1)
            a.out[(size_t)(qrow0 + head) * S + t] = Lr > 0.f ? (M + __log2f(Lr)) * kLn2f : -INFINITY;
        }
        m = -INFINITY;
        l = 0.f;
        ++g;
        b = 0;
      }
    }
  }
  fence_before();
  __syncthreads();
  if (warp == T6_MMA_WARP) tmem_dealloc(tmem, 512);
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*,
                                  const cuuint64_t*, const cuuint64_t*, const cuuint32_t*,
                                  const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// [heads][S][128] bf16, boxes of 64 columns x `rows` rows of one head
cudaError_t encode_heads(CUtensorMap* map, const void* base, long long heads, int S, int rows) {
  static const EncodeTiledFn fn = [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) !=
            cudaSuccess || q != cudaDriverEntryPointSuccess)
      p = nullptr;
    return reinterpret_cast<EncodeTiledFn>(p);
  }();
  if (!fn) return cudaErrorNotSupported;
  cuuint64_t dims[3] = {128, (cuuint64_t)S, (cuuint64_t)heads};
  cuuint64_t strides[2] = {256, (cuuint64_t)S * 256};
  cuuint32_t box[3] = {64, (cuuint32_t)rows, 1};
  cuuint32_t estr[3] = {1, 1, 1};
  const CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box, estr,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                        CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

template <int G, bool FUTURE>
cudaError_t launch_lse_t5(const void* Q, const void* K, LseArgs a, int n_pairs, cudaStream_t stream) {
  constexpr int NQ = FUTURE ? T6_ROWS : T6_ROWS / G;
  // rows and columns: (keys, queries) of the future pass, (queries, keys) of the normalisers
  a.A = static_cast<const bf16*>(FUTURE ? K : Q);
  CUtensorMap map;
  cudaError_t e = encode_heads(&map, FUTURE ? Q : K, (long long)n_pairs * (FUTURE ? G : 1), a.S, T6_BN);
  if (e == cudaSuccess) e = raise_smem_limit(lse_t5_kernel<G, FUTURE>, T6_SMEM);
  if (e != cudaSuccess) return e;
  lse_t5_kernel<G, FUTURE><<<(unsigned)n_pairs * ((a.S + NQ - 1) / NQ), T6_THREADS, T6_SMEM, stream>>>(map,
                                                                                                           a);
  return cudaGetLastError();
}

template <bool FUTURE>
cudaError_t dispatch_lse_t5(const void* Q, const void* K, const LseArgs& a, int G, int n_pairs, cudaStream_t stream) {
  if (G == 4) return launch_lse_t5<4, FUTURE>(Q, K, a, n_pairs, stream);
  if (G == 2) return launch_lse_t5<2, FUTURE>(Q, K, a, n_pairs, stream);
  return launch_lse_t5<1, FUTURE>(Q, K, a, n_pairs, stream);
}

// ---------------------------------------------------------------- aggregation
struct AggArgs {
  const float* logm;         // [n][H*G][S]
  const int32_t* len;
  float* target;             // [n][H][S]
  int n_pairs, H, G, S, w, la, agg, count_norm;
  float log_eps;             // log(eps), -inf for eps = 0
};

__global__ void aggregate_kernel(AggArgs a) {
  const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (size_t)a.n_pairs * a.S) return;
  const int pair = (int)(i / a.S), t = (int)(i - (size_t)pair * a.S);
  const int seq = pair / a.H, h = pair - seq * a.H;
  const int L = a.len ? max(0, min(a.len[seq], a.S)) : a.S;
  if (t >= L) return;
  float logN = 0.f;
  if (a.count_norm) {
    int n = max(1, L - (t + a.w));
    if (a.la > 0) n = min(n, a.la + 1);
    logN = logf((float)n);
  }
  const float* lm = a.logm + ((size_t)seq * a.H * a.G + (size_t)h * a.G) * a.S + t;
  float x;
  if (a.agg == 0) {
    x = -INFINITY;
    for (int g = 0; g < a.G; ++g) x = fmaxf(x, lm[(size_t)g * a.S]);
  } else {
    float mx = -INFINITY;
    for (int g = 0; g < a.G; ++g) mx = fmaxf(mx, lm[(size_t)g * a.S]);
    float sum = 0.f;
    if (mx != -INFINITY)
      for (int g = 0; g < a.G; ++g) sum += expf(lm[(size_t)g * a.S] - mx);
    x = mx == -INFINITY ? -INFINITY : mx + logf(sum / (float)a.G);
  }
  x -= logN;
  // log(eps + exp(x)) without overflow
  const float hi = fmaxf(a.log_eps, x), lo = fminf(a.log_eps, x);
  a.target[i] = lo == -INFINITY ? hi : hi + log1pf(expf(lo - hi));
}

}  // namespace

// Causal normalisers of bf16 prompts with d = 128 (d and dtype checked by the caller).
cudaError_t launch_causal_lse_t5(const void* Q, const void* K, const int32_t* len, int n_seq, int H, int G,
                                 int S, float* lse, int32_t* err, cudaStream_t stream) {
  const LseArgs a{nullptr, nullptr, len, lse, n_seq * H, H, S, 0, 0, kLog2e / sqrtf(128.f), err};
  return dispatch_lse_t5<false>(Q, K, a, G, n_seq * H, stream);
}

cudaError_t launch_future_target(const void* Q, const void* K, const float* lse, const int32_t* len,
                                 int n_seq, int H, int G, int d, int S, int w, int la, int dtype,
                                 float* logm, float* target, int agg, int count_norm, float eps,
                                 int32_t* err, cudaStream_t stream) {
  if (n_seq <= 0 || S <= 0) return cudaSuccess;
  // beyond S both say the same as S, and no position is computed past 3 S
  w = std::min(w, S);
  la = std::min(la, S);
  TargetArgs a{Q, K, lse, len, logm, H, G, S, w, la, 1.4426950408889634f / sqrtf((float)d), err};
  const int n_pairs = n_seq * H;
  static const bool mma_sync = [] {
    const char* e = getenv("KVPOP_TARGET_MMA_SYNC");
    return e && e[0] == '1';
  }();
  if (dtype == KVPOP_BF16 && d == 128 && !mma_sync) {
    const LseArgs la_{nullptr, lse, len, logm, n_pairs, H, S, w, la, a.kscale, err};
    cudaError_t e = dispatch_lse_t5<true>(Q, K, la_, G, n_pairs, stream);
    if (e != cudaSuccess) return e;
  } else if (dtype == KVPOP_BF16) {
    const size_t smem = d == 128 ? TgP<128>::SMEM : TgP<64>::SMEM;
    dim3 grid((S + TgP<128>::ROWS - 1) / TgP<128>::ROWS, n_pairs);
    if (d == 128) {
      cudaError_t e = raise_smem_limit(target_tc_kernel<128>, smem);
      if (e != cudaSuccess) return e;
      target_tc_kernel<128><<<grid, TgP<128>::THREADS, smem, stream>>>(a);
    } else {
      cudaError_t e = raise_smem_limit(target_tc_kernel<64>, smem);
      if (e != cudaSuccess) return e;
      target_tc_kernel<64><<<grid, TgP<64>::THREADS, smem, stream>>>(a);
    }
  } else {
    cudaError_t e = d == 128 ? launch_target_f32<128>(a, n_pairs, stream)
                             : launch_target_f32<64>(a, n_pairs, stream);
    if (e != cudaSuccess) return e;
  }
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess || !target) return e;
  AggArgs g{logm, len, target, n_pairs, H, G, S, w, la, agg, count_norm,
            eps > 0.f ? logf(eps) : -INFINITY};
  const size_t n = (size_t)n_pairs * S;
  aggregate_kernel<<<(unsigned)((n + 255) / 256), 256, 0, stream>>>(g);
  return cudaGetLastError();
}

}  // namespace kvpop
