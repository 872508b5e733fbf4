// Stateful delayed mLSTM scorer (App. A, App. E.3, App. E.4): decode ingest and
// prompt prefill.
//
// Per KV head, x_t = [k_t; v_t]; q~ = phi(W_q x), k~ = phi(W_k x), v~ = W_v x with
// W_* in R^{2d x d/2} and the Hedgehog map phi(y) = [softmax(y); softmax(-y)];
// gates i = exp(w_i.x + b_i), f = sigmoid(w_f.x + b_f).  The state (C [d][d/2],
// z [d]) absorbs every token, kept in the stabilised form with a running
// log-scale m:  m' = max(log f + m, log i),  C' = e^{log f + m - m'} C +
// e^{log i - m'} k~ v~^T  (same for z).  At position p, after absorbing token p,
// the token u = p - D that leaves the window is read out with the current state,
// h = (q~_u^T C) / (q~_u^T z), and scored r = a . SiLU(h) + b; the keep-or-drop
// rule is the one of the MLP path (kvpop_evict.cuh).
//
// Weights are packed per head as one matrix Wcat [2d][NC] whose columns are
// [W_k | W_v | W_q | w_i | w_f | 0 pad], so one pass over x gives every
// projection.  The decode kernel loads its head's Wcat whole into shared memory
// with bulk copies (200 KB for d = 128) and serves 8 sequences per CTA.
#include <algorithm>

#include "kvpop_evict.cuh"
#include "kvpop_mma.cuh"
#include "kvpop_tc05.cuh"

namespace kvpop {
namespace {

constexpr int SBM = 8;             // sequences per decode CTA (one warp each)
constexpr int NTM = 256;
constexpr int UTM = 32;            // prompt tokens per projection CTA

struct MState {
  float* C;                        // [pairs][d][d/2]
  float* z;                        // [pairs][d]
  float* m;                        // [pairs]
  const float* Wcat;               // [H][2d][NC]
  const float* bi;                 // [H]
  const float* bf;                 // [H]
  const float* a;                  // [H][d/2]
  const float* b;                  // [H]
  int NC;
};

template <typename T>
struct MIngestArgs {
  State st;
  Dims dm;
  MState ms;
  const T* q;
  const T* k;
  const T* v;
  const float* override_;
  int32_t* evict_info;
  float* score_out;
};

__device__ __forceinline__ float warp_max(float x) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x = fmaxf(x, __shfl_xor_sync(0xffffffffu, x, o));
  return x;
}
__device__ __forceinline__ float warp_sum(float x) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
  return x;
}
__device__ __forceinline__ float softplus(float x) {
  return fmaxf(x, 0.f) + log1pf(expf(-fabsf(x)));
}

// Hedgehog features of y[0..hh) (hh = d/2, held 32 lanes x HP values): out[0..2hh).
template <int HP>
__device__ __forceinline__ void hedgehog_warp(const float* y, float* out, int hh) {
  const int lane = threadIdx.x & 31;
  float v[HP];
  float mp = -INFINITY, mn = -INFINITY;
#pragma unroll
  for (int t = 0; t < HP; ++t) {
    const int i = lane + 32 * t;
    v[t] = i < hh ? y[i] : 0.f;
    if (i < hh) { mp = fmaxf(mp, v[t]); mn = fmaxf(mn, -v[t]); }
  }
  mp = warp_max(mp);
  mn = warp_max(mn);
  float ep[HP], en[HP], sp = 0.f, sn = 0.f;
#pragma unroll
  for (int t = 0; t < HP; ++t) {
    const int i = lane + 32 * t;
    ep[t] = i < hh ? expf(v[t] - mp) : 0.f;
    en[t] = i < hh ? expf(-v[t] - mn) : 0.f;
    sp += ep[t];
    sn += en[t];
  }
  sp = warp_sum(sp);
  sn = warp_sum(sn);
#pragma unroll
  for (int t = 0; t < HP; ++t) {
    const int i = lane + 32 * t;
    if (i < hh) { out[i] = ep[t] / sp; out[hh + i] = en[t] / sn; }
  }
}

// C <- fs C + is k~ v~^T on this lane's columns (NJ of them) and y += q~^T C, rows
// in chunks of 32 whose loads are all issued before the first store.
template <int NJ>
__device__ __forceinline__ void state_rows(float* __restrict__ C, int d, int hh, float fs, float is,
                                           const float* kt, const float* qt, const float (&vj)[2],
                                           float (&yj)[2]) {
  const int lane = threadIdx.x & 31;
  for (int i0 = 0; i0 < d; i0 += 32) {
    float c[32][NJ];
#pragma unroll
    for (int r = 0; r < 32; ++r)
#pragma unroll
      for (int t = 0; t < NJ; ++t) c[r][t] = __ldcg(C + (size_t)(i0 + r) * hh + lane + 32 * t);
#pragma unroll
    for (int r = 0; r < 32; ++r) {
      const float ki = is * kt[i0 + r], qi = qt[i0 + r];
#pragma unroll
      for (int t = 0; t < NJ; ++t) {
        const float cn = fmaf(fs, c[r][t], ki * vj[t]);
        C[(size_t)(i0 + r) * hh + lane + 32 * t] = cn;
        yj[t] = fmaf(qi, cn, yj[t]);
      }
    }
  }
}

__host__ __device__ inline size_t mlstm_ingest_smem(int d, int NC, int esz) {
  return (size_t)2 * d * NC * 4 + 2 * (size_t)2 * d * SBM * 4 + (size_t)SBM * NC * 4 +
         2 * (size_t)SBM * d * esz;
}

template <typename T>
__global__ void __launch_bounds__(NTM, 1) ingest_mlstm_kernel(MIngestArgs<T> a) {
  const Dims& dm = a.dm;
  const int d = dm.d, D = dm.D, H = dm.H, NC = a.ms.NC, hh = d / 2;
  const int in2 = 2 * d;
  const int h = blockIdx.y, b0 = blockIdx.x * SBM;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

  extern __shared__ __align__(128) unsigned char smem[];
  float* Ws = reinterpret_cast<float*>(smem);                  // [2d][NC]
  float* Xp = Ws + (size_t)in2 * NC;                           // [2d][SBM]  x of the new token
  float* Xu = Xp + in2 * SBM;                                  // [2d][SBM]  x of the leaving token
  float* proj = Xu + in2 * SBM;                                // [SBM][NC]
  T* rawk = reinterpret_cast<T*>(proj + SBM * NC);             // [SBM][d]
  T* rawv = rawk + SBM * d;
  float* feat = Xp;                                            // [SBM][2][d] after the projections
  __shared__ __align__(8) uint64_t bar;
  __shared__ int s_p[SBM];

  if (tid == 0) {
    mbar_init(smem_u32(&bar), 1);
    mbar_fence_init();
    const uint32_t bytes = (uint32_t)(in2 * NC * 4);
    mbar_arrive_expect_tx(smem_u32(&bar), bytes);
    const unsigned char* src = reinterpret_cast<const unsigned char*>(a.ms.Wcat + (size_t)h * in2 * NC);
    for (uint32_t off = 0; off < bytes; off += 32768)
      bulk_g2s(smem_u32(smem + off), src + off, min(32768u, bytes - off), smem_u32(&bar));
  }
  // The weights above never change, all that follows is state or input that the kernel before
  // this one may still write.  The attention may be scheduled after that, and not earlier: it
  // starts on keys that this step does not change.
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  T* ringK = static_cast<T*>(a.st.ringK);
  T* ringV = static_cast<T*>(a.st.ringV);
  {
    const int b = b0 + warp;
    int p = -1;
    if (b < dm.batch) {
      const int pair = b * H + h;
      p = a.st.len[pair];
      const int ri = p % D;
      const T* kp = a.k + (size_t)pair * d;
      const T* vp = a.v + (size_t)pair * d;
      T* rk = ringK + ((size_t)pair * D + ri) * d;
      T* rv = ringV + ((size_t)pair * D + ri) * d;
      for (int i = lane; i < d; i += 32) {
        const T ku = rk[i], vu = rv[i];
        rawk[warp * d + i] = ku;
        rawv[warp * d + i] = vu;
        Xu[i * SBM + warp] = p >= D ? to_f(ku) : 0.f;
        Xu[(d + i) * SBM + warp] = p >= D ? to_f(vu) : 0.f;
        const T kn = kp[i], vn = vp[i];
        Xp[i * SBM + warp] = to_f(kn);
        Xp[(d + i) * SBM + warp] = to_f(vn);
      }
      __syncwarp();
      for (int i = lane; i < d; i += 32) {     // the new token takes u's window slot
        rk[i] = kp[i];
        rv[i] = vp[i];
      }
    } else {
      for (int i = lane; i < in2; i += 32) { Xp[i * SBM + warp] = 0.f; Xu[i * SBM + warp] = 0.f; }
    }
    if (lane == 0) s_p[warp] = p;
  }
  __syncthreads();
  const bool ok = mbar_wait(smem_u32(&bar), 0, a.st.err, DEVERR_TIMEOUT_FULL);

  // ---- all projections of the 8 sequences: column c of Wcat per thread -------------
  for (int c = tid; c < NC; c += NTM) {
    const float* X = (c >= d && c < d + hh) ? Xu : Xp;     // W_q reads the leaving token
    float acc[SBM];
#pragma unroll
    for (int s = 0; s < SBM; ++s) acc[s] = 0.f;
    if (ok) {
#pragma unroll 4
      for (int i = 0; i < in2; ++i) {
        const float w = Ws[(size_t)i * NC + c];
        const float4 x0 = *reinterpret_cast<const float4*>(X + i * SBM);
        const float4 x1 = *reinterpret_cast<const float4*>(X + i * SBM + 4);
        acc[0] = fmaf(x0.x, w, acc[0]); acc[1] = fmaf(x0.y, w, acc[1]);
        acc[2] = fmaf(x0.z, w, acc[2]); acc[3] = fmaf(x0.w, w, acc[3]);
        acc[4] = fmaf(x1.x, w, acc[4]); acc[5] = fmaf(x1.y, w, acc[5]);
        acc[6] = fmaf(x1.z, w, acc[6]); acc[7] = fmaf(x1.w, w, acc[7]);
      }
    }
#pragma unroll
    for (int s = 0; s < SBM; ++s) proj[s * NC + c] = acc[s];
  }
  __syncthreads();

  // ---- per sequence: features, state update, delayed readout, keep-or-drop ---------
  const int b = b0 + warp;
  if (b >= dm.batch || !ok) return;
  const int pair = b * H + h;
  const int p = s_p[warp];
  const float* pr = proj + warp * NC;
  float* kt = feat + (size_t)warp * 2 * d;          // k~ [d]
  float* qt = kt + d;                                // q~ [d]
  if (hh > 32) {
    hedgehog_warp<2>(pr, kt, hh);
    hedgehog_warp<2>(pr + d, qt, hh);
  } else {
    hedgehog_warp<1>(pr, kt, hh);
    hedgehog_warp<1>(pr + d, qt, hh);
  }
  __syncwarp();
  const float ai = pr[3 * hh] + a.ms.bi[h];
  const float af = pr[3 * hh + 1] + a.ms.bf[h];
  const float lf = -softplus(-af);
  const float m_old = a.ms.m[pair];
  const float m_new = fmaxf(lf + m_old, ai);
  const float fs = (m_old == -INFINITY) ? 0.f : expf(lf + m_old - m_new);
  const float is = expf(ai - m_new);
  // columns j = lane (+32) of C and of the readout: rows are loaded 32 at a time
  // (independent loads in flight) before they are updated and stored
  float vj[2], yj[2] = {0.f, 0.f};
  const int nj = hh / 32;
  for (int t = 0; t < nj; ++t) vj[t] = pr[hh + lane + 32 * t];
  float* __restrict__ C = a.ms.C + (size_t)pair * d * hh;
  if (nj == 2) state_rows<2>(C, d, hh, fs, is, kt, qt, vj, yj);
  else         state_rows<1>(C, d, hh, fs, is, kt, qt, vj, yj);
  float den = 0.f;
  float* z = a.ms.z + (size_t)pair * d;
  for (int i = lane; i < d; i += 32) {
    const float zn = fmaf(fs, z[i], is * kt[i]);
    z[i] = zn;
    den = fmaf(qt[i], zn, den);
  }
  den = warp_sum(den);
  if (lane == 0) a.ms.m[pair] = m_new;
  if (p < D) {
    if (lane == 0) {
      a.st.len[pair] = p + 1;
      if (a.evict_info) { a.evict_info[2 * pair] = -1; a.evict_info[2 * pair + 1] = -1; }
      if (a.score_out) a.score_out[pair] = __int_as_float(0x7fc00000);
    }
    return;
  }
  float rpart = 0.f;
  for (int t = 0; t < nj; ++t) {
    const float hv = yj[t] / den;
    const float silu = hv / (1.f + expf(-hv));
    rpart = fmaf(a.ms.a[(size_t)h * hh + lane + 32 * t], silu, rpart);
  }
  float r = warp_sum(rpart) + a.ms.b[h];
  if (a.override_) r = a.override_[pair];
  evict_and_scatter<T>(a.st, dm, pair, h, p, r, rawk + warp * d, rawv + warp * d, a.evict_info,
                       a.score_out);
}

// ------------------------------------------------------------------ prefill
struct MProjArgs {
  Dims dm;
  MState ms;
  const float* K;                  // [n_seq][H][Pmax][d]
  const float* V;
  const int32_t* plen;
  float* feat;                     // [n_seq*H][Pmax][NF]: k~ (d) | v~ (d/2) | q~ (d) | a_i | a_f
  int Pmax, NF;
};

// fp32 K/V: column c of Wcat per thread, 32 tokens per CTA.
__global__ void __launch_bounds__(NTM) mlstm_proj_kernel(MProjArgs a) {
  const Dims& dm = a.dm;
  const int d = dm.d, H = dm.H, NC = a.ms.NC, hh = d / 2, in2 = 2 * d, NF = a.NF;
  const int lp = blockIdx.y, bl = lp / H, h = lp - bl * H;
  const int P = a.plen[bl];
  const int t0 = blockIdx.x * UTM;
  if (t0 >= P) return;
  const int nrow = min(UTM, P - t0);
  extern __shared__ __align__(128) unsigned char smem[];
  float* Xt = reinterpret_cast<float*>(smem);                  // [2d][UTM]
  float* pj = Xt + in2 * UTM;                                  // [UTM][NC]
  const size_t Pm = a.Pmax;
  const float* Kp = a.K + ((size_t)bl * H + h) * Pm * d;
  const float* Vp = a.V + ((size_t)bl * H + h) * Pm * d;
  for (int idx = threadIdx.x; idx < UTM * d; idx += NTM) {
    const int r = idx / d, i = idx - r * d;
    const bool in = r < nrow;
    Xt[i * UTM + r] = in ? Kp[(size_t)(t0 + r) * d + i] : 0.f;
    Xt[(d + i) * UTM + r] = in ? Vp[(size_t)(t0 + r) * d + i] : 0.f;
  }
  __syncthreads();
  const float* W = a.ms.Wcat + (size_t)h * in2 * NC;
  for (int c = threadIdx.x; c < NC; c += NTM) {
    float acc[UTM];
#pragma unroll
    for (int r = 0; r < UTM; ++r) acc[r] = 0.f;
#pragma unroll 2
    for (int i = 0; i < in2; ++i) {
      const float w = __ldg(W + (size_t)i * NC + c);
      const float4* xr = reinterpret_cast<const float4*>(Xt + i * UTM);
#pragma unroll
      for (int r4 = 0; r4 < UTM / 4; ++r4) {
        const float4 x = xr[r4];
        acc[4 * r4 + 0] = fmaf(x.x, w, acc[4 * r4 + 0]);
        acc[4 * r4 + 1] = fmaf(x.y, w, acc[4 * r4 + 1]);
        acc[4 * r4 + 2] = fmaf(x.z, w, acc[4 * r4 + 2]);
        acc[4 * r4 + 3] = fmaf(x.w, w, acc[4 * r4 + 3]);
      }
    }
#pragma unroll
    for (int r = 0; r < UTM; ++r) pj[r * NC + c] = acc[r];
  }
  __syncthreads();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float* out = a.feat + ((size_t)lp * Pm) * NF;
  for (int r = warp; r < nrow; r += NTM / 32) {
    float* o = out + (size_t)(t0 + r) * NF;
    const float* pr = pj + r * NC;
    if (hh > 32) { hedgehog_warp<2>(pr, o, hh); hedgehog_warp<2>(pr + d, o + d + hh, hh); }
    else         { hedgehog_warp<1>(pr, o, hh); hedgehog_warp<1>(pr + d, o + d + hh, hh); }
    for (int j = lane; j < hh; j += 32) o[d + j] = pr[hh + j];
    if (lane == 0) {
      o[2 * d + hh] = pr[3 * hh] + a.ms.bi[h];
      o[2 * d + hh + 1] = pr[3 * hh + 1] + a.ms.bf[h];
    }
  }
}

// The same projections for bf16 K/V on tcgen05 with fp32 accuracy: x is exact in bf16 and every
// weight is split exactly into three bf16 parts (8 + 8 + 8 bits, W^T stored once per cache as
// the shared-memory image of its tiles), so W x is three products whose terms are exact.  The
// tensor unit rounds a running sum toward zero; to keep that below the rounding of a chain of
// fp32 FMAs, each 64 inputs are summed on their own, smallest parts first, and added in fp32
// (two accumulators of 128 inputs each: out.score 1.1e-6 from 64 bits, 6.8e-7 this way; the scores
// of prompts of 250 to 4009 tokens, with the readout below, 2.1e-7 to 2.9e-7 in the mean and 4.2e-6
// at most, against 5.4e-7 to 6.4e-7 and 1.8e-5 with chains of fp32 FMAs).  A CTA
// takes 128 tokens: one warp copies the weights (80 KB per 64 inputs, two buffers) and issues
// the MMAs (M = 128, N = 208); 8 warps load the tokens and, one thread per token and feature
// map, add up the token's accumulator rows and run the Hedgehog softmaxes on them, then hand
// whole rows of features to a bulk store.  Bound by the
// weights' way from L2 (320 KB per CTA) and the exponentials.  64 pairs of up to 4009 tokens,
// d = 128: 205 us, against 283 us on mma.sync and 1125 us with fp32 FMAs.
constexpr int PT_TOK = 128;
constexpr int PT_KC = 64;                          // inputs per chunk: one 128-byte row
constexpr int PT_THREADS = NTM + 32;
enum : int { PTERR_WAIT = 31 };

template <int HD>
struct PtP {
  static constexpr int HH = HD / 2;
  static constexpr int NCP = (3 * HH + 2 + 15) / 16 * 16;   // columns: W_k, W_v, W_q, gates, zeros
  static constexpr int IN2 = 2 * HD;
  static constexpr int NKC = IN2 / PT_KC;
  static constexpr int NF = ((2 * HD + HH + 2) + 3) & ~3;
  static constexpr int XB = PT_TOK * IN2 * 2;      // tokens: NKC tiles of [128][64]
  static constexpr int WT = NCP * PT_KC * 2;       // one part of one chunk
  static constexpr int WB = 3 * WT;
  static constexpr int ROUNDS = NKC / 2;           // two chunks, one per accumulator, a round
  static constexpr int OFF_BAR = XB + 2 * WB;
  static constexpr int SMEM = OFF_BAR + 64 + 1024;
  static constexpr int TM_COLS = 2 * NCP <= 256 ? 256 : 512;
  static_assert(PT_TOK * NF * 4 <= OFF_BAR, "the features are staged over the operands");
  static_assert(NF * 4 % 16 == 0, "rows of features leave by bulk copies");
};

// W^T parts: wt [H][NKC][3][NCP][64] in the 128-byte-swizzled order of a K-major tile, from
// Wcat [H][2d][NC]
template <int HD>
__global__ void mlstm_split_kernel(const float* __restrict__ Wcat, int NC, int H, bf16* __restrict__ wt) {
  using P = PtP<HD>;
  const int n = H * P::IN2 * P::NCP;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const int c = i % P::NCP, k = (i / P::NCP) % P::IN2, h = i / (P::NCP * P::IN2);
    const float w = c < NC ? Wcat[((size_t)h * P::IN2 + k) * NC + c] : 0.f;
    bf16 part[3] = {__float2bfloat16_rz(w), __float2bfloat16_rz(0.f), __float2bfloat16_rz(0.f)};
    if (isfinite(w)) {
      const float r1 = w - __bfloat162float(part[0]);
      part[1] = __float2bfloat16_rz(r1);
      part[2] = __float2bfloat16_rz(r1 - __bfloat162float(part[1]));
    }
    const int kk = k % PT_KC;
    for (int q = 0; q < 3; ++q)
      wt[(((size_t)h * P::NKC + k / PT_KC) * 3 + q) * P::NCP * PT_KC + swz(c, kk / 8, 128) / 2 + kk % 8] = part[q];
  }
}

struct MProjTcArgs {
  const bf16* K;                   // [n_seq][H][Pmax][d]
  const bf16* V;
  const bf16* wt;
  const float* bi;
  const float* bf;
  const int32_t* plen;
  float* feat;
  int32_t* err;
  int H, Pmax;
};

template <int HD>
__global__ void __launch_bounds__(PT_THREADS, 1) mlstm_proj_tc_kernel(MProjTcArgs a) {
  using namespace tc05;
  using P = PtP<HD>;
  constexpr int HH = P::HH, NF = P::NF;
  extern __shared__ unsigned char sm_pt_raw[];
  unsigned char* sm = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(sm_pt_raw) + 1023) & ~(uintptr_t)1023);
  const int lp = blockIdx.y, bl = lp / a.H, h = lp - bl * a.H;
  const int L = a.plen[bl], t0 = blockIdx.x * PT_TOK;
  if (t0 >= L) return;
  const int nrow = min(PT_TOK, L - t0);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t sb = smem_u32(sm);
  auto bar = [&](int i) { return sb + P::OFF_BAR + 8u * (uint32_t)i; };
  if (tid == 0) {                                  // 0, 1 W; 2 x; 3, 4 MMAs done; 5 sums read
    for (int i = 0; i < 6; ++i) mbar_init(bar(i), i == 2 || i == 5 ? NTM : 1);
    mbar_fence_init();
  }
  if (warp == NTM / 32) tmem_alloc(sb + P::OFF_BAR + 48, P::TM_COLS);
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = *reinterpret_cast<volatile uint32_t*>(sm + P::OFF_BAR + 48);
  if (warp == NTM / 32) {
    // ---------------------------------------------------------------- weights, MMA issue
    const bf16* wt = a.wt + (size_t)h * P::NKC * 3 * P::NCP * PT_KC;
    const bool lead = elect_one();
    auto load_w = [&](int kc) {
      if (lead) {
        mbar_arrive_expect_tx(bar(kc & 1), P::WB);
        for (int q = 0; q < 3; ++q)
          bulk_g2s(sb + P::XB + (kc & 1) * P::WB + q * P::WT, wt + (size_t)(3 * kc + q) * P::NCP * PT_KC, P::WT,
                   bar(kc & 1));
      }
      __syncwarp();
    };
    auto all = [](bool x) { return __all_sync(0xffffffffu, x); };
    const uint32_t id = idesc_bf16(128, P::NCP, 0);
    const uint64_t xd0 = kmajor_desc(sb, PT_TOK, 0), wd0 = kmajor_desc(sb + P::XB, P::NCP, 0);
    int asked = 0, waited = 0;                     // chunks requested, chunks seen to land
    for (; asked < 2 && asked < P::NKC; ++asked) load_w(asked);
    bool ok = all(mbar_wait(bar(2), 0, a.err, PTERR_WAIT));
    if (ok) fence_async_smem();
    for (int kc = 0; kc < P::NKC && ok; ++kc) {
      if (!(ok = all(mbar_wait(bar(kc & 1), (kc >> 1) & 1, a.err, PTERR_WAIT)))) break;
      waited = kc + 1;
      if (kc >= 2 && kc % 2 == 0 && !(ok = all(mbar_wait(bar(5), (kc / 2 - 1) & 1, a.err, PTERR_WAIT)))) break;
      fence_after();
      if (lead) {
        const uint64_t xd = desc_at(xd0, kc * PT_TOK * 128), wd = desc_at(wd0, (kc & 1) * P::WB);
#pragma unroll
        for (int q = 2; q >= 0; --q)               // smallest part first
#pragma unroll
          for (int ks = 0; ks < 4; ++ks)
            mma_bf16(tmem + (kc & 1) * P::NCP, kmajor_step(xd, PT_TOK, ks),
                     kmajor_step(desc_at(wd, q * P::WT), P::NCP, ks), id, !(q == 2 && ks == 0));
        commit(bar(3 + (kc & 1)));
      }
      __syncwarp();
      if (asked < P::NKC) {                        // the buffer's next chunk, once its MMAs are done
        if (!(ok = all(mbar_wait(bar(3 + (kc & 1)), (kc >> 1) & 1, a.err, PTERR_WAIT)))) break;
        load_w(asked++);
      }
    }
    if (!ok)                                       // copies in flight land before the CTA ends
      for (int kc = waited; kc < asked; ++kc) mbar_wait(bar(kc & 1), (kc >> 1) & 1, nullptr, 0);
    __syncwarp();
  } else {
    // ---------------------------------------------------------------- tokens, features
    const bf16* Kp = a.K + (size_t)lp * a.Pmax * HD;
    const bf16* Vp = a.V + (size_t)lp * a.Pmax * HD;
    for (int i = tid; i < PT_TOK * (P::IN2 / 8); i += NTM) {
      const int r = i / (P::IN2 / 8), c = i - r * (P::IN2 / 8);
      const bool in = r < nrow;
      const size_t row = (size_t)(in ? t0 + r : t0) * HD;
      const bf16* src = c < HD / 8 ? Kp + row + 8 * c : Vp + row + 8 * c - HD;
      cp_async16(sb + (c >> 3) * (PT_TOK * 128) + swz(r, c & 7, 128), src, in ? 16 : 0);
    }
    cp_async_arrive_noinc(bar(2));
    // thread: token r = 32 (warp mod 4) + lane; warps 0-3 take k~ and half of v~, 4-7 q~, the
    // other half of v~ and the gates
    const int quarter = warp & 3, sel = warp >> 2, r = quarter * 32 + lane;
    const uint32_t tr = tmem + ((uint32_t)(quarter * 32) << 16);
    float* row = reinterpret_cast<float*>(sm) + (size_t)r * NF;
    constexpr int NV = HH / 32;                    // 32-column groups of one projection
    constexpr int G0 = 3 * HH - (P::NCP - 16);     // gate a_i in the last 16 columns, a_f next to it
    static_assert(G0 >= 0 && G0 + 1 < 16, "");
    const bool with_v = NV == 2 || sel == 0;       // v~: one group each, or the only one
    float y[NV][32], x[32], gi = 0.f, gf = 0.f;
    bool ok = true;
#pragma unroll
    for (int rd = 0; rd < P::ROUNDS; ++rd) {
      ok = ok && mbar_wait(bar(3), rd & 1, a.err, PTERR_WAIT) && mbar_wait(bar(4), rd & 1, a.err, PTERR_WAIT);
      ok = __all_sync(0xffffffffu, ok);
      fence_after();
      if (!ok) break;
      auto columns = [&](int c0, float (&v)[32]) {   // 32 columns of the token's projections
        float u[32], w[32];
        tmem_ld32(tr + c0, u);
        tmem_ld32(tr + P::NCP + c0, w);
        tmem_wait_ld();
#pragma unroll
        for (int i = 0; i < 32; ++i) v[i] = rd ? v[i] + (u[i] + w[i]) : u[i] + w[i];
      };
#pragma unroll
      for (int g = 0; g < NV; ++g) columns((sel ? 2 * HH : 0) + 32 * g, y[g]);
      if (with_v) columns(HH + (NV == 2 ? 32 * sel : 0), x);
      if (sel == 1) {
        // the gates' tile (the columns past them hold zeros or belong to the other accumulator)
        float u[32], w[32];
        tmem_ld32(tr + P::NCP - 16, u);
        tmem_ld32(tr + 2 * P::NCP - 32, w);
        tmem_wait_ld();
        gi += u[G0] + w[G0 + 16];
        gf += u[G0 + 1] + w[G0 + 17];
      }
      if (rd + 1 < P::ROUNDS) {
        fence_before();
        mbar_arrive(bar(5));
      }
    }
    cp_wait<0>();
    if (ok) {
      auto put = [&](int at, const float (&v)[32]) {
#pragma unroll
        for (int i = 0; i < 32; i += 4)
          *reinterpret_cast<float4*>(row + at + i) = make_float4(v[i], v[i + 1], v[i + 2], v[i + 3]);
      };
      // the operands are read: features take their place, rows of NF floats
      if (with_v) put(HD + (NV == 2 ? 32 * sel : 0), x);
      if (sel == 1)
        *reinterpret_cast<float4*>(row + 2 * HD + HH) = make_float4(gi + a.bi[h], gf + a.bf[h], 0.f, 0.f);
      float ep[NV][32], en[NV][32];
      float mp = -INFINITY, mn = -INFINITY;
#pragma unroll
      for (int g = 0; g < NV; ++g)
#pragma unroll
        for (int i = 0; i < 32; ++i) {
          mp = fmaxf(mp, y[g][i]);
          mn = fmaxf(mn, -y[g][i]);
        }
      float ps[4] = {}, ns[4] = {};
#pragma unroll
      for (int g = 0; g < NV; ++g)
#pragma unroll
        for (int i = 0; i < 32; ++i) {
          ep[g][i] = expf(y[g][i] - mp);
          en[g][i] = expf(-y[g][i] - mn);
          ps[i & 3] += ep[g][i];
          ns[i & 3] += en[g][i];
        }
      const float sp = (ps[0] + ps[1]) + (ps[2] + ps[3]), sn = (ns[0] + ns[1]) + (ns[2] + ns[3]);
#pragma unroll
      for (int g = 0; g < NV; ++g)
#pragma unroll
        for (int i = 0; i < 32; ++i) {
          ep[g][i] /= sp;
          en[g][i] /= sn;
        }
      const int at = sel ? HD + HH : 0;
#pragma unroll
      for (int g = 0; g < NV; ++g) {
        put(at + 32 * g, ep[g]);
        put(at + HH + 32 * g, en[g]);
      }
    }
    // the quarter's rows leave together: both warps' parts are there
    fence_async_smem();
    asm volatile("bar.sync %0, 64;" ::"r"(1 + quarter) : "memory");
    if (sel == 0 && lane == 0 && ok && quarter * 32 < nrow) {
      const uint32_t bytes = (uint32_t)(min(32, nrow - quarter * 32) * NF * 4);
      asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(
                       a.feat + ((size_t)lp * a.Pmax + t0 + quarter * 32) * NF),
                   "r"(sb + (uint32_t)(quarter * 32 * NF * 4)), "r"(bytes)
                   : "memory");
      asm volatile("cp.async.bulk.commit_group;" ::: "memory");
      asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
    }
    __syncwarp();
  }
  fence_before();
  __syncthreads();
  if (warp == NTM / 32) tmem_dealloc(tmem, P::TM_COLS);
}

struct MScanArgs {
  State st;
  Dims dm;
  MState ms;
  const int32_t* plen;
  const float* feat;
  const float* override_;          // [n_seq][H][Pmax] or nullptr
  float* prio;                     // [n_seq][H][Pmax]
  float* seg;                      // [pairs][nseg - 1][d d/2 + d] states between segments
  float* seg_scal;                 // [pairs][nseg][2] log-scale and log forget sum of a segment
  float* seg_m;                    // [pairs][nseg] log-scale at a segment's start
  int first_seq, Pmax, NF;
  int n, nseg;                     // chunks per segment, segments
};

// Chunkwise form of the same recurrence (App. A: the mLSTM as linear attention with
// gates).  Within a chunk of L tokens starting at t0, with F_s the cumulative log
// forget gate of the chunk up to token s and g_s = log i_s - F_s, the state after
// absorbing token t is, up to one common scale,
//   C(t) = e^{m - R_t} C + sum_{s <= t} e^{g_s - R_t} k~_s v~_s^T,   R_t = max(m, max_{s<=t} g_s)
// (same for z), where (C, z, m) is the stabilised state at the chunk start; the
// scale e^{F_t + R_t} cancels in the readout ratio, and at the chunk's end it is the
// new log-scale m' = F_{L-1} + R_{L-1}, which equals the token-by-token stabiliser.
// Every exponent is <= 0.  The readout of row t (token u = t0 + t - D) is
//   h = (e^{m-R_t} q~_u^T C + sum_s W_ts v~_s) / (e^{m-R_t} q~_u^T z + sum_s W_ts),
//   W_ts = e^{g_s - R_t} (q~_u . k~_s)  for s <= t,
// so a chunk costs three small dense products (q~ K^T, q~ C, W V) plus the state
// update C' = e^{m - R_{L-1}} C + K^T diag(e^{g - R_{L-1}}) V.
//
// Chunks depend on each other only through (C, z, m), so a pair's chunks are cut into
// segments: mlstm_seg_kernel takes every segment (but a pair's last) from an empty state,
// mlstm_link_kernel chains those states, and mlstm_chunk_kernel reads out all segments at
// once, each from its own start.  64 pairs of up to 4009 tokens, d = 128: 561 us
// together, against 1557 us with the chunks of a pair one after another on 64 SMs.
constexpr int CL = 64;             // tokens per chunk
constexpr int NTC = 512;           // threads of the readout: two groups of 256

template <int N>
__device__ __forceinline__ void ld_vec(float (&x)[N], const float* p) {
  if constexpr (N == 2) {
    const float2 v = *reinterpret_cast<const float2*>(p);
    x[0] = v.x; x[1] = v.y;
  } else {
#pragma unroll
    for (int i = 0; i < N; i += 4) {
      const float4 v = *reinterpret_cast<const float4*>(p + i);
      x[i] = v.x; x[i + 1] = v.y; x[i + 2] = v.z; x[i + 3] = v.w;
    }
  }
}
template <int N>
__device__ __forceinline__ void st_vec(float* p, const float (&x)[N]) {
  if constexpr (N == 2) {
    *reinterpret_cast<float2*>(p) = make_float2(x[0], x[1]);
  } else {
#pragma unroll
    for (int i = 0; i < N; i += 4)
      *reinterpret_cast<float4*>(p + i) = make_float4(x[i], x[i + 1], x[i + 2], x[i + 3]);
  }
}

template <int HD>
struct ChunkLayout {
  static constexpr int HH = HD / 2;
  static constexpr int QS = HD + 4;              // row strides (floats), multiples of 4
  static constexpr int VS = HH + 4;
  static constexpr int WS = CL + 4;
  // one buffer of a chunk's features (two of them, the next chunk's in flight)
  static constexpr int B_K = 0;                  // [CL][QS]  k~ of the chunk's tokens
  static constexpr int B_V = B_K + CL * QS;      // [CL][VS]  v~
  static constexpr int B_G = B_V + CL * VS;      // [CL][4]   a_i, a_f
  static constexpr int B_Q = B_G + CL * 4;       // [CL][QS]  q~ of the read-out tokens
  static constexpr int BUF = B_Q + CL * QS;
  static constexpr int BUF_S = B_Q;              // without q~ (segment states)
  static constexpr int SEG = HD * HH + HD;       // floats of a state in global memory
};

// Gates of one chunk by one warp (two tokens per lane): g_s, R_t, e^{g_s - R_{L-1}}, and
// F_{L-1} in sc[1].
__device__ __forceinline__ void chunk_gates(const float* G, int t0, int P, float m, float* gs, float* Rs,
                                            float* es, float* sc) {
  const int lane = threadIdx.x & 31;
  float lfv[2], aiv[2];
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    const int r = 2 * lane + k;
    const bool in = t0 + r < P;
    aiv[k] = in ? G[4 * r] : -INFINITY;
    lfv[k] = in ? -softplus(-G[4 * r + 1]) : 0.f;
  }
  const float f1 = lfv[0] + lfv[1];
  float inc = f1;                                  // inclusive scan over lane pairs
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const float y = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += y;
  }
  const float Fa = inc - f1 + lfv[0], Fb = inc;    // F of tokens 2 lane, 2 lane + 1
  const float ga = aiv[0] - Fa, gb = aiv[1] - Fb;
  float run = fmaxf(ga, gb);                       // inclusive prefix max
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const float y = __shfl_up_sync(0xffffffffu, run, o);
    if (lane >= o) run = fmaxf(run, y);
  }
  const float prev = __shfl_up_sync(0xffffffffu, run, 1);
  const float before = lane == 0 ? -INFINITY : prev;
  const float RL = fmaxf(m, __shfl_sync(0xffffffffu, run, 31));
  gs[2 * lane] = ga;
  gs[2 * lane + 1] = gb;
  if (Rs) {
    Rs[2 * lane] = fmaxf(m, fmaxf(before, ga));
    Rs[2 * lane + 1] = fmaxf(m, run);
  }
  es[2 * lane] = __expf(ga - RL);
  es[2 * lane + 1] = __expf(gb - RL);
  if (lane == 31) {
    sc[1] = Fb;                                    // F of the chunk's last token
    sc[2] = RL;
  }
}

// Copies one chunk's features into a buffer (rows past the prompt zero-filled).
template <int HD, bool WITH_Q>
__device__ __forceinline__ void load_chunk(const float* F, int NF, int t0, int P, int D, float* buf, int nt) {
  using Ly = ChunkLayout<HD>;
  const int tid = threadIdx.x;
  const uint32_t b = smem_u32(buf);
  for (int e = tid; e < CL * (HD / 4); e += nt) {
    const int r = e / (HD / 4), c = e - r * (HD / 4), t = t0 + r, u = t - D;
    const bool in = t < P;
    cp_async16(b + (Ly::B_K + r * Ly::QS + 4 * c) * 4, F + (size_t)(in ? t : 0) * NF + 4 * c, in ? 16 : 0);
    if (WITH_Q) {
      const bool iq = in && u >= 0;
      cp_async16(b + (Ly::B_Q + r * Ly::QS + 4 * c) * 4, F + (size_t)(iq ? u : 0) * NF + HD + Ly::HH + 4 * c,
                 iq ? 16 : 0);
    }
  }
  for (int e = tid; e < CL * (Ly::HH / 4); e += nt) {
    const int r = e / (Ly::HH / 4), c = e - r * (Ly::HH / 4), t = t0 + r;
    cp_async16(b + (Ly::B_V + r * Ly::VS + 4 * c) * 4, F + (size_t)(t < P ? t : 0) * NF + HD + 4 * c, t < P ? 16 : 0);
  }
  for (int r = tid; r < CL; r += nt)
    cp_async16(b + (Ly::B_G + 4 * r) * 4, F + (size_t)(t0 + r < P ? t0 + r : 0) * NF + 2 * HD + Ly::HH,
               t0 + r < P ? 16 : 0);
}

// acc += K^T diag(es) V on this thread's HD / 16 rows x HH / 16 columns of the state
template <int HD>
__device__ __forceinline__ void state_update(float (&acc)[HD / 16][HD / 32], const float* Ks, const float* Vs,
                                             const float* es, int ty, int tx) {
  using Ly = ChunkLayout<HD>;
  constexpr int NR = HD / 16, NB = HD / 32;
#pragma unroll 4
  for (int s = 0; s < CL; ++s) {
    float v[NB], k[NR];
    ld_vec<NB>(v, Vs + s * Ly::VS + NB * tx);
    ld_vec<NR>(k, Ks + s * Ly::QS + NR * ty);
    const float w = es[s];
#pragma unroll
    for (int j = 0; j < NB; ++j) v[j] *= w;
#pragma unroll
    for (int i = 0; i < NR; ++i)
#pragma unroll
      for (int j = 0; j < NB; ++j) acc[i][j] = fmaf(k[i], v[j], acc[i][j]);
  }
}

// State that a segment's tokens leave from an empty one (every segment but a pair's last).
template <int HD>
__global__ void __launch_bounds__(NTM) mlstm_seg_kernel(MScanArgs a) {
  using Ly = ChunkLayout<HD>;
  constexpr int HH = Ly::HH, NR = HD / 16, NB = HD / 32;
  extern __shared__ __align__(16) float smf[];
  __shared__ float gs[CL], es[CL], sc[4];
  const int lp = blockIdx.y, seg = blockIdx.x;
  const int P = a.plen[lp / a.dm.H];
  const int c0 = seg * a.n, c1 = c0 + a.n;
  if (c1 * CL >= P) return;                        // the pair's last segment, or past it
  const int tid = threadIdx.x, ty = tid >> 4, tx = tid & 15;
  const float* F = a.feat + (size_t)lp * a.Pmax * a.NF;
  float acc[NR][NB], zn = 0.f, m = -INFINITY, Ft = 0.f;
#pragma unroll
  for (int i = 0; i < NR; ++i)
#pragma unroll
    for (int j = 0; j < NB; ++j) acc[i][j] = 0.f;
  load_chunk<HD, false>(F, a.NF, c0 * CL, P, 0, smf, NTM);
  cp_commit();
  for (int c = c0; c < c1; ++c) {
    const float* buf = smf + ((c - c0) & 1) * Ly::BUF_S;
    if (c + 1 < c1) load_chunk<HD, false>(F, a.NF, (c + 1) * CL, P, 0, smf + ((c + 1 - c0) & 1) * Ly::BUF_S, NTM);
    cp_commit();
    cp_wait<1>();
    __syncthreads();
    if (tid < 32) chunk_gates(buf + Ly::B_G, c * CL, P, m, gs, nullptr, es, sc);
    __syncthreads();
    const float RL = sc[2], wc = __expf(m - RL);
#pragma unroll
    for (int i = 0; i < NR; ++i)
#pragma unroll
      for (int j = 0; j < NB; ++j) acc[i][j] *= wc;
    state_update<HD>(acc, buf + Ly::B_K, buf + Ly::B_V, es, ty, tx);
    if (tid < HD) {
      zn *= wc;
      for (int s = 0; s < CL; ++s) zn = fmaf(es[s], buf[Ly::B_K + s * Ly::QS + tid], zn);
    }
    m = sc[1] + RL;
    Ft += sc[1];
    __syncthreads();
  }
  float* out = a.seg + ((size_t)lp * (a.nseg - 1) + seg) * Ly::SEG;
#pragma unroll
  for (int i = 0; i < NR; ++i) st_vec<NB>(out + (NR * ty + i) * HH + NB * tx, acc[i]);
  if (tid < HD) out[HD * HH + tid] = zn;
  if (tid == 0) {
    a.seg_scal[((size_t)lp * a.nseg + seg) * 2] = m;
    a.seg_scal[((size_t)lp * a.nseg + seg) * 2 + 1] = Ft;
  }
}

// Chains the segments' states: slot j becomes the state at the start of segment j + 1.
template <int HD>
__global__ void __launch_bounds__(NTM) mlstm_link_kernel(MScanArgs a) {
  using Ly = ChunkLayout<HD>;
  const int lp = blockIdx.y, e = blockIdx.x * NTM + threadIdx.x;
  const int P = a.plen[lp / a.dm.H];
  const int last = P > 0 ? ((P + CL - 1) / CL - 1) / a.n : 0;
  float* seg = a.seg + (size_t)lp * (a.nseg - 1) * Ly::SEG;
  const float* sc = a.seg_scal + (size_t)lp * a.nseg * 2;
  const bool in = e < Ly::SEG;
  float c = 0.f, m = -INFINITY;
  for (int j0 = 0; j0 < last; j0 += 8) {
    float x[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) x[k] = in && j0 + k < last ? seg[(size_t)(j0 + k) * Ly::SEG + e] : 0.f;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      if (j0 + k >= last) break;
      const float mc = sc[2 * (j0 + k)], m1 = m + sc[2 * (j0 + k) + 1];
      const float mn = fmaxf(m1, mc);
      c = expf(m1 - mn) * c + expf(mc - mn) * x[k];
      m = mn;
      if (in) seg[(size_t)(j0 + k) * Ly::SEG + e] = c;
      if (e == 0) a.seg_m[(size_t)lp * a.nseg + j0 + k + 1] = m;
    }
  }
}

// Readout of one segment.  Threads 0-255 form S = q~ K^T, then the state update; threads
// 256-511 the products with the state, then W V and the scores, so the two halves of a
// chunk's FMAs run side by side.
template <int HD>
__global__ void __launch_bounds__(NTC, 1) mlstm_chunk_kernel(MScanArgs a) {
  using Ly = ChunkLayout<HD>;
  constexpr int HH = Ly::HH, QS = Ly::QS, VS = Ly::VS, WS = Ly::WS;
  constexpr int NB = HD / 32, NR = HD / 16;      // columns, rows of the state per thread
  const Dims& dm = a.dm;
  const int D = dm.D, H = dm.H, NF = a.NF;
  const int lp = blockIdx.y, bl = lp / H, h = lp - bl * H;
  const int P = a.plen[bl];
  const int seg = blockIdx.x, c0 = seg * a.n, nch = (P + CL - 1) / CL;
  if (seg > 0 && c0 >= nch) return;
  const int c1 = min(c0 + a.n, nch);
  const bool last = c1 == nch;
  const size_t Pm = a.Pmax;
  const int tid = threadIdx.x, lane = tid & 31;
  const bool front = tid < 256;
  const int gt = tid & 255, ty = gt >> 4, tx = gt & 15;
  extern __shared__ __align__(16) float smf[];
  float* Cs = smf + 2 * Ly::BUF;                 // [HD][VS]  state C
  float* Ws = Cs + HD * VS;                      // [CL][WS]  W_ts
  float* zs = Ws + CL * WS;                      // [HD]
  float* gs = zs + HD;                           // [CL] g_s
  float* Rs = gs + CL;                           // [CL] R_t
  float* es = Rs + CL;                           // [CL] e^{g_s - R_{L-1}}
  float* qz = es + CL;                           // [CL] q~ . z
  float* sc = qz + CL;                           // [4] m, F_{L-1}, R_{L-1}
  const float* F = a.feat + (size_t)lp * Pm * NF;
  float* prio = a.prio + (size_t)lp * Pm;
  if (c0 < c1) load_chunk<HD, true>(F, NF, c0 * CL, P, D, smf, NTC);
  cp_commit();
  {
    const float* s0 = seg > 0 ? a.seg + ((size_t)lp * (a.nseg - 1) + seg - 1) * Ly::SEG : nullptr;
    for (int e = tid; e < HD * (HH / 4); e += NTC) {
      const int r = e / (HH / 4), c = e - r * (HH / 4);
      *reinterpret_cast<float4*>(Cs + r * VS + 4 * c) =
          s0 ? *reinterpret_cast<const float4*>(s0 + r * HH + 4 * c) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    for (int e = tid; e < HD; e += NTC) zs[e] = s0 ? s0[HD * HH + e] : 0.f;
    if (tid == 0) sc[0] = seg > 0 ? a.seg_m[(size_t)lp * a.nseg + seg] : -INFINITY;
  }
  float av[NB];
#pragma unroll
  for (int j = 0; j < NB; ++j) av[j] = a.ms.a[(size_t)h * HH + NB * tx + j];
  const float bsc = a.ms.b[h];

  for (int ch = c0; ch < c1; ++ch) {
    const int t0 = ch * CL;
    const float* buf = smf + ((ch - c0) & 1) * Ly::BUF;
    const float* Qs = buf + Ly::B_Q;
    const float* Ks = buf + Ly::B_K;
    const float* Vs = buf + Ly::B_V;
    if (ch + 1 < c1) load_chunk<HD, true>(F, NF, t0 + CL, P, D, smf + ((ch + 1 - c0) & 1) * Ly::BUF, NTC);
    cp_commit();
    cp_wait<1>();
    __syncthreads();
    const float m = sc[0];
    float acc[4][4], num[4][NB];
    if (front) {
      // ---- S = q~ K^T ------------------------------------------------------------------
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;
#pragma unroll 4
      for (int c = 0; c < HD; c += 4) {
        float4 qa[4], kb[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) qa[i] = *reinterpret_cast<const float4*>(Qs + (ty + 16 * i) * QS + c);
#pragma unroll
        for (int j = 0; j < 4; ++j) kb[j] = *reinterpret_cast<const float4*>(Ks + (tx + 16 * j) * QS + c);
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int j = 0; j < 4; ++j)
            acc[i][j] = fmaf(qa[i].x, kb[j].x, fmaf(qa[i].y, kb[j].y,
                        fmaf(qa[i].z, kb[j].z, fmaf(qa[i].w, kb[j].w, acc[i][j]))));
      }
    } else {
      if (tid >= NTC - 32) chunk_gates(buf + Ly::B_G, t0, P, m, gs, Rs, es, sc);
      // ---- q~ C and q~ . z --------------------------------------------------------------
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < NB; ++j) num[i][j] = 0.f;
#pragma unroll 2
      for (int c = 0; c < HD; c += 4) {
        float4 qa[4];
        float cr[4][NB];
#pragma unroll
        for (int i = 0; i < 4; ++i) qa[i] = *reinterpret_cast<const float4*>(Qs + (ty + 16 * i) * QS + c);
#pragma unroll
        for (int x = 0; x < 4; ++x) ld_vec<NB>(cr[x], Cs + (c + x) * VS + NB * tx);
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int j = 0; j < NB; ++j)
            num[i][j] = fmaf(qa[i].x, cr[0][j], fmaf(qa[i].y, cr[1][j],
                        fmaf(qa[i].z, cr[2][j], fmaf(qa[i].w, cr[3][j], num[i][j]))));
      }
      // warp w of the group takes rows 8w .. 8w + 7
      const int w8 = gt >> 5;
#pragma unroll
      for (int rr = 0; rr < CL / 8; ++rr) {
        const int t = w8 * (CL / 8) + rr;
        float s = 0.f;
        for (int c = lane; c < HD; c += 32) s = fmaf(Qs[t * QS + c], zs[c], s);
        s = warp_sum(s);
        if (lane == 0) qz[t] = s;
      }
    }
    __syncthreads();                 // gates known; C and z read
    if (front) {
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int t = ty + 16 * i;
        const float R = Rs[t];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const int s = tx + 16 * j;
          Ws[t * WS + s] = (s <= t) ? __expf(gs[s] - R) * acc[i][j] : 0.f;
        }
      }
    }
    __syncthreads();                 // W written
    if (!front) {
      // ---- readout rows: num = e^{m-R} q~C + W V, den = e^{m-R} q~.z + sum_s W ----------
      float den[4], coef[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        coef[i] = __expf(m - Rs[ty + 16 * i]);
        den[i] = 0.f;
#pragma unroll
        for (int j = 0; j < NB; ++j) num[i][j] *= coef[i];
      }
#pragma unroll 4
      for (int s = 0; s < CL; s += 4) {
        float4 wa[4];
        float v[4][NB];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          wa[i] = *reinterpret_cast<const float4*>(Ws + (ty + 16 * i) * WS + s);
          den[i] += (wa[i].x + wa[i].y) + (wa[i].z + wa[i].w);
        }
#pragma unroll
        for (int x = 0; x < 4; ++x) ld_vec<NB>(v[x], Vs + (s + x) * VS + NB * tx);
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int j = 0; j < NB; ++j)
            num[i][j] = fmaf(wa[i].x, v[0][j], fmaf(wa[i].y, v[1][j],
                        fmaf(wa[i].z, v[2][j], fmaf(wa[i].w, v[3][j], num[i][j]))));
      }
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int t = ty + 16 * i;
        const float dn = fmaf(coef[i], qz[t], den[i]);
        float r = 0.f;
#pragma unroll
        for (int j = 0; j < NB; ++j) {
          const float hv = num[i][j] / dn;
          r = fmaf(av[j], hv / (1.f + expf(-hv)), r);
        }
#pragma unroll
        for (int o = 1; o < 16; o <<= 1) r += __shfl_xor_sync(0xffffffffu, r, o);
        const int T = t0 + t, u = T - D;
        if (tx == 0 && T < P && u >= 0) {
          float rv = r + bsc;
          if (a.override_) rv = a.override_[(size_t)lp * Pm + u];
          prio[u] = static_priority(canon_score(rv), u, a.st.log_gamma, h);
        }
      }
    } else if (last || ch + 1 < c1) {
      // ---- state update C' = e^{m-R_L} C + K^T diag(e^{g-R_L}) V;  z likewise -------------
      const float RL = sc[2], wc = __expf(m - RL);
      float cn[NR][NB];
#pragma unroll
      for (int i = 0; i < NR; ++i) {
        ld_vec<NB>(cn[i], Cs + (NR * ty + i) * VS + NB * tx);
#pragma unroll
        for (int j = 0; j < NB; ++j) cn[i][j] *= wc;
      }
      state_update<HD>(cn, Ks, Vs, es, ty, tx);
#pragma unroll
      for (int i = 0; i < NR; ++i) st_vec<NB>(Cs + (NR * ty + i) * VS + NB * tx, cn[i]);
      if (gt < HD) {
        float zn = wc * zs[gt];
        for (int s = 0; s < CL; ++s) zn = fmaf(es[s], Ks[s * QS + gt], zn);
        zs[gt] = zn;
      }
      if (gt == 0) sc[3] = sc[1] + RL;
    }
    __syncthreads();                 // the chunk is done: its buffer, W and the gates are free
    if (tid == 0) sc[0] = sc[3];
  }
  cp_wait<0>();
  __syncthreads();
  if (!last) return;
  const int pair = (a.first_seq + bl) * H + h;
  float* Cg = a.ms.C + (size_t)pair * HD * HH;
  for (int e = tid; e < HD * HH; e += NTC) Cg[e] = Cs[(e / HH) * VS + (e % HH)];
  for (int e = tid; e < HD; e += NTC) a.ms.z[(size_t)pair * HD + e] = zs[e];
  if (tid == 0) a.ms.m[pair] = sc[0];
}

template <int HD>
size_t chunk_smem() {
  using Ly = ChunkLayout<HD>;
  return (size_t)(2 * Ly::BUF + HD * Ly::VS + CL * Ly::WS + HD + 4 * CL + 4) * 4;
}
template <int HD>
size_t seg_smem() { return (size_t)2 * ChunkLayout<HD>::BUF_S * 4; }

// Chunks per segment: one (no state is updated twice) while the states between segments stay
// below 256 MB, else as many as that takes; all of a prompt's (no states between) where the caller
// has no room for them.
int seg_chunks(int d, int pairs, int Pmax, bool one_segment) {
  if (one_segment) return std::max(1, (Pmax + CL - 1) / CL);
  const double bytes = (double)pairs * ((Pmax + CL - 1) / CL) * (d * (d / 2) + d) * 4.0;
  return std::max(1, (int)(bytes / 256e6) + 1);
}
int seg_count(int d, int pairs, int Pmax, bool one_segment) {
  const int nch = (Pmax + CL - 1) / CL, n = seg_chunks(d, pairs, Pmax, one_segment);
  return std::max(1, (nch + n - 1) / n);
}

template <int HD>
cudaError_t launch_scan(MScanArgs sa, int pairs, cudaStream_t stream) {
  if (sa.nseg > 1) {
    mlstm_seg_kernel<HD><<<dim3(sa.nseg - 1, pairs), NTM, seg_smem<HD>(), stream>>>(sa);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    mlstm_link_kernel<HD><<<dim3((ChunkLayout<HD>::SEG + NTM - 1) / NTM, pairs), NTM, 0, stream>>>(sa);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  mlstm_chunk_kernel<HD><<<dim3(sa.nseg, pairs), NTC, chunk_smem<HD>(), stream>>>(sa);
  return cudaGetLastError();
}

template <int HD>
cudaError_t launch_proj_tc(const MlstmDev& m, const void* K, const void* V, const int32_t* plen, int pairs,
                           int H, int Pmax, float* feat, int32_t* err, cudaStream_t stream) {
  MProjTcArgs a{static_cast<const bf16*>(K), static_cast<const bf16*>(V), static_cast<const bf16*>(m.Wt),
                m.bi, m.bf, plen, feat, err, H, Pmax};
  mlstm_proj_tc_kernel<HD><<<dim3((Pmax + PT_TOK - 1) / PT_TOK, pairs), PT_THREADS, PtP<HD>::SMEM, stream>>>(a);
  return cudaGetLastError();
}

}  // namespace

int mlstm_nc(int d) { return ((3 * (d / 2) + 2) + 3) & ~3; }
int mlstm_nf(int d) { return ((2 * d + d / 2 + 2) + 3) & ~3; }
size_t mlstm_wt_bytes(int d, int H) {
  return d == 128 ? (size_t)H * PtP<128>::NKC * PtP<128>::WB : (size_t)H * PtP<64>::NKC * PtP<64>::WB;
}
cudaError_t launch_mlstm_split(const Dims& dm, const MlstmDev& m, cudaStream_t stream) {
  bf16* wt = static_cast<bf16*>(m.Wt);
  if (dm.d == 128) mlstm_split_kernel<128><<<512, 256, 0, stream>>>(m.Wcat, m.NC, dm.H, wt);
  else mlstm_split_kernel<64><<<512, 256, 0, stream>>>(m.Wcat, m.NC, dm.H, wt);
  return cudaGetLastError();
}
// Workspace of the prompt scores: every token's features, then the segments' states and scalars.
size_t mlstm_prefill_bytes(int d, int pairs, int Pmax, bool one_segment) {
  const size_t nseg = seg_count(d, pairs, Pmax, one_segment);
  return ((size_t)pairs * Pmax * mlstm_nf(d) + (size_t)pairs * (nseg - 1) * (d * (d / 2) + d) +
          3 * (size_t)pairs * nseg) * 4;
}

static MState to_mstate(const MlstmDev& m) {
  MState s;
  s.C = m.C; s.z = m.z; s.m = m.m; s.Wcat = m.Wcat; s.bi = m.bi; s.bf = m.bf; s.a = m.a; s.b = m.b;
  s.NC = m.NC;
  return s;
}

cudaError_t prepare_mlstm(const Dims& dm) {
  const int NC = mlstm_nc(dm.d);
  const int esz = dm.dtype == KVPOP_F32 ? 4 : 2;
  const int ism = (int)mlstm_ingest_smem(dm.d, NC, esz);
  const int psm = (int)((size_t)2 * dm.d * UTM * 4 + (size_t)UTM * NC * 4);
  cudaError_t e;
  if (dm.dtype == KVPOP_F32) {
    e = raise_smem_limit(ingest_mlstm_kernel<float>, ism);
    if (e == cudaSuccess) e = raise_smem_limit(mlstm_proj_kernel, psm);
  } else {
    e = raise_smem_limit(ingest_mlstm_kernel<bf16>, ism);
  }
  auto raise = [&](auto* chunk, size_t cs, auto* segk, size_t ss, auto* pk, size_t ps) {
    if (e == cudaSuccess) e = raise_smem_limit(chunk, cs);
    if (e == cudaSuccess) e = raise_smem_limit(segk, ss);
    if (e == cudaSuccess) e = raise_smem_limit(pk, ps);
  };
  if (dm.d == 128)
    raise(mlstm_chunk_kernel<128>, chunk_smem<128>(), mlstm_seg_kernel<128>, seg_smem<128>(),
          mlstm_proj_tc_kernel<128>, PtP<128>::SMEM);
  else
    raise(mlstm_chunk_kernel<64>, chunk_smem<64>(), mlstm_seg_kernel<64>, seg_smem<64>(),
          mlstm_proj_tc_kernel<64>, PtP<64>::SMEM);
  return e;
}

bool mlstm_ok(const Dims& dm) {
  const int esz = dm.dtype == KVPOP_F32 ? 4 : 2;
  return mlstm_ingest_smem(dm.d, mlstm_nc(dm.d), esz) <= 227 * 1024;
}

cudaError_t launch_ingest_mlstm(const State& st, const Dims& dm, const MlstmDev& m, const void* q,
                                const void* k, const void* v, const float* override_,
                                int32_t* evict_info, float* score_out, cudaStream_t stream) {
  dim3 grid((dm.batch + SBM - 1) / SBM, dm.H);
  const int esz = dm.dtype == KVPOP_F32 ? 4 : 2;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.gridDim = grid;
  cfg.blockDim = dim3(NTM);
  cfg.dynamicSmemBytes = mlstm_ingest_smem(dm.d, m.NC, esz);
  cfg.stream = stream;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if (dm.dtype == KVPOP_F32) {
    MIngestArgs<float> a{st, dm, to_mstate(m), (const float*)q, (const float*)k, (const float*)v,
                         override_, evict_info, score_out};
    return cudaLaunchKernelEx(&cfg, ingest_mlstm_kernel<float>, a);
  }
  MIngestArgs<bf16> a{st, dm, to_mstate(m), (const bf16*)q, (const bf16*)k, (const bf16*)v,
                      override_, evict_info, score_out};
  return cudaLaunchKernelEx(&cfg, ingest_mlstm_kernel<bf16>, a);
}

cudaError_t launch_prefill_mlstm_scores(const State& st, const Dims& dm, const MlstmDev& m,
                                        const void* K, const void* V, const int32_t* plen,
                                        int first_seq, int n_seq, int Pmax, const float* override_,
                                        float* feat, bool one_segment, float* prio,
                                        cudaStream_t stream) {
  const int NF = mlstm_nf(dm.d);
  const int pairs = n_seq * dm.H;
  if (Pmax > 0) {
    cudaError_t e;
    if (dm.dtype == KVPOP_F32) {
      const size_t psm = (size_t)2 * dm.d * UTM * 4 + (size_t)UTM * m.NC * 4;
      MProjArgs a{dm, to_mstate(m), (const float*)K, (const float*)V, plen, feat, Pmax, NF};
      mlstm_proj_kernel<<<dim3((Pmax + UTM - 1) / UTM, pairs), NTM, psm, stream>>>(a);
      e = cudaGetLastError();
    } else {
      e = dm.d == 128 ? launch_proj_tc<128>(m, K, V, plen, pairs, dm.H, Pmax, feat, st.err, stream)
                      : launch_proj_tc<64>(m, K, V, plen, pairs, dm.H, Pmax, feat, st.err, stream);
    }
    if (e != cudaSuccess) return e;
  }
  MScanArgs sa{st, dm, to_mstate(m), plen, feat, override_, prio, nullptr, nullptr, nullptr, first_seq, Pmax, NF,
               seg_chunks(dm.d, pairs, Pmax, one_segment), seg_count(dm.d, pairs, Pmax, one_segment)};
  sa.seg = feat + (size_t)pairs * Pmax * NF;
  sa.seg_scal = sa.seg + (size_t)pairs * (sa.nseg - 1) * (dm.d * (dm.d / 2) + dm.d);
  sa.seg_m = sa.seg_scal + (size_t)2 * pairs * sa.nseg;
  return dm.d == 128 ? launch_scan<128>(sa, pairs, stream) : launch_scan<64>(sa, pairs, stream);
}

}  // namespace kvpop
