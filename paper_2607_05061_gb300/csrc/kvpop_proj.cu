// Projections of the decode stack: y = bf16(x W) for a few rows x (one per sequence), as one
// launch for W_q, W_k and W_v, and x' = bf16(x + bf16(bf16(o) W_o)) as one launch from the
// attention's fp32 output (the bf16 storage points of the layer stack).
//
// Bound by the stream of the weights.  One CTA per SM owns up to 6 groups of 8 output columns
// over the whole contraction, so nothing is exchanged between CTAs.  Each of its 8 warps takes
// its own part of the contraction through a private ring of cp.async stages (32 weight rows of
// up to 96 bytes, and the same 32 columns of x), with no barrier until the warps' fp32 sums
// meet in shared memory at the end, in warp order.  While the kernel before this one still runs,
// the first stages' weights go to L2, which is only a hint and so needs no order with a kernel
// that may write them, and into the ring after griddepcontrol.wait; weights that the caller
// states to be settled go into the ring at once (hidden 4096, batch 1: 11.6 us, 12.7 otherwise).
// The next kernel may start after that wait, and so after all that came before this one.  The
// products run on mma.sync with the weights as the 16-row operand and the sequences as the
// 8-column one: at so few rows the tensor work is far below the stream.
// Device time at hidden 4096, 32 query and 8 KV heads, alone and cold: q, k, v at 1 to 8 rows
// 14 us (7.5 us at the copy rate) against 32 us of cuBLAS's six launches, the output 13 us
// (5 us) against 18 us of four; a 4-layer step at batch 1 230 -> 198 us, at batch 8 284 -> 245.
#include <algorithm>

#include "kvpop_mma.cuh"
#include "kvpop_ptx.cuh"

namespace kvpop {
namespace {

constexpr int PJ_NW = 8;
constexpr int PJ_NT = PJ_NW * 32;
constexpr int PJ_NG = 6;               // column groups of 8 per CTA at most
constexpr int PJ_KS = 32;              // weight rows per stage
constexpr int PJ_WROW = 112;           // bytes of a staged weight row: 96 and a pad (conflict-free)
constexpr int PJ_WST = PJ_KS * PJ_WROW;

struct ProjArgs {
  const void* x;                       // [M][K] bf16, or fp32 rounded to bf16 on use (XF32)
  const bf16* W[3];                    // [K][N[i]] row-major
  bf16* y[3];                          // [M][N[i]]
  const bf16* res;                     // [M][N[0]] added after the rounding, or null
  int groups[3];                       // column groups up to and including matrix i
  int N[3];
  int M, K;
  int settled;                         // nothing that may still run writes the weights
};

template <int MT, bool XF32>
struct PjP {
  static constexpr int XROW = PJ_KS * (XF32 ? 4 : 2);              // bytes of a staged row of x
  static constexpr int STAGE = PJ_WST + 8 * MT * XROW;
  // 4 stages: more than half of the shared memory, so that an early launch cannot put two CTAs
  // of the grid on one SM (2 or 3 stages: a 4-layer step at batch 1 takes 240 and 233 us, 198
  // with 4, 201 with 6)
  static constexpr int ST = std::min(4, 200 * 1024 / (PJ_NW * STAGE));
  static constexpr int RED = PJ_NW * PJ_NG * 8 * 8 * MT * 4;       // the warps' sums
  static constexpr int SMEM = std::max(PJ_NW * ST * STAGE, RED);
  static_assert(ST >= 2, "");
};

// MT: 8-row groups of x (M <= 8 MT).
template <int MT, bool XF32>
__global__ void __launch_bounds__(PJ_NT, 1) proj_kernel(ProjArgs a) {
  using P = PjP<MT, XF32>;
  extern __shared__ __align__(128) unsigned char sm_pj[];
  constexpr int ST = P::ST;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int K = a.K, total = a.groups[2];
  const int c0 = (int)((long long)blockIdx.x * total / gridDim.x);
  const int ng = (int)((long long)(blockIdx.x + 1) * total / gridDim.x) - c0;
  // group j of the CTA: matrix and first column (a CTA's groups lie in at most two matrices)
  auto column = [&](int j, int& m) {
    const int c = c0 + j;
    m = c < a.groups[0] ? 0 : c < a.groups[1] ? 1 : 2;
    return (c - (m ? a.groups[m - 1] : 0)) * 8;
  };

  // the warp's stages of the contraction
  const int nst = K / PJ_KS;
  const int s0 = warp * nst / PJ_NW, ns = (warp + 1) * nst / PJ_NW - s0;
  unsigned char* ring = sm_pj + (size_t)warp * ST * P::STAGE;
  const uint32_t rb = smem_u32(ring);
  // this lane's 16-byte pieces of a stage's weights: piece i = row i / ng, group i % ng
  const bf16* src[PJ_NG];
  uint32_t dst[PJ_NG];
  size_t step[PJ_NG];
#pragma unroll
  for (int j = 0; j < PJ_NG; ++j) {
    const int i = j * 32 + lane, row = i / ng, grp = i - row * ng;
    int m;
    const int col = column(j < ng ? grp : 0, m);
    src[j] = a.W[m] + (size_t)(s0 * PJ_KS + row) * a.N[m] + col;
    step[j] = (size_t)PJ_KS * a.N[m];
    dst[j] = (uint32_t)(row * PJ_WROW + grp * 16);
  }
  auto load_w = [&](int s) {           // stage s of the warp
    const uint32_t base = rb + (s % ST) * P::STAGE;
#pragma unroll
    for (int j = 0; j < PJ_NG; ++j)
      if (j < ng) {
        cp_async16(base + dst[j], src[j], 16);
        src[j] += step[j];
      }
  };
  constexpr int XC = P::XROW / 16;     // 16-byte pieces of a staged row of x
  const unsigned char* xg = static_cast<const unsigned char*>(a.x);
  auto load_x = [&](int s) {
    const uint32_t base = rb + (s % ST) * P::STAGE + PJ_WST;
    const size_t at = (size_t)(s0 + s) * P::XROW;
#pragma unroll
    for (int i = lane; i < 8 * MT * XC; i += 32) {
      const int m = i / XC, c = i - m * XC;
      const int sw = XF32 ? c ^ (m & 7) : c ^ ((m >> 1) & 3);
      cp_async16(base + m * P::XROW + sw * 16, xg + (size_t)(m < a.M ? m : 0) * K * (P::XROW / PJ_KS) + at + c * 16,
                 m < a.M ? 16 : 0);
    }
  };
  if (a.settled) {
#pragma unroll
    for (int s = 0; s < ST; ++s)
      if (s < ns) load_w(s);
  } else {
#pragma unroll
    for (int s = 0; s < ST; ++s)
#pragma unroll
      for (int j = 0; j < PJ_NG; ++j)
        if (s < ns && j < ng) prefetch_l2_line(src[j] + s * step[j]);
  }
  cp_commit();
  asm volatile("griddepcontrol.wait;" ::: "memory");
  // a kernel that starts from here on starts after all that precedes this one
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  if (!a.settled) {
#pragma unroll
    for (int s = 0; s < ST; ++s)
      if (s < ns) load_w(s);
  }
#pragma unroll
  for (int s = 0; s < ST; ++s) {
    if (s < ns) load_x(s);
    cp_commit();
  }

  const int g = lane >> 2, t4 = lane & 3;
  float acc[3][MT][4];
#pragma unroll
  for (int n = 0; n < 3; ++n)
#pragma unroll
    for (int m = 0; m < MT; ++m) acc[n][m][0] = acc[n][m][1] = acc[n][m][2] = acc[n][m][3] = 0.f;
  for (int s = 0; s < ns; ++s) {
    cp_wait<ST - 1>();                 // the groups of the stages after this one may be in flight
    __syncwarp();
    const uint32_t wb = rb + (s % ST) * P::STAGE, xb = wb + PJ_WST;
    uint32_t b[MT][4];                 // x: k 0-7, 8-15, 16-23, 24-31 of the stage
#pragma unroll
    for (int m = 0; m < MT; ++m) {
      if constexpr (XF32) {
        const unsigned char* xr = ring + (s % ST) * P::STAGE + PJ_WST + (8 * m + g) * P::XROW;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const float2 v = *reinterpret_cast<const float2*>(xr + (((2 * k + (t4 >> 1)) ^ g) * 16) + (t4 & 1) * 8);
          b[m][k] = pack_bf16(v.x, v.y);
        }
      } else {
        const int row = 8 * m + (lane & 7);
        ldsm_x4(xb + row * P::XROW + (((lane >> 3) ^ ((row >> 1) & 3)) << 4), b[m][0], b[m][1], b[m][2], b[m][3]);
      }
    }
#pragma unroll
    for (int kk = 0; kk < 2; ++kk) {
      const uint32_t wr = wb + (16 * kk + (lane & 7) + ((lane >> 4) & 1) * 8) * PJ_WROW + ((lane >> 3) & 1) * 16;
#pragma unroll
      for (int n = 0; n < 3; ++n) {
        if (2 * n >= ng) break;
        uint32_t w0, w1, w2, w3;
        ldsm_x4_t(wr + n * 32, w0, w1, w2, w3);
#pragma unroll
        for (int m = 0; m < MT; ++m) mma_bf16(acc[n][m], w0, w1, w2, w3, b[m][2 * kk], b[m][2 * kk + 1]);
      }
    }
    __syncwarp();                      // every lane has read the stage
    if (s + ST < ns) {
      load_w(s + ST);
      load_x(s + ST);
    }
    cp_commit();
  }
  cp_wait<0>();
  __syncthreads();                     // the rings are free
  constexpr int MP = 8 * MT;
  float* red = reinterpret_cast<float*>(sm_pj);              // [warp][48 columns][MP]
#pragma unroll
  for (int n = 0; n < 3; ++n)
#pragma unroll
    for (int m = 0; m < MT; ++m) {
      float* p = red + ((size_t)warp * PJ_NG * 8 + 16 * n + g) * MP + 8 * m + 2 * t4;
      *reinterpret_cast<float2*>(p) = make_float2(acc[n][m][0], acc[n][m][1]);
      *reinterpret_cast<float2*>(p + 8 * MP) = make_float2(acc[n][m][2], acc[n][m][3]);
    }
  __syncthreads();
  for (int i = tid; i < 8 * ng * a.M; i += PJ_NT) {
    const int m = i / (8 * ng), c = i - m * 8 * ng;
    float sum = 0.f;
#pragma unroll
    for (int w = 0; w < PJ_NW; ++w) sum += red[((size_t)w * PJ_NG * 8 + c) * MP + m];
    int mat;
    const int col = column(c >> 3, mat) + (c & 7);
    const size_t at = (size_t)m * a.N[mat] + col;
    bf16 o = __float2bfloat16_rn(sum);
    if (a.res) o = __float2bfloat16_rn(__bfloat162float(a.res[at]) + __bfloat162float(o));
    a.y[mat][at] = o;
  }
}

template <int MT, bool XF32>
cudaError_t launch_proj_t(const ProjArgs& a, cudaStream_t stream) {
  using P = PjP<MT, XF32>;
  int dev = 0, sms = 152;
  if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  cudaError_t e = raise_smem_limit(proj_kernel<MT, XF32>, P::SMEM);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)std::max(std::min(sms, a.groups[2]), (a.groups[2] + PJ_NG - 1) / PJ_NG));
  cfg.blockDim = dim3(PJ_NT);
  cfg.dynamicSmemBytes = P::SMEM;
  cfg.stream = stream;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, proj_kernel<MT, XF32>, a);
}

template <bool XF32>
cudaError_t launch_proj(const ProjArgs& a, cudaStream_t stream) {
  if (a.M <= 8) return launch_proj_t<1, XF32>(a, stream);
  if constexpr (!XF32)
    if (a.M > 16) return launch_proj_t<4, XF32>(a, stream);
  return launch_proj_t<2, XF32>(a, stream);
}

}  // namespace

// Rows, contraction and column counts the kernel takes: whole stages, whole column groups, and
// matrices wide enough that a CTA's groups lie in at most two.  Every CTA reads all of x, in
// fp32 twice the bytes, so the rows end where that traffic outweighs what the launch saves:
// at 32 rows (hidden 4096) q, k, v take 21 us in one launch against 32 in cuBLAS's five, the
// output 24 us against 18 in cuBLAS's product, the rounding copy and the sum.
bool proj_ok(int M, int K, int N, bool x_f32) {
  return M >= 1 && M <= (x_f32 ? 16 : 32) && K >= PJ_KS && K % PJ_KS == 0 && N >= 8 * PJ_NG && N % 8 == 0;
}

// Where the kernel is the faster way, of the sizes it takes.  Its columns have to fit the SMs at
// once: a CTA holds an SM for its part of the columns, so a second wave leaves most of the SMs idle
// (a layer of hidden 8192 with 64 query and 16 KV heads at batch 1 and 16, cuBLAS / q, k, v here /
// the output here: 82 / 84 / 95 us and 108 / 116 / 128; with 7168 and 56 heads, 1344 and 896 column
// groups for 912 places, 76 / 77 / 75 at batch 1).  Within that q, k, v are faster throughout (hidden
// 8192, 32 heads, batch 16: 79.5 / 79.6; batch 1: 65.7 / 59.5).  For the output every CTA reads all
// rows of fp32 x through L2, and more of them than 2^16 values cost what the launches save (8192
// wide, batch 8: 79.9 / 77.7 us a layer, batch 16: 99.0 / 101.3).
bool proj_faster(int M, int K, int columns, bool x_f32) {
  int dev = 0, sms = 152;
  if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  cudaGetLastError();                  // no device: the rule for GB300
  return columns / 8 <= PJ_NG * sms && (!x_f32 || (long long)M * K <= 1 << 16);
}

cudaError_t launch_proj_qkv(const void* x, const void* Wq, const void* Wk, const void* Wv, int M, int K,
                            int nq, int nkv, void* q, void* k, void* v, bool settled, cudaStream_t stream) {
  ProjArgs a{};
  a.settled = settled;
  a.x = x;
  const void* W[3] = {Wq, Wk, Wv};
  void* y[3] = {q, k, v};
  const int N[3] = {nq, nkv, nkv};
  for (int i = 0, t = 0; i < 3; ++i) {
    a.W[i] = static_cast<const bf16*>(W[i]);
    a.y[i] = static_cast<bf16*>(y[i]);
    a.N[i] = N[i];
    a.groups[i] = t += N[i] / 8;
  }
  a.M = M;
  a.K = K;
  return launch_proj<false>(a, stream);
}

cudaError_t launch_proj_out(const float* o, const void* Wo, const void* res, int M, int K, int N,
                            void* y, bool settled, cudaStream_t stream) {
  ProjArgs a{};
  a.settled = settled;
  a.x = o;
  a.W[0] = static_cast<const bf16*>(Wo);
  a.y[0] = static_cast<bf16*>(y);
  a.res = static_cast<const bf16*>(res);
  a.N[0] = N;
  a.groups[0] = a.groups[1] = a.groups[2] = N / 8;
  a.M = M;
  a.K = K;
  return launch_proj<true>(a, stream);
}

}  // namespace kvpop
