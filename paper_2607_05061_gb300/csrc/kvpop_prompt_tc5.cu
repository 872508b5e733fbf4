// Masked prompt attention on the 5th-generation tensor cores (tcgen05), bf16
// with head dimension 128 (App. C.1 mask, App. C.3).
//
// Same key lists as the m16n8k16 kernel (kvpop_prompt.cu), built for 256 / G
// consecutive queries of one (sequence, KV head): the CTA's 256 (query, head)
// rows form two 128-row halves that share every gathered K/V block, so each
// gathered byte feeds two M = 128 MMAs.  Roles:
//  * 3 producer warps gather the block's K and V rows by position with 16-byte
//    cp.async into 128B-swizzled tiles (2 to 4 stages, as shared memory
//    allows); completion arrives on the stage's mbarrier asynchronously
//    (cp.async.mbarrier.arrive.noinc).
//  * 1 MMA warp: one lane issues, per half, S = Q K^T (M 128, N 64, K 128;
//    Q and K K-major) into one of two tensor-memory S buffers, and O += P V
//    (M 128, N 128, K 64; P from tensor memory, V read MN-major straight
//    from its gathered rows) into the half's tensor-memory accumulator;
//    tcgen05.commit signals S ready, P consumed and the stage free.  Tensor
//    memory: O of both halves (256 columns) and their S double buffers (256).
//  * 2 softmax warpgroups, one per half, one thread per row: read the row of S
//    (32x32b loads), apply the mask on the few blocks that need it, keep a
//    running maximum that is only raised when a logit exceeds it by 2^8 (the
//    row of the accumulator is then rescaled in place), write the bf16
//    probabilities over the row's logits and hand them over.  (S_{j+2} follows
//    PV_j into the buffer, in the order the MMAs are issued.)
// What bounds it: the shared-memory bytes of a 64-key block (query tile and keys of S 96 KB,
// values 32, the gathered rows written 32: 1250 clocks at 128 bytes each) and the tensor unit
// (1280) are both close to the 1700 clocks it takes; a tile's prologue and epilogue add about
// 20000.  One 32768-token prompt of 8 heads (4096 keys a query), us: 2768 at first; 2368 with
// the MMA warp's operands kept warp-uniform; 2053 with the mask reduced to a run of queries per
// key and the longest tiles of all pairs first; 1967 with the prologue's loads in flight
// together and the outputs stored as whole rows; 1833 with P in tensor memory instead of a
// shared tile (64 KB less per block, and a fourth stage).  2 x 8192 tokens with a window of
// 256: 1034 -> 458.
// Outputs as the other kernels: y in fp32 and the natural-log normaliser.
// Every wait is bounded; on expiry the kernel records an error code, stops
// issuing work, lets its copies drain and frees its tensor memory.  Every
// tensor-memory access, and every branch around one, is warp-uniform.
#include "kvpop_mma.cuh"
#include "kvpop_prompt.cuh"
#include "kvpop_ptx.cuh"
#include "kvpop_tc05.cuh"

namespace kvpop {
namespace {

using namespace prompt;
using namespace tc05;

constexpr int T5_HALF = 128;                     // rows per half (MMA M)
constexpr int T5_ROWS = 2 * T5_HALF;             // (query, head) rows per CTA
constexpr int T5_BN = 64;                        // keys per block
constexpr int T5_MMA_WARP = 8;                   // warps 0-7: softmax, 8: MMA, 9-11: producers
constexpr int T5_NPROD = 3;
constexpr int T5_PT = 32 * T5_NPROD;
constexpr int T5_THREADS = 32 * (T5_MMA_WARP + 1 + T5_NPROD);   // 12 warps: 168 registers fit
static_assert(T5_THREADS / 32 + 2 <= 16, "the prologue's per-warp reduction slots");
constexpr int T5_TMEM_COLS = 512;                // O_h: 128 h .. ; S_{h,b}: 256 + 128 h + 64 b
constexpr float T5_THR = 8.0f;
constexpr int T5_POS_BITS = 18;                  // of a packed position

constexpr int QB = T5_HALF * 256;                // Q tile of one half, bytes
constexpr int KVB = T5_BN * 256;                 // K (or V) block, bytes
constexpr int OFF_Q = 0;
constexpr int OFF_KV = OFF_Q + 2 * QB;           // stages of [K | V]
template <int ST>
struct Lay {
  static constexpr int OFF_BAR = OFF_KV + ST * 2 * KVB;
  static constexpr int OFF_TMEM = OFF_BAR + 256;
  static constexpr int OFF_TAU = OFF_TMEM + 16;
  static constexpr int OFF_RED = OFF_TAU + T5_ROWS * 4;
  static constexpr int OFF_LIST = OFF_RED + 16 * 4;
};
// barrier indices
constexpr int B_FULL = 0;          // [4]  producers -> MMA
constexpr int B_EMPTY = 4;         // [4]  MMA -> producers
constexpr int B_SFULL = 8;         // [2 halves][2 buffers]  MMA -> softmax
constexpr int B_PFULL = 12;        // [2][2]  softmax -> MMA
constexpr int B_ODONE = 16;        // [2]  MMA -> softmax (one per half)
constexpr int B_QFULL = 18;
enum : int { T5ERR_WAIT = 21 };

// PACK: an M entry's position and the length of its run of queries share a word (below), so that
// long windows keep their lists in shared memory once.
template <int G, int ST, bool PACK>
__global__ void __launch_bounds__(T5_THREADS, 1) prompt_t5_kernel(PromptArgs a) {
  using L = Lay<ST>;
  constexpr int BM = T5_ROWS / G;
  extern __shared__ __align__(1024) unsigned char sm5[];
  const uint32_t sb = smem_u32(sm5);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  auto bar = [&](int i) { return sb + L::OFF_BAR + 8u * (uint32_t)i; };
  int* tauS = reinterpret_cast<int*>(sm5 + L::OFF_TAU);
  int* red = reinterpret_cast<int*>(sm5 + L::OFF_RED);
  int32_t* posA = reinterpret_cast<int32_t*>(sm5 + L::OFF_LIST);
  int32_t* posM = posA + a.capA;
  uint32_t* keepM = reinterpret_cast<uint32_t*>(PACK ? posM : posM + a.capM);   // [capM + T5_BN]

  if (tid == 0) {
    for (int i = 0; i < ST; ++i) {
      mbar_init(bar(B_FULL + i), T5_PT);
      mbar_init(bar(B_EMPTY + i), 1);
    }
    for (int i = 0; i < 4; ++i) {
      mbar_init(bar(B_SFULL + i), 1);
      mbar_init(bar(B_PFULL + i), T5_HALF / 32);
    }
    mbar_init(bar(B_ODONE + 0), 1);
    mbar_init(bar(B_ODONE + 1), 1);
    mbar_init(bar(B_QFULL), T5_THREADS);
    mbar_fence_init();
  }
  if (warp == T5_MMA_WARP) tmem_alloc(sb + L::OFF_TMEM, T5_TMEM_COLS);
  TileInfo ti;
  // the query rows travel while the key lists are built; their arrival is counted below
  if (tile_bounds(a, BM, ti)) {
    const bf16* Qb = static_cast<const bf16*>(a.Q) + ((size_t)ti.seq * a.H * G + (size_t)ti.h * G) * a.S * 128;
    for (int i = tid; i < T5_ROWS * 16; i += T5_THREADS) {
      const int r = i >> 4, c = i & 15;
      const int q = ti.q0 + r / G, g = r % G;
      const bool ok = q <= ti.q1;
      cp_async16(sb + OFF_Q + (r >> 7) * QB + tile_off(r & 127, c, T5_HALF),
                 Qb + ((size_t)g * a.S + (ok ? q : ti.q0)) * 128 + c * 8, ok ? 16 : 0);
    }
  }
  const bool live = tile_setup<T5_THREADS>(a, BM, tauS, red, posA, posM, ti);
  if (live) {
    cp_async_arrive_noinc(bar(B_QFULL));            // the barriers are set up: a block sync lies between
    // Which queries of the tile keep an M entry: a run that starts at the key's own position and
    // ends where the cutoff falls below its rank (once dropped a key stays dropped), found once
    // per entry as (first query, number) instead of testing the mask for every row.
    const int32_t* rank = a.rank + (size_t)ti.pair * a.S;
    const int nq = ti.q1 - ti.q0 + 1;
    for (int i = tid; i < ti.nM + T5_BN; i += T5_THREADS) {
      uint32_t word = 0;                            // past the list: no query
      if (i < ti.nM) {
        const int t = posM[i], r = __ldg(rank + t);
        const int first = max(0, t - ti.q0);
        int lo = first, hi = nq;                    // the run's end lies in [lo, hi]
        while (lo < hi) {
          const int mid = (lo + hi) >> 1;
          if (keep_key(ti.q0 + mid, t, r, tauS[mid], a.s, a.w)) lo = mid + 1; else hi = mid;
        }
        word = PACK ? (uint32_t)t | (uint32_t)(lo - first) << T5_POS_BITS
                    : (uint32_t)first | (uint32_t)(lo - first) << 16;
      }
      keepM[i] = word;
    }
  }
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = *reinterpret_cast<volatile uint32_t*>(sm5 + L::OFF_TMEM);
  if (live) {
    const int H = a.H, S = a.S, nA = ti.nA, nU = ti.nA + ti.nM;
    const int nblk = (nU + T5_BN - 1) / T5_BN;
    const size_t pair_off = (size_t)ti.pair * S;
    auto entry = [&](int e) -> int {
      constexpr int mask = PACK ? (1 << T5_POS_BITS) - 1 : -1;
      if (e < nA) return posA[e];
      return e < nU ? posM[e - nA] & mask : (nA > 0 ? posA[0] : posM[0] & mask);
    };
    if (warp > T5_MMA_WARP) {
      // ---------------------------------------------------------------- producers
      const int pt = tid - 32 * (T5_MMA_WARP + 1);
      const bf16* Kp = static_cast<const bf16*>(a.K) + pair_off * 128;
      const bf16* Vp = static_cast<const bf16*>(a.V) + pair_off * 128;
      for (int j = 0; j < nblk; ++j) {
        const int st = j % ST;
        if (j >= ST && !mbar_wait(bar(B_EMPTY + st), ((j / ST) - 1) & 1, a.err, T5ERR_WAIT)) break;
        const uint32_t kd = sb + OFF_KV + st * 2 * KVB, vd = kd + KVB;
        // 8 threads per key row, 32 bytes (two 16-byte chunks) of K and of V each:
        // one position lookup per row and thread, rows T5_PT / 8 apart
        const int c2 = 2 * (pt & 7);
#pragma unroll 2
        for (int key = pt >> 3; key < T5_BN; key += T5_PT / 8) {
          const size_t t = (size_t)entry(j * T5_BN + key) * 128 + c2 * 8;
          const uint32_t o0 = tile_off(key, c2, T5_BN), o1 = tile_off(key, c2 + 1, T5_BN);
          cp_async16(kd + o0, Kp + t, 16);
          cp_async16(kd + o1, Kp + t + 8, 16);
          cp_async16(vd + o0, Vp + t, 16);
          cp_async16(vd + o1, Vp + t + 8, 16);
        }
        cp_async_arrive_noinc(bar(B_FULL + st));
      }
      cp_wait<0>();
    } else if (warp == T5_MMA_WARP) {
      // ---------------------------------------------------------------- MMA issue
      // all lanes run the loop, one issues (see elect_one)
      const uint32_t idS = idesc_bf16(128, T5_BN, 0);
      const uint32_t idO = idesc_bf16(128, 128, 1);
      const bool lead = elect_one();
      const uint64_t qd0 = kmajor_desc(sb + OFF_Q, T5_HALF, 0), kd0 = kmajor_desc(sb + OFF_KV, T5_BN, 0);
      const uint64_t vd0 = mnmajor_desc(sb + OFF_KV + KVB, T5_BN, 0);
      bool ok = __all_sync(0xffffffffu, mbar_wait(bar(B_QFULL), 0, a.err, T5ERR_WAIT));
      if (ok) fence_async_smem();
      auto issue_s = [&](int j) {
        const int st = j % ST;
        ok = ok && mbar_wait(bar(B_FULL + st), (j / ST) & 1, a.err, T5ERR_WAIT);
        if (!(ok = __all_sync(0xffffffffu, ok))) return;
        fence_async_smem();
        fence_after();
        if (lead) {
          const uint64_t kd = desc_at(kd0, st * 2 * KVB);
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const uint32_t dS = tmem + 256 + h * 128 + (uint32_t)(j & 1) * T5_BN;
            const uint64_t qd = desc_at(qd0, h * QB);
#pragma unroll
            for (int ks = 0; ks < 8; ++ks)
              mma_bf16(dS, kmajor_step(qd, T5_HALF, ks), kmajor_step(kd, T5_BN, ks), idS, ks > 0);
            commit(bar(B_SFULL + 2 * h + (j & 1)));
          }
        }
        __syncwarp();
      };
      issue_s(0);
      if (nblk > 1) issue_s(1);
      for (int j = 0; j < nblk && ok; ++j) {
        const int st = j % ST;
        const uint64_t vd = desc_at(vd0, st * 2 * KVB);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          ok = ok && mbar_wait(bar(B_PFULL + 2 * h + (j & 1)), (j >> 1) & 1, a.err, T5ERR_WAIT);
          if (!(ok = __all_sync(0xffffffffu, ok))) break;
          fence_after();
          if (lead) {
            const uint32_t tP = tmem + 256 + h * 128 + (uint32_t)(j & 1) * T5_BN;
#pragma unroll
            for (int kk = 0; kk < 4; ++kk)
              mma_bf16_ts(tmem + h * 128, tP + 8 * kk, desc_at(vd, kk * 16 * 128), idO, (j > 0 || kk > 0));
            commit(bar(B_ODONE + h));
            if (h == 1) commit(bar(B_EMPTY + st));
          }
          __syncwarp();
        }
        if (!ok) break;
        if (j + 2 < nblk) issue_s(j + 2);
      }
      __syncwarp();
    } else {
      // ---------------------------------------------------------------- softmax rows
      const int h = warp >> 2;                      // half
      const int r = (warp & 3) * 32 + lane;         // row of the half = tensor-memory lane
      const int rr = h * T5_HALF + r;               // row of the CTA tile
      const int ql = rr / G, g = rr - ql * G;
      const int q = ti.q0 + ql;
      const bool valid = q <= ti.q1;
      const uint32_t trow = (uint32_t)((warp & 3) * 32) << 16;
      const uint32_t tO = tmem + trow + h * 128, tS = tmem + trow + 256 + h * 128;
      const float c2 = a.qscale;
      float m = -INFINITY, l = 0.f;
      bool ok = true;
      auto uniform = [](bool x) { return __all_sync(0xffffffffu, x); };
      for (int j = 0; j < nblk; ++j) {
        const int b = j & 1;
        if (!(ok = uniform(mbar_wait(bar(B_SFULL + 2 * h + b), (j >> 1) & 1, a.err, T5ERR_WAIT))))
          break;
        fence_after();
        float s[64];
        tmem_ld32(tS + b * T5_BN, *reinterpret_cast<float(*)[32]>(s));
        tmem_ld32(tS + b * T5_BN + 32, *reinterpret_cast<float(*)[32]>(s + 32));
        tmem_wait_ld();
        if ((j + 1) * T5_BN > nA) {                 // block holds keys that need the mask
          const int nf = nA - j * T5_BN;            // entries before it need none
#pragma unroll
          for (int i = 0; i < 64; ++i) {
            if (i >= nf) {
              const uint32_t kw = keepM[i - nf];
              const int first = PACK ? max(0, (int)(kw & ((1u << T5_POS_BITS) - 1)) - ti.q0) : (int)(kw & 0xffffu);
              if ((uint32_t)(ql - first) >= (kw >> (PACK ? T5_POS_BITS : 16))) s[i] = -INFINITY;
            }
          }
        }
        // 8 independent chains of three-input maxima (one 64-long chain would serialise)
        float pm[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) pm[k] = s[k];
#pragma unroll
        for (int i = 8; i < 56; i += 16)
#pragma unroll
          for (int k = 0; k < 8; ++k) pm[k] = fmax3(pm[k], s[i + k], s[i + 8 + k]);
#pragma unroll
        for (int k = 0; k < 8; ++k) pm[k] = fmaxf(pm[k], s[56 + k]);
        const float mx = fmax3(fmax3(pm[0], pm[1], pm[2]), fmax3(pm[3], pm[4], pm[5]), fmaxf(pm[6], pm[7]));
        const float mxs = mx * c2;                  // row maximum, log2 units
        float alpha = 1.f, m_new = m;
        bool resc = false;
        if (mxs > m + T5_THR) {
          m_new = mxs;
          alpha = ex2(m - m_new);
          resc = m != -INFINITY;
        }
        const float base = m_new == -INFINITY ? 0.f : m_new;
        // probabilities 2^(s c2 - base): scale-and-shift and the partial sums in packed pairs
        const uint64_t cc = f2_pack(c2, c2), nb = f2_pack(-base, -base);
        uint64_t ps2[4] = {0ull, 0ull, 0ull, 0ull};
#pragma unroll
        for (int i = 0; i < 64; i += 8) {
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            float x0, x1;
            f2_unpack(f2_fma(f2_pack(s[i + 2 * k], s[i + 2 * k + 1]), cc, nb), x0, x1);
            s[i + 2 * k] = ex2(x0);
            s[i + 2 * k + 1] = ex2(x1);
            ps2[k] = f2_add(ps2[k], f2_pack(s[i + 2 * k], s[i + 2 * k + 1]));
          }
        }
        float ps[8];
#pragma unroll
        for (int k = 0; k < 4; ++k) f2_unpack(ps2[k], ps[2 * k], ps[2 * k + 1]);
        const float sum = ((ps[0] + ps[1]) + (ps[2] + ps[3])) + ((ps[4] + ps[5]) + (ps[6] + ps[7]));
        l = l * alpha + sum;
        m = m_new;
        if (j >= 1 && __any_sync(0xffffffffu, resc)) {
          // PV_{j-1} must have landed in O before O changes (PV_{j-2} has: S_j came after it)
          if (!(ok = uniform(mbar_wait(bar(B_ODONE + h), (j - 1) & 1, a.err, T5ERR_WAIT)))) break;
          fence_after();
          const float f = resc ? alpha : 1.f;
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            float o[32];
            tmem_ld32(tO + c * 32, o);
            tmem_wait_ld();
#pragma unroll
            for (int i = 0; i < 32; ++i) o[i] *= f;
            tmem_st32(tO + c * 32, o);
          }
        }
        // the probabilities take the place of their logits, two to a word: the A operand of PV_j
        float pw[32];
#pragma unroll
        for (int i = 0; i < 32; ++i) pw[i] = __uint_as_float(pack_bf16(s[2 * i], s[2 * i + 1]));
        tmem_st32(tS + b * T5_BN, pw);
        tmem_wait_st();
        fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(bar(B_PFULL + 2 * h + b));
      }
      const size_t row = ((size_t)ti.seq * H * G + (size_t)ti.h * G + g) * S + q;
      if (ok && nblk > 0) {
        ok = uniform(mbar_wait(bar(B_ODONE + h), (nblk - 1) & 1, a.err, T5ERR_WAIT));
        fence_after();
        if (ok) {
          // a warp's 32 rows pass through shared memory, so that a store writes one whole row:
          // half 0 in the query tile (every S is done), half 1, whose last product is the last
          // of all, in the first K/V stages
          const float inv = 1.f / l;
          const uint32_t tile = sb + (h ? OFF_KV : OFF_Q) + (warp & 3) * (32 * 512);
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            float o[32];
            tmem_ld32(tO + c * 32, o);
            tmem_wait_ld();
#pragma unroll
            for (int i = 0; i < 8; ++i)
              *reinterpret_cast<float4*>(sm5 + (tile - sb) + lane * 512 + (((c * 8 + i) ^ lane) << 4)) =
                  make_float4(o[4 * i] * inv, o[4 * i + 1] * inv, o[4 * i + 2] * inv, o[4 * i + 3] * inv);
          }
          __syncwarp();
          const int r0 = h * T5_HALF + (warp & 3) * 32;
          float* Yp = a.Y + ((size_t)ti.seq * H * G + (size_t)ti.h * G) * S * 128;
#pragma unroll 8
          for (int i = 0; i < 32; ++i) {
            const int qi = ti.q0 + (r0 + i) / G;
            if (qi > ti.q1) break;
            const float4 v = *reinterpret_cast<const float4*>(sm5 + (tile - sb) + i * 512 + ((lane ^ i) << 4));
            *reinterpret_cast<float4*>(Yp + ((size_t)((r0 + i) % G) * S + qi) * 128 + 4 * lane) = v;
          }
        }
      }
      if (ok && valid && a.lse) a.lse[row] = l > 0.f ? (m + __log2f(l)) * kLn2 : -INFINITY;
    }
  }
  cp_wait<0>();
  fence_before();
  __syncthreads();
  if (warp == T5_MMA_WARP) tmem_dealloc(tmem, T5_TMEM_COLS);
}

template <int ST, bool PACK>
size_t t5_smem(long long capA, long long capM) {
  return (size_t)Lay<ST>::OFF_LIST + (size_t)(capA + (PACK ? 1 : 2) * capM + T5_BN) * 4;
}

template <int G, int ST, bool PACK>
cudaError_t launch_t5_st(const PromptArgs& a, size_t smem, cudaStream_t stream) {
  constexpr int BM = T5_ROWS / G;
  auto k = prompt_t5_kernel<G, ST, PACK>;
  cudaError_t e = raise_smem_limit(k, smem);
  if (e != cudaSuccess) return e;
  k<<<tile_grid(a, BM), T5_THREADS, smem, stream>>>(a);
  return cudaGetLastError();
}

// As many stages as the lists leave room for; packed lists where not even two are left otherwise
// (windows beyond about 12000 tokens).
template <int G>
cudaError_t launch_t5_g(PromptArgs a, cudaStream_t stream) {
  constexpr int BM = T5_ROWS / G;
  a.capM = a.s + 2 * BM + a.w;
  const size_t s4 = t5_smem<4, false>(a.capA, a.capM), s3 = t5_smem<3, false>(a.capA, a.capM);
  const size_t s2 = t5_smem<2, false>(a.capA, a.capM), sp = t5_smem<2, true>(a.capA, a.capM);
  if (s4 <= 227 * 1024) return launch_t5_st<G, 4, false>(a, s4, stream);
  if (s3 <= 227 * 1024) return launch_t5_st<G, 3, false>(a, s3, stream);
  if (s2 <= 227 * 1024) return launch_t5_st<G, 2, false>(a, s2, stream);
  if (sp <= 227 * 1024) return launch_t5_st<G, 2, true>(a, sp, stream);
  return cudaErrorInvalidValue;
}

}  // namespace

bool prompt_t5_ok(int d, int G, int S, int s, int w, int k) {
  if (d != 128 || !(G == 1 || G == 2 || G == 4)) return false;
  const long long capM = (long long)s + 2 * T5_ROWS + w;
  return (S <= 1 << T5_POS_BITS ? t5_smem<2, true>((long long)s + k, capM)
                                : t5_smem<2, false>((long long)s + k, capM)) <= 227 * 1024;
}

cudaError_t launch_prompt_t5(const PromptArgs& a, int G, cudaStream_t stream) {
  if (G == 4) return launch_t5_g<4>(a, stream);
  if (G == 2) return launch_t5_g<2>(a, stream);
  return launch_t5_g<1>(a, stream);
}

}  // namespace kvpop
