// Running top-k cutoffs over a prompt (App. C.1 mask, App. C.2 cutoff scan).
//
// Kernel 1 ranks a row's tokens by static priority, higher first, equal priorities by
// position: a stable least-significant-digit radix sort of the order-reversed fp32 bit
// pattern, 4 passes of 8 bits.  A cluster of up to 8 CTAs holds the row in registers and
// shared memory (rank_cluster_kernel); rows too long for that, and short ones, take one CTA that
// sorts through global memory (rank_kernel).  The last pass writes rank[position] directly.
//
// Kernel 2 computes tau_q for every query position, a row's queries split over CTAs and
// their warps.  The paper inserts each newly eligible rank into a Fenwick tree and reads
// the k-th smallest by binary lifting.  Here the same value comes from the observation
// that tau_q never increases once k tokens are eligible: a bitset over ranks
// (8 KB for 65536 tokens, in shared memory) marks the inserted ranks, and when a
// newcomer ranks below the current cutoff the cutoff steps down to the next
// marked rank below it -- the warp scans 32 bitset words per ballot.  A chunk's warp
// starts from the state the scan would have reached: it marks the ranks of the tokens
// already eligible and takes the min(k, n)-th marked rank as the cutoff (a popcount
// prefix over the bitset).
// While fewer than k tokens are eligible every one of them is kept, so tau_q is
// the largest inserted rank (-1 while none is).
#include <cooperative_groups.h>

#include <algorithm>
#include <climits>

#include "kvpop_internal.cuh"

namespace kvpop {
namespace {

namespace cg = cooperative_groups;

constexpr int RK_NT = 512;
constexpr int RK_NW = RK_NT / 32;
constexpr int CUT_MAX_WARPS = 16;

struct RankArgs {
  const float* prio;         // [n_rows][S]
  const int32_t* len;        // [n_rows / rows_per_len] or nullptr (every row has S tokens)
  int rows_per_len;
  int tail;                  // trailing positions of a row without a priority (-> -inf)
  int n_rows, S;
  uint32_t* ka;              // workspace: keys / positions, two buffers of [n_rows][S]
  int32_t* pa;
  uint32_t* kb;
  int32_t* pb;
  int32_t* rank;             // [n_rows][S]
  int32_t* order;            // [n_rows][S] position of each rank (inverse of rank; the pb buffer)
};

// Ascending key = descending priority; NaN -> -inf, -0 -> +0 (as the decode scores).
__device__ __forceinline__ uint32_t rank_key(float f) {
  if (f != f) f = -INFINITY;
  f = __fadd_rn(f, 0.0f);
  const uint32_t b = __float_as_uint(f);
  const uint32_t o = (b & 0x80000000u) ? ~b : (b | 0x80000000u);
  return ~o;
}

__device__ __forceinline__ int row_length(const int32_t* len, int rows_per_len, int row, int S) {
  if (!len) return S;
  return max(0, min(len[row / rows_per_len], S));
}

// A row's sort by a cluster: CTA c holds elements [c * SEG, (c + 1) * SEG), SEG = 512 * I,
// each thread I of them in registers (warp-striped, so (warp, item, lane) is the element
// order and the sort stays stable).  Per pass a warp ranks its elements inside their digit
// (match + a running count per warp and digit), the CTAs exchange their 256 digit totals
// through distributed shared memory, and every (key, position) goes to its place in the
// owner's shared memory: no global traffic but the priorities in and the ranks out.
// Latency-bound (two cluster barriers and I match rounds per pass), so a row is spread
// over as many CTAs as leave the GPU about two CTAs per SM.  Device time, against one CTA
// per row through global memory: 8 rows of 32768 tokens 35 us (458), 16 of 8192 21 us (117),
// 48 of up to 2801 19 us (45), 8 of 2039 14 us (32).
template <int I>
__global__ void __launch_bounds__(RK_NT) rank_cluster_kernel(RankArgs a) {
  constexpr int SEG = RK_NT * I;
  extern __shared__ uint2 rk_buf[];              // [SEG] (key, position)
  __shared__ uint32_t cnt[RK_NW][256];
  __shared__ uint32_t tot[256], base[256], wsum[8];
  cg::cluster_group cl = cg::this_cluster();
  const int C = (int)cl.num_blocks(), c = (int)cl.block_rank();
  const int row = blockIdx.x / C;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int S = a.S;
  const int L = row_length(a.len, a.rows_per_len, row, S);
  const int nsc = max(L - a.tail, 0);
  const size_t ro = (size_t)row * S;
  const uint32_t lt_mask = (1u << lane) - 1u;
  const int e0 = warp * 32 * I + lane;           // element i of the thread: e0 + 32 i
  uint32_t key[I];
  int32_t pos[I];
#pragma unroll
  for (int i = 0; i < I; ++i) {
    const int t = c * SEG + e0 + 32 * i;
    pos[i] = t;
    key[i] = t < nsc ? rank_key(a.prio[ro + t]) : rank_key(-INFINITY);
  }
  for (int p = 0; p < 4; ++p) {
    for (int j = tid; j < RK_NW * 256; j += RK_NT) (&cnt[0][0])[j] = 0;
    __syncthreads();
    uint32_t rk[I];
#pragma unroll
    for (int i = 0; i < I; ++i) {
      const bool ok = c * SEG + e0 + 32 * i < L;
      const uint32_t dig = ok ? ((key[i] >> (8 * p)) & 255u) : 256u;
      const uint32_t peers = __match_any_sync(0xffffffffu, dig);
      const uint32_t within = __popc(peers & lt_mask);
      const uint32_t old = ok ? cnt[warp][dig] : 0u;
      __syncwarp();
      if (ok && within == 0) cnt[warp][dig] = old + __popc(peers);
      __syncwarp();
      rk[i] = old + within;
    }
    __syncthreads();
    if (tid < 256) {
      uint32_t run = 0;
#pragma unroll
      for (int w = 0; w < RK_NW; ++w) {
        const uint32_t n = cnt[w][tid];
        cnt[w][tid] = run;
        run += n;
      }
      tot[tid] = run;
    }
    cl.sync();                                   // every CTA's totals are written
    uint32_t before = 0, all = 0, x = 0;
    if (tid < 256) {
      for (int r = 0; r < C; ++r) {
        const uint32_t n = cl.map_shared_rank(tot, r)[tid];
        if (r < c) before += n;
        all += n;
      }
      x = all;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
      }
      if (lane == 31) wsum[warp] = x;
    }
    __syncthreads();
    if (tid < 256) {
      uint32_t off = 0;
      for (int w = 0; w < warp; ++w) off += wsum[w];
      base[tid] = off + x - all + before;
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < I; ++i) {
      if (c * SEG + e0 + 32 * i < L) {
        const uint32_t dig = (key[i] >> (8 * p)) & 255u;
        const uint32_t dst = base[dig] + cnt[warp][dig] + rk[i];
        if (p < 3) {
          cl.map_shared_rank(rk_buf, dst / SEG)[dst % SEG] = make_uint2(key[i], (uint32_t)pos[i]);
        } else {
          a.rank[ro + pos[i]] = (int32_t)dst;
          a.order[ro + dst] = pos[i];
        }
      }
    }
    cl.sync();          // all elements placed; after the last pass: all totals read
    if (p < 3) {
#pragma unroll
      for (int i = 0; i < I; ++i) {
        if (c * SEG + e0 + 32 * i < L) {
          const uint2 v = rk_buf[e0 + 32 * i];
          key[i] = v.x;
          pos[i] = (int32_t)v.y;
        }
      }
    }
  }
  for (int i = L + c * RK_NT + tid; i < S; i += C * RK_NT) a.rank[ro + i] = -1;
}

// Short rows (kShortRow), and rows longer than 8 * 512 * 32 tokens: one CTA per row, keys and
// positions in global memory.
// Within a round of RK_NT tokens the stable offset of each token inside its digit bucket
// comes from a warp match on the digit plus per-warp bucket counts; one histogram pass up
// front gives every pass its bucket bases.
__global__ void __launch_bounds__(RK_NT) rank_kernel(RankArgs a) {
  __shared__ uint32_t hist[4][256];
  __shared__ uint32_t base[256];
  __shared__ uint32_t cnt[RK_NW][256];
  const int row = blockIdx.x;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int S = a.S;
  const int L = row_length(a.len, a.rows_per_len, row, S);
  const int nsc = max(L - a.tail, 0);
  const size_t ro = (size_t)row * S;
  const float* prio = a.prio + ro;
  const uint32_t lt_mask = (1u << lane) - 1u;
  const uint32_t neg_inf_key = rank_key(-INFINITY);

  for (int i = tid; i < 4 * 256; i += RK_NT) (&hist[0][0])[i] = 0;
  __syncthreads();
  // histograms of all four digits, warp-aggregated per digit value
  for (int i0 = 0; i0 < L; i0 += RK_NT) {
    const int i = i0 + tid;
    const bool ok = i < L;
    const uint32_t key = ok ? (i < nsc ? rank_key(prio[i]) : neg_inf_key) : 0u;
#pragma unroll
    for (int p = 0; p < 4; ++p) {
      const uint32_t dig = ok ? ((key >> (8 * p)) & 255u) : 256u;
      const uint32_t peers = __match_any_sync(0xffffffffu, dig);
      if (ok && (__ffs(peers) - 1) == lane) atomicAdd(&hist[p][dig], (uint32_t)__popc(peers));
    }
  }
  __syncthreads();

  for (int p = 0; p < 4; ++p) {
    // bucket bases: exclusive prefix of the digit histogram (8 warps x 32 digits)
    if (tid < 256) {
      const uint32_t h = hist[p][tid];
      uint32_t x = h;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
      }
      cnt[0][tid] = x;          // inclusive within the warp's 32 digits (scratch)
    }
    __syncthreads();
    if (tid < 256) {
      uint32_t off = 0;
      for (int w = 0; w < (tid >> 5); ++w) off += cnt[0][w * 32 + 31];
      base[tid] = off + cnt[0][tid] - hist[p][tid];
    }
    __syncthreads();
    const uint32_t* sk = (p == 1) ? a.ka + ro : (p == 2) ? a.kb + ro : (p == 3) ? a.ka + ro : nullptr;
    const int32_t* sp = (p == 1) ? a.pa + ro : (p == 2) ? a.pb + ro : (p == 3) ? a.pa + ro : nullptr;
    uint32_t* dk = (p == 0 || p == 2) ? a.ka + ro : a.kb + ro;
    int32_t* dp = (p == 0 || p == 2) ? a.pa + ro : a.pb + ro;
    for (int i0 = 0; i0 < L; i0 += RK_NT) {
      const int i = i0 + tid;
      const bool ok = i < L;
      uint32_t key = 0;
      int32_t pos = i;
      if (ok) {
        if (p == 0) {
          key = i < nsc ? rank_key(prio[i]) : neg_inf_key;
        } else {
          key = sk[i];
          pos = sp[i];
        }
      }
      const uint32_t dig = ok ? ((key >> (8 * p)) & 255u) : 256u;
      for (int j = lane; j < 256; j += 32) cnt[warp][j] = 0;
      __syncwarp();
      const uint32_t peers = __match_any_sync(0xffffffffu, dig);
      const uint32_t within = __popc(peers & lt_mask);
      if (ok && within == 0) cnt[warp][dig] = __popc(peers);
      __syncthreads();
      if (tid < 256) {
        uint32_t run = base[tid];
        for (int w = 0; w < RK_NW; ++w) {
          const uint32_t c = cnt[w][tid];
          cnt[w][tid] = run;
          run += c;
        }
        base[tid] = run;
      }
      __syncthreads();
      if (ok) {
        const uint32_t dst = cnt[warp][dig] + within;
        if (p < 3) {
          dk[dst] = key;
          dp[dst] = pos;
        } else {
          a.rank[ro + pos] = (int32_t)dst;
          a.order[ro + dst] = pos;          // pb is free in the last pass
        }
      }
      __syncwarp();
    }
    __syncthreads();     // this pass's global writes are visible to the next pass
  }
  for (int i = L + tid; i < S; i += RK_NT) a.rank[ro + i] = -1;
}

struct CutArgs {
  const int32_t* rank;       // [n_rows][S]
  const int32_t* len;
  int rows_per_len;
  int n_rows, S, s, w, k;
  int32_t* tau;              // [n_rows][S]
};

// Largest marked rank below r (one exists whenever this is called).
__device__ __forceinline__ int marked_below(const uint32_t* bits, int r, int lane) {
  const int wi = r >> 5;
  const uint32_t m = bits[wi] & ((1u << (r & 31)) - 1u);
  if (m) return (wi << 5) + 31 - __clz(m);
  for (int top = wi - 1; top >= 0; top -= 32) {
    const int idx = top - lane;
    const uint32_t v = idx >= 0 ? bits[idx] : 0u;
    const uint32_t bal = __ballot_sync(0xffffffffu, v != 0u);
    if (bal) {
      const int l = __ffs(bal) - 1;
      const uint32_t vs = __shfl_sync(0xffffffffu, v, l);
      return ((top - l) << 5) + 31 - __clz(vs);
    }
  }
  return -1;
}

// Smallest marked rank whose count of marked ranks at or below it reaches c
// (c >= 1 and at least c ranks marked); warp-collective.
__device__ __forceinline__ int kth_marked(const uint32_t* bits, int words, int c, int lane) {
  int base = 0;
  for (int w0 = 0; w0 < words; w0 += 32) {
    const int wi = w0 + lane;
    const uint32_t v = wi < words ? bits[wi] : 0u;
    const int cnt = __popc(v);
    const int total = __reduce_add_sync(0xffffffffu, cnt);
    if (base + total >= c) {
      int incl = cnt;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
      }
      const uint32_t hit = __ballot_sync(0xffffffffu, base + incl >= c);
      const int l = __ffs(hit) - 1;
      uint32_t word = __shfl_sync(0xffffffffu, v, l);
      int need = c - (base + __shfl_sync(0xffffffffu, incl - cnt, l));
      int bit = 0;
      for (; bit < 32; ++bit) {
        if ((word >> bit) & 1u) {
          if (--need == 0) break;
        }
      }
      return (w0 + l) * 32 + bit;
    }
    base += total;
  }
  return -1;
}

// CTA (row, y) takes warps * chunk consecutive queries, warp c of it `chunk` of them.  The
// CTA marks the ranks of the tokens already eligible at its first query once; each warp
// copies that bitset, adds the tokens up to its own first query and so has the state the
// scan has there -- the ranks inserted so far and the cutoff, the min(k, n)-th smallest of
// them -- then runs the same per-query update, so every chunk's cutoffs equal those of
// one scan over the whole row.  Bound by the serial chain of a warp's queries; with every
// warp rebuilding its own state from the row's start a chunk had to be 512 queries long.
// Device time before and now: 8 rows of 32768 tokens 489 -> 56 us, 16 of 8192 183 -> 22 us,
// 48 of up to 2801 73 -> 17 us.
__global__ void cutoff_kernel(CutArgs a, int chunk) {
  extern __shared__ uint32_t bitsets[];          // [words] of the CTA, then [warps][words]
  __shared__ int n_base;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int row = blockIdx.x;
  const int S = a.S, words = (S + 31) >> 5;
  const int L = row_length(a.len, a.rows_per_len, row, S);
  const int32_t* rank = a.rank + (size_t)row * S;
  int32_t* tau_out = a.tau + (size_t)row * S;
  const int qcta = blockIdx.y * (blockDim.x >> 5) * chunk;
  for (int i = max(L, qcta) + tid; i < min(S, qcta + (int)(blockDim.x >> 5) * chunk); i += blockDim.x)
    tau_out[i] = -1;
  if (qcta >= L) return;
  const int s = a.s, w = a.w, k = a.k;
  for (int i = tid; i < words; i += blockDim.x) bitsets[i] = 0u;
  if (tid == 0) n_base = 0;
  __syncthreads();
  // tokens inserted before query qcta: positions s .. qcta - 1 - w
  int cnt = 0;
#pragma unroll 8
  for (int t = s + tid; t <= qcta - 1 - w; t += blockDim.x) {
    const int r = rank[t];
    if (r >= 0 && r < S) {
      atomicOr(&bitsets[r >> 5], 1u << (r & 31));
      ++cnt;
    }
  }
  cnt = __reduce_add_sync(0xffffffffu, cnt);
  if (lane == 0 && cnt) atomicAdd(&n_base, cnt);
  __syncthreads();
  const int qa = qcta + warp * chunk;
  if (qa >= L) return;
  const int qb = min(qa + chunk, L);
  uint32_t* bits = bitsets + (size_t)(1 + warp) * words;
  for (int i = lane; i < words; i += 32) bits[i] = bitsets[i];
  __syncwarp();
  cnt = 0;
  for (int t = max(s, qcta - w) + lane; t <= qa - 1 - w; t += 32) {
    const int r = rank[t];
    if (r >= 0 && r < S) {
      atomicOr(&bits[r >> 5], 1u << (r & 31));
      ++cnt;
    }
  }
  cnt = __reduce_add_sync(0xffffffffu, cnt);
  __syncwarp();
  int n = n_base + cnt;
  int tau = n > 0 ? kth_marked(bits, words, min(k, n), lane) : -1;
  for (int q0 = qa; q0 < qb; q0 += 32) {
    const int tl = q0 + lane - w;
    int r_l = -1;
    if (tl >= s && tl < L) r_l = rank[tl];
    int mine = -1;
    const int nq = min(32, qb - q0);
    for (int j = 0; j < nq; ++j) {
      const int t = q0 + j - w;
      if (t >= s) {
        const int r = __shfl_sync(0xffffffffu, r_l, j);
        if (r >= 0 && r < S) {
          ++n;
          if (n <= k || r < tau) {               // ranks above a full cutoff never matter again
            if (lane == 0) bits[r >> 5] |= 1u << (r & 31);
            __syncwarp();
            if (n <= k) tau = max(tau, r);
            else tau = marked_below(bits, tau, lane);
          }
        }
      }
      if (lane == j) mine = (k > 0) ? tau : -1;
    }
    if (lane < nq) tau_out[q0 + lane] = mine;
  }
}

template <int I>
cudaError_t launch_rank_cluster(const RankArgs& ra, int C, cudaStream_t stream) {
  const size_t smem = (size_t)RK_NT * I * sizeof(uint2);
  cudaError_t e = raise_smem_limit(rank_cluster_kernel<I>, smem);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)(ra.n_rows * C));
  cfg.blockDim = dim3(RK_NT);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = (unsigned)C;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, rank_cluster_kernel<I>, ra);
}

// Rows up to here take the one-CTA rank kernel, whose passes over so few tokens cost less than the
// cluster kernel's set-up (ranks and cutoffs, us: 1 row of 256 tokens 14.4 against 16.5, 20000 of 64
// 318 against 422, 4000 of 256 123 against 130; from 512 on the cluster kernel, 1000 rows 61 against
// 67), and their queries are spread over all warps of one CTA: 16, or 8 where there are rows for
// more than two CTAs an SM (20000 of 64: 363 with 16, 318 with 8; 300 of 128: 14.5 and 16.5).
constexpr int kShortRow = 384;

// CTAs per row C (a power of two up to 8) and items per thread: the largest C that keeps the
// grid within two CTAs per SM and gives every CTA at least 1024 elements, more where the row
// does not fit otherwise.
cudaError_t launch_rank(const RankArgs& ra, int sms, cudaStream_t stream) {
  int C = 1;
  while (C < 8 && (long long)ra.n_rows * (2 * C) <= 2 * sms && ra.S > 2 * RK_NT * C) C *= 2;
  while (C < 8 && ra.S > 32 * RK_NT * C) C *= 2;
  const int per = (ra.S + C - 1) / C;
  if (ra.S <= kShortRow || per > 32 * RK_NT || (long long)ra.n_rows * C > INT_MAX) {
    rank_kernel<<<ra.n_rows, RK_NT, 0, stream>>>(ra);
    return cudaGetLastError();
  }
  if (per <= 2 * RK_NT) return launch_rank_cluster<2>(ra, C, stream);
  if (per <= 4 * RK_NT) return launch_rank_cluster<4>(ra, C, stream);
  if (per <= 8 * RK_NT) return launch_rank_cluster<8>(ra, C, stream);
  if (per <= 16 * RK_NT) return launch_rank_cluster<16>(ra, C, stream);
  return launch_rank_cluster<32>(ra, C, stream);
}

}  // namespace

size_t topk_workspace_bytes(int n_rows, int S) {
  return (size_t)n_rows * (size_t)S * 16 + 1024;
}

const int32_t* topk_order(const void* workspace, int n_rows, int S) {
  const size_t n = (size_t)n_rows * S;
  const size_t al = (n * 4 + 255) & ~size_t(255);
  return reinterpret_cast<const int32_t*>(static_cast<const char*>(workspace) + 3 * al);
}

cudaError_t launch_topk(const float* prio, const int32_t* len, int rows_per_len, int tail,
                        int n_rows, int S, int s, int w, int k, int32_t* rank, int32_t* tau,
                        int32_t* order, void* workspace, cudaStream_t stream) {
  if (n_rows <= 0 || S <= 0) return cudaSuccess;
  // no token is eligible either way, and no position is computed past 2 S
  s = std::min(s, S);
  w = std::min(w, S);
  const size_t n = (size_t)n_rows * S;
  char* ws = static_cast<char*>(workspace);
  auto al = [](size_t x) { return (x + 255) & ~size_t(255); };
  RankArgs ra{prio, len, rows_per_len, tail, n_rows, S,
              reinterpret_cast<uint32_t*>(ws), reinterpret_cast<int32_t*>(ws + al(n * 4)),
              reinterpret_cast<uint32_t*>(ws + 2 * al(n * 4)),
              reinterpret_cast<int32_t*>(ws + 3 * al(n * 4)), rank,
              order ? order : reinterpret_cast<int32_t*>(ws + 3 * al(n * 4))};
  int dev = 0, sms = 152;
  if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  cudaError_t e = launch_rank(ra, sms, stream);
  if (e != cudaSuccess) return e;
  // warps per CTA: up to 16, each with its own bitset of S bits beside the CTA's
  const size_t words_bytes = (size_t)((S + 31) / 32) * 4;
  int nch = (int)std::max<size_t>(1, std::min<size_t>(CUT_MAX_WARPS, (200 * 1024) / words_bytes - 1));
  // queries per warp: enough CTAs for about two per SM, at least 32 (a warp's reads of the
  // newcomers' ranks) and at most 512 (the serial chain of one warp)
  const int want = std::max(1, (2 * sms + n_rows - 1) / n_rows);
  const int per = (S + nch * want - 1) / (nch * want);
  int chunk = std::min(512, std::max(32, (per + 31) / 32 * 32));
  if (S <= kShortRow) {
    nch = n_rows > 2 * sms ? CUT_MAX_WARPS / 2 : CUT_MAX_WARPS;
    chunk = (S + nch - 1) / nch;
  }
  const int split = (S + nch * chunk - 1) / (nch * chunk);
  const size_t smem = (size_t)(nch + 1) * words_bytes;
  e = raise_smem_limit(cutoff_kernel, smem);
  if (e != cudaSuccess) return e;
  CutArgs ca{rank, len, rows_per_len, n_rows, S, s, w, k, tau};
  cutoff_kernel<<<dim3(n_rows, split), nch * 32, smem, stream>>>(ca, chunk);
  return cudaGetLastError();
}

}  // namespace kvpop
