// Split-K schedule and partial merge shared by the decode-attention kernels.
//
// The key stream of every (sequence, KV head) pair -- used slots first, then
// the window -- is cut into tiles of `tile` keys.  The concatenated tile list
// over all pairs is split into NC equal contiguous ranges, one per CTA, so the
// work per CTA is balanced whatever the per-pair lengths (ragged batches).
// A pair whose tiles span several CTAs gets one (m, l, o) partial from each;
// the last CTA to finish it (atomic counter, no waiting) merges them in CTA
// order, which keeps the result independent of arrival order.
#pragma once

#include <type_traits>

#include "kvpop_internal.cuh"

namespace kvpop {

__device__ __forceinline__ int tiles_of(int nv, int np, int tile) {
  return (nv + tile - 1) / tile + (np + tile - 1) / tile;
}

// CTA whose tile range [c*T/N, (c+1)*T/N) contains tile t (requires N <= T).
__device__ __forceinline__ long long cta_of(long long t, long long T, long long N) {
  return ((t + 1) * N - 1) / T;
}
__device__ __forceinline__ long long cta_begin(long long c, long long T, long long N) {
  return c * T / N;
}

// Block-wide exclusive prefix of per-pair tile counts into prefix[0..npairs]
// (prefix[npairs] = total).  `scan` holds one int per warp.  Contains
// __syncthreads; every thread of the block must call it.
// The counts are read from L2: a kernel may call this before and after the wait for the
// kernel that writes them, and no line of the first reading may serve the second.
template <int NT>
__device__ __forceinline__ void build_schedule(const int32_t* __restrict__ nvalid,
                                               const int32_t* __restrict__ len, int npairs, int B,
                                               int D, int tile, int* prefix, int* scan,
                                               int32_t* err) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int per = (npairs + NT - 1) / NT;
  const int beg = min(tid * per, npairs), end = min(beg + per, npairs);
  int local = 0;
  for (int i = beg; i < end; ++i)
    local += tiles_of(used_slots(__ldcg(nvalid + i), B, err), window_rows(__ldcg(len + i), D, err), tile);
  int incl = local;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, incl, off);
    if (lane >= off) incl += y;
  }
  if (lane == 31) scan[warp] = incl;
  __syncthreads();
  if (tid == 0) {
    int run = 0;
    for (int w = 0; w < NT / 32; ++w) { const int x = scan[w]; scan[w] = run; run += x; }
    prefix[npairs] = run;
  }
  __syncthreads();
  int run = scan[warp] + incl - local;
  for (int i = beg; i < end; ++i) {
    prefix[i] = run;
    run += tiles_of(used_slots(__ldcg(nvalid + i), B, nullptr), window_rows(__ldcg(len + i), D, nullptr), tile);
  }
  __syncthreads();
}

// Whether some pair's tile count is no longer the one in `prefix` (block-wide; every thread
// calls it).  One round of reads where a rebuild takes two and the scan.
template <int NT>
__device__ __forceinline__ bool schedule_changed(const int32_t* __restrict__ nvalid,
                                                 const int32_t* __restrict__ len, int npairs, int B,
                                                 int D, int tile, const int* prefix, int32_t* err) {
  bool differs = false;
  for (int i = threadIdx.x; i < npairs; i += NT)
    differs |= tiles_of(used_slots(__ldcg(nvalid + i), B, err), window_rows(__ldcg(len + i), D, err),
                        tile) != prefix[i + 1] - prefix[i];
  return __syncthreads_or(differs);
}

// Merges the partials that CTAs ca..cb left for one pair, in CTA order, and writes its output.
// A partial's place is fixed by the split: the pair's first tile lies in CTA ca (second slot
// of its two), every later CTA starts inside the pair (first slot).  The (max, sum) pairs are
// fetched once for all threads into `fac` (2 G (cb - ca + 1) floats of shared memory), and the
// rows are loaded RB at a time with them, so a merge costs an L2 latency or two instead of one
// chain of 2 (cb - ca + 1) per thread: a pair at batch 1 spreads over 19 CTAs,
// and from its last arrival to the end of the launch went 8 us with 8 single rows in flight, 6
// with 20 double ones (a 4-layer step at batch 1: 316 us with the chain, 235 with this and the
// early launches below).
constexpr int kMaxAttendGrid = 256;      // CTAs whose factors fit in the warps' partials (4 HD)

template <int G, int HD, int NCT, int RB = 20, typename SyncFn, typename ExpFn>
__device__ __forceinline__ void merge_partials(long long ca, long long cb, const float* part, float* out,
                                               float* fac, SyncFn sync, ExpFn ex) {
  constexpr int PSTRIDE = G * HD + 2 * G;
  const int tid = threadIdx.x;
  const int n = (int)(cb - ca) + 1;
  const float* first = part + ((size_t)ca * 2 + 1) * PSTRIDE;
  auto at = [&](int c) { return c == 0 ? first : part + (size_t)(ca + c) * 2 * PSTRIDE; };
  for (int i = tid; i < n * G; i += NCT) {
    const float* pc = at(i / G) + G * HD + i % G;
    fac[2 * i] = __ldcg(pc);
    fac[2 * i + 1] = __ldcg(pc + G);
  }
  // V neighbouring outputs per thread, RB rows in flight; the first ones travel with the factors
  constexpr int V = (G * HD) % (2 * NCT) == 0 ? 2 : 1;
  using Vec = std::conditional_t<V == 2, float2, float>;
  auto load = [&](Vec (&row)[RB], int c0, int idx) {
#pragma unroll
    for (int k = 0; k < RB; ++k)
      if (c0 + k < n) row[k] = __ldcg(reinterpret_cast<const Vec*>(at(c0 + k) + idx));
  };
  Vec row[RB];
  if (V * tid < G * HD) load(row, 0, V * tid);
  sync();
  for (int idx = V * tid; idx < G * HD; idx += V * NCT) {
    const int g = idx / HD;
    float ms = -INFINITY;
    for (int c = 0; c < n; ++c) ms = fmaxf(ms, fac[2 * (c * G + g)]);
    float L = 0.f, O[V] = {};
    for (int c0 = 0; c0 < n; c0 += RB) {
      if (c0 > 0 || idx >= V * NCT) load(row, c0, idx);
#pragma unroll
      for (int k = 0; k < RB; ++k) {
        if (c0 + k >= n) break;
        const float mc = fac[2 * ((c0 + k) * G + g)];
        const float f = (mc == -INFINITY) ? 0.f : ex(mc - ms);
        L = fmaf(fac[2 * ((c0 + k) * G + g) + 1], f, L);
        if constexpr (V == 2) {
          O[0] = fmaf(row[k].x, f, O[0]);
          O[1] = fmaf(row[k].y, f, O[1]);
        } else {
          O[0] = fmaf(row[k], f, O[0]);
        }
      }
    }
#pragma unroll
    for (int v = 0; v < V; ++v) out[idx + v] = O[v] / L;
  }
}

// Pair p's segment in this CTA is complete; mo/ml/mm hold NW warp partials
// (log2-domain running max mm, sum ml, unnormalised output mo[w][g][d]).
// Writes the output, or this CTA's partial and -- when it is the last
// contributor -- the merged output.  Called by the NCT consumer threads
// (tid < NCT) together; `sync` is their barrier; `flag` is one shared int.
template <int G, int HD, int NW, int NCT, typename SyncFn>
__device__ __forceinline__ void finish_pair(int p, const int* prefix, long long Ttot, long long NC,
                                            long long t0, float* mo, const float* ml,
                                            const float* mm, float* out, float* part,
                                            int32_t* part_count, int* flag, SyncFn sync) {
  constexpr int PSTRIDE = G * HD + 2 * G;
  const int tid = threadIdx.x;
  const long long ca = cta_of(prefix[p], Ttot, NC);
  const long long cb = cta_of(prefix[p + 1] - 1, Ttot, NC);
  const bool complete = (ca == cb);
  float* mypart = nullptr;
  if (!complete) {
    const int slot = (prefix[p] < t0) ? 0 : 1;
    mypart = part + ((size_t)blockIdx.x * 2 + slot) * PSTRIDE;
  }
  for (int idx = tid; idx < G * HD; idx += NCT) {
    const int g = idx / HD, i = idx - g * HD;
    float ms = -INFINITY;
#pragma unroll
    for (int w = 0; w < NW; ++w) ms = fmaxf(ms, mm[w * G + g]);
    float L = 0.f, O = 0.f;
#pragma unroll
    for (int w = 0; w < NW; ++w) {
      const float mw = mm[w * G + g];
      const float f = (mw == -INFINITY) ? 0.f : exp2f(mw - ms);
      L = fmaf(ml[w * G + g], f, L);
      O = fmaf(mo[(w * G + g) * HD + i], f, O);
    }
    if (complete) {
      out[((size_t)p * G + g) * HD + i] = O / L;
    } else {
      mypart[g * HD + i] = O;
      if (i == 0) { mypart[G * HD + g] = ms; mypart[G * HD + G + g] = L; }
    }
  }
  if (!complete) {
    __threadfence();
    sync();
    if (tid == 0) {
      const int old = atomicAdd(&part_count[p], 1);
      const int last = (old == (int)(cb - ca));
      if (last) part_count[p] = 0;
      *flag = last;
    }
    sync();
    if (*flag) {
      __threadfence();
      // the warps' own partials have been folded: their room holds the merge's factors
      merge_partials<G, HD, NCT>(ca, cb, part, out + (size_t)p * G * HD, mo, sync,
                                 [](float x) { return exp2f(x); });
    }
  }
  sync();
}

}  // namespace kvpop
