// Ranking of cells by splitting: the same stable order as the digit passes of
// sort.cu, from two splits and a sort in shared memory instead of four digit
// passes over memory.
//
//   k_msd_map    : histogram of the intensities' keys over 2^14 counters and from
//                  it a piecewise-linear map of (key, cell) to [0, 2^32) that
//                  follows the distribution; it only balances the buckets, no
//                  result depends on it.  Every cell is counted: samples of 1/4
//                  to 1/16 misjudged the extremes, which lie together in a few
//                  peaks and voids, and overflowed their buckets.  The map's 2048
//                  knots go where the cells are: one to each of 512 spans of the
//                  key range, and 2^g, as many as there are, to those that hold
//                  more than half a final bucket.  A few intensities at or below
//                  zero, which mean free paths below 3 leave in any large field,
//                  stretch the key range over all exponents; equal knots, a
//                  quarter octave wide there, then misjudged the bulk and
//                  overflowed (512^3, l = 2: a solve 10.05 ms, with the spans 5.73)
//   k_msd_split  : cells to buckets of the map, by tiles: shared-memory atomics
//                  give each cell a slot of its bucket's run in the tile and
//                  global ones each run a place in the bucket's region (any
//                  order: the local sort restores cell order in ties), and the
//                  tile is written run by run.  One split makes up to 1024
//                  final buckets; larger fields take two of about sqrt each
//   k_msd_local  : a final bucket (3840 cells on average, at most 4608) in
//                  shared memory: a counting pass over 8192 sub-buckets, linear
//                  in (key, cell) over the bucket's range, leaves each cell among
//                  about 1.5; it then counts which of those precede it.  Where
//                  ties share a sub-bucket they are counted again by cell, or
//                  merge sorted (sort_ties).  With the masses the bucket is also
//                  matched there (scan.cuh): its rank order never goes to memory
//   fallback     : a field the map does not balance (a bucket outgrows its
//                  region, or the map sees it coming) is ranked by the digit
//                  passes, in one cooperative launch that otherwise ends at
//                  once: 8.3 ms a pass at 1024^3, 6.9 in launches of their own
//
// A stable digit pass pays for its order with eight ballots per cell and is
// bound by instruction issue (6.6 ms each at 1024^3); a split needs none, carries
// 9 bits' worth and is bound by the shared-memory pipe (77 % busy, 7.1 ms), the
// local sort by both (64 % and 2 instructions a cycle).  Digit passes with their
// histogram against this, masses carried along: 33 000 cells 61 -> 28 us, 2^21
// 132 -> 67 us, 2^24 505 -> 400 us, 2^27 3.51 -> 2.75 ms, 2^30 28.6 -> 24.7 ms.
#include <type_traits>

#include "fixed128.cuh"
#include "msd.cuh"
#include "scan.cuh"

namespace amber {

// Each kernel's work is that of CTA blk of nblk on one ranking: of the launch, or
// (k_msd_*_multi) of the launch's row blockIdx.y, one ranking each.
template <int FINE>
__device__ __forceinline__ void msd_map_body(const MsdArgs& a, uint32_t blk, uint32_t nblk) {
  constexpr int NC = kMsdSpans << FINE, NT = 1024;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  uint32_t* h = reinterpret_cast<uint32_t*>(smem_raw);  // [NC]
  __shared__ uint32_t s_last, wsum[32], whvy[32];
  const int tid = threadIdx.x;
  for (int i = tid; i < NC; i += NT) h[i] = 0;
  const uint32_t gt = blk * NT + tid, ng = nblk * NT;
  for (uint32_t i = gt; i < a.nb1; i += ng) a.mc->cnt1[i * msd_cnt1_step(a.nb1)] = 0;
  if (a.nb2 > 1)
    for (uint32_t i = gt; i < a.nb1 * a.nb2; i += ng) a.cnt2[i] = 0;
  if (gt == 0) {
    a.mc->overflow = 0;
    a.mc->bar = 0;
    a.mc->given_up = 0;
    // what amber_sort_passes reports: the digits the key range would take
    const int bits = 32 - __clz((int)((uint32_t)a.ctrl->kmax - (uint32_t)a.ctrl->kmin));
    a.ctrl->npasses = max((bits + a.digit_bits - 1) / a.digit_bits, 1);
  }
  if (a.state) {
    for (uint32_t i = gt; i < a.nb1 * a.nb2; i += ng) a.state[i] = 0;
    if (gt < kAssignCtrlBytes / 4) reinterpret_cast<uint32_t*>(a.actrl)[gt] = 0;
  }
  const MsdRange R = msd_range(a.ctrl, FINE);
  const int shift = R.L - FINE;
  __syncthreads();
  const uint32_t n = (uint32_t)a.n;
  bool bad = false;
  auto count = [&](float x) {
    atomicAdd(&h[min((enc_desc(x, bad) - R.kbase) >> shift, (uint32_t)NC - 1u)], 1u);
  };
  // 16-byte loads from a 16-byte aligned array, else element by element
  const uint32_t nv = (reinterpret_cast<uintptr_t>(a.J) & 15) == 0 ? n / 4 : 0;
  const float4* J4 = reinterpret_cast<const float4*>(a.J);
  uint32_t v = gt;
  for (; v + ng < nv; v += 2 * ng) {  // (v + 2 ng < 2^30)
    const float4 x = J4[v], y = J4[v + ng];
    count(x.x);
    count(x.y);
    count(x.z);
    count(x.w);
    count(y.x);
    count(y.y);
    count(y.z);
    count(y.w);
  }
  if (v < nv) {
    const float4 x = J4[v];
    count(x.x);
    count(x.y);
    count(x.z);
    count(x.w);
  }
  for (uint32_t i = nv * 4 + gt; i < n; i += ng) count(a.J[i]);
  __syncthreads();
  // two counters per atomic (none exceeds 32 bits), each CTA from a place of its
  // own: all of them walking the same lines together took twice as long
  unsigned long long* hist2 = reinterpret_cast<unsigned long long*>(a.mc->hist);
  for (int i = tid; i < NC / 2; i += NT) {
    const int at = (int)((i + blk * 96u) & (NC / 2 - 1u));
    const unsigned long long v = reinterpret_cast<const unsigned long long*>(h)[at];
    if (v) atomicAdd(hist2 + at, v);
  }
  __threadfence();
  __syncthreads();
  if (tid == 0) s_last = atomicAdd(&a.mc->done, 1u) == nblk - 1;
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  // two threads to a span, half of its counters each
  constexpr int PER = NC / NT;
  static_assert(PER % 4 == 0 && PER * 2 == 1 << FINE, "whole 16-byte words; two threads per span");
  uint32_t c[PER], sum = 0;
  uint4* hist4 = reinterpret_cast<uint4*>(a.mc->hist) + tid * (PER / 4);
#pragma unroll
  for (int q = 0; q < PER / 4; ++q) {
    const uint4 v4 = __ldcg(hist4 + q);
    hist4[q] = make_uint4(0, 0, 0, 0);  // clean for the next ranking
    c[4 * q] = v4.x;
    c[4 * q + 1] = v4.y;
    c[4 * q + 2] = v4.z;
    c[4 * q + 3] = v4.w;
    sum += v4.x + v4.y + v4.z + v4.w;
  }
  uint32_t x = sum;
  const int lane = tid & 31, warp = tid >> 5;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  const bool heavy = sum + __shfl_xor_sync(0xffffffffu, sum, 1) > n / (2u * a.nb1 * a.nb2);
  const uint32_t hm = __ballot_sync(0xffffffffu, heavy);
  if (lane == 31) wsum[warp] = x;
  if (lane == 0) whvy[warp] = __popc(hm);
  __syncthreads();
  uint32_t pre = 0, hpre = 0, H = 0;
  for (int w = 0; w < 32; ++w) {
    pre += w < warp ? wsum[w] : 0u;
    hpre += w < warp ? whvy[w] : 0u;
    H += whvy[w];
  }
  hpre = (hpre + __popc(hm & ((1u << (lane & ~1)) - 1u))) / 2;  // heavy spans before this one
  H /= 2;
  int g = 0;  // the heavy spans take 2^g knots each
  while (g < FINE && H * ((2u << g) - 1u) <= (uint32_t)(kMsdKnots - kMsdSpans)) ++g;
  // where the heavy spans are that many, all get four: the splits then find a
  // knot without the table (their lookups: 512^3 53 us of a split's 750)
  static_assert(kMsdKnots == kMsdSpans * 4, "four knots per span");
  const bool equal = g <= 3;
  const int ls = equal ? 2 : heavy ? g : 0, span = tid / 2;
  const uint32_t first = equal ? span * 4u : span + hpre * ((1u << g) - 1u);
  const uint32_t total = equal ? (uint32_t)kMsdKnots : kMsdSpans + H * ((1u << g) - 1u);
  uint32_t run = pre + x - sum;
#pragma unroll
  for (int q = 0; q < PER; ++q) {
    const int at = (tid & 1) * PER + q;
    if ((at & ((1 << (FINE - ls)) - 1)) == 0) a.mc->map[first + (at >> (FINE - ls))] = (uint32_t)((run * a.scale) >> 32);
    run += c[q];
  }
  if ((tid & 1) == 0) a.mc->span[span] = ((int)first - (span << ls)) * 32 + (R.L - ls);
  for (uint32_t i = total + tid; i <= (uint32_t)kMsdKnots; i += NT) a.mc->map[i] = 0xffffffffu;
  if (tid == 0) {
    a.mc->equal = equal ? R.L - 2 : -1;
    if (!equal && a.n > kMsdTieCells && H > (a.n > kMsdTieCells2 ? kMsdTieSpans2 : kMsdTieSpans)) a.mc->overflow = a.mc->given_up = 1;
    a.mc->done = 0;
  }
}

template <int FINE> __global__ void __launch_bounds__(1024, 2) k_msd_map(const MsdArgs a) {
  pdl_begin();
  msd_map_body<FINE>(a, blockIdx.x, gridDim.x);
}

template <int FINE> __global__ void __launch_bounds__(1024, 2) k_msd_map_multi(const MsdArgs* __restrict__ args) {
  __shared__ MsdArgs a;
  if (threadIdx.x == 0) a = args[blockIdx.y];
  __syncthreads();
  msd_map_body<FINE>(a, blockIdx.x, gridDim.x);
}

// Sum of the first `warp` entries of per-warp totals (at most 32 of them).
__device__ __forceinline__ uint32_t warps_before(const uint32_t* wsum, int nw, int lane, int warp) {
  return __reduce_add_sync(0xffffffffu, lane < nw && lane < warp ? wsum[lane] : 0u);
}

template <int NT, int IT, bool FIRST, bool MASS>
__device__ __forceinline__ void msd_split_body(const MsdArgs& a, uint32_t blk, uint32_t nblk) {
  constexpr int TILE = NT * IT;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  uint4* rec = reinterpret_cast<uint4*>(smem_raw);               // [TILE] (key, cell, mass, digit)
  uint2* map = reinterpret_cast<uint2*>(rec + TILE);             // [knots] (start, width)
  int32_t* spans = reinterpret_cast<int32_t*>(map + kMsdKnots);  // [spans]
  uint32_t* cnt = reinterpret_cast<uint32_t*>(spans + kMsdSpans);  // [digits] counts, then starts
  uint32_t* gb = cnt + kMsdMaxDigits;                            // [digits] global base - start
  __shared__ uint32_t wsum[NT / 32];
  __shared__ u128 wmass[NT / 32];
  if (!FIRST && (*reinterpret_cast<volatile uint32_t*>(&a.mc->overflow) & 1u)) return;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t nd = FIRST ? a.nb1 : a.nb2;
  for (int i = tid; i < kMsdKnots; i += NT) {
    const uint32_t b0 = a.mc->map[i];
    map[i] = make_uint2(b0, a.mc->map[i + 1] - b0);
  }
  for (int i = tid; i < kMsdSpans; i += NT) spans[i] = a.mc->span[i];
  const MsdRange R = msd_range(a.ctrl, a.fine);
  const int equal = a.mc->equal;
  const uint32_t n = (uint32_t)a.n;
  const uint32_t per = FIRST ? 1u : (a.cap1 + TILE - 1) / TILE;  // tiles per first-split bucket
  const uint32_t tiles = FIRST ? (n + TILE - 1) / TILE : a.nb1 * per;
  const uint32_t cap = FIRST ? a.cap1 : (uint32_t)kMsdCap;
  const uint32_t nb1 = a.nb1, nb2 = a.nb2;
  const int ishift = a.idx_shift;
  const float* __restrict__ min_ = FIRST ? a.mass : a.mass1;
  uint2* __restrict__ kvo = FIRST ? a.kv1 : a.kv2;
  float* __restrict__ mo = FIRST ? a.mass1 : a.mass2;
  bool bad = false;
  MassSum msum;
  uint32_t done = 0;
  // where the map has given up, the masses are summed and nothing is split
  const bool given_up = FIRST && a.n > kMsdTieCells && a.mc->given_up;
  for (uint32_t tile = blk; tile < tiles && !given_up; tile += nblk) {
    uint32_t start, have, bucket = 0;
    if (FIRST) {
      start = tile * (uint32_t)TILE;
      have = min(n - start, (uint32_t)TILE);
    } else {
      bucket = tile / per;
      const uint32_t at = (tile - bucket * per) * TILE, c = a.mc->cnt1[bucket * msd_cnt1_step(a.nb1)];
      if (at >= c) continue;  // uniform
      start = bucket * a.cap1 + at;
      have = min(c - at, (uint32_t)TILE);
    }
    for (uint32_t i = tid; i < nd; i += NT) cnt[i] = 0;
    __syncthreads();  // also: the previous tile's staged cells are written
    uint32_t key[IT], idx[IT], ds[IT];
    float m[IT];
    auto digits = [&](auto full_tag, auto equal_tag) {
      constexpr bool FULL = decltype(full_tag)::value, EQUAL = decltype(equal_tag)::value;
      const uint32_t p0 = start + tid;
#pragma unroll
      for (int it = 0; it < IT; ++it)
        if (FULL || it * NT + tid < have) {
          if (FIRST) {
            key[it] = __float_as_uint(a.J[p0 + it * NT]);
          } else {
            const uint2 v = a.kv1[p0 + it * NT];
            key[it] = v.x;
            idx[it] = v.y;
          }
        }
      if (MASS) {
#pragma unroll
        for (int it = 0; it < IT; ++it)
          if (FULL || it * NT + tid < have) m[it] = min_[p0 + it * NT];
      }
#pragma unroll
      for (int it = 0; it < IT; ++it)
        if (FULL || it * NT + tid < have) {
          if (FIRST) {
            key[it] = enc_desc(__uint_as_float(key[it]), bad) - R.kbase;
            idx[it] = p0 + it * NT;
          }
          // (a NaN's key may lie outside the range: the last span and knot)
          const int32_t sp = EQUAL ? equal : spans[min(key[it] >> R.L, (uint32_t)kMsdSpans - 1u)];
          const uint32_t kn = EQUAL ? key[it] >> equal : (key[it] >> (sp & 31)) + (uint32_t)(sp >> 5);
          const uint2 k = map[min(kn, (uint32_t)kMsdKnots - 1u)];
          const uint32_t phi = k.x + __umulhi(__funnelshift_r(idx[it] << ishift, key[it], sp & 31), k.y);
          const uint32_t d = FIRST ? __umulhi(phi, nb1) : __umulhi(phi * nb1, nb2);
          ds[it] = d << 16 | atomicAdd(&cnt[d], 1u);
          if (MASS && FIRST) msum.add(m[it], bad);
        }
    };
    const bool full = have == (uint32_t)TILE;
    if (equal >= 0) {
      if (full) digits(std::true_type{}, std::true_type{});
      else digits(std::false_type{}, std::true_type{});
    } else {
      if (full) digits(std::true_type{}, std::false_type{});
      else digits(std::false_type{}, std::false_type{});
    }
    __syncthreads();
    // starts of the tile's runs, and their places in the buckets' regions
    {
      constexpr int DPT = (kMsdMaxDigits + NT - 1) / NT;
      uint32_t c[DPT], sum = 0;
#pragma unroll
      for (int q = 0; q < DPT; ++q) {
        const uint32_t d = tid * DPT + q;
        c[q] = d < nd ? cnt[d] : 0u;
        sum += c[q];
      }
      uint32_t g[DPT];
#pragma unroll
      for (int q = 0; q < DPT; ++q) {
        const uint32_t d = tid * DPT + q;
        g[q] = 0;
        if (c[q]) g[q] = atomicAdd(FIRST ? &a.mc->cnt1[d * msd_cnt1_step(a.nb1)] : &a.cnt2[bucket * nb2 + d], c[q]);
      }
      uint32_t x = sum;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
      }
      if (lane == 31) wsum[warp] = x;
      __syncthreads();
      uint32_t st = x - sum + warps_before(wsum, NT / 32, lane, warp);
#pragma unroll
      for (int q = 0; q < DPT; ++q) {
        const uint32_t d = tid * DPT + q;
        if (d < nd) {
          cnt[d] = st;
          if (g[q] + c[q] > cap) {
            atomicOr(&a.mc->overflow, FIRST ? 1u : 2u);  // the run is dropped: the other ranking takes over
            gb[d] = 0x80000000u;
          } else {
            gb[d] = (FIRST ? d * cap : (bucket * nb2 + d) * cap) + g[q] - st;
          }
          st += c[q];
        }
      }
    }
    __syncthreads();
    auto place = [&](auto full_tag) {
      constexpr bool FULL = decltype(full_tag)::value;
#pragma unroll
      for (int it = 0; it < IT; ++it)
        if (FULL || it * NT + tid < have) {
          const uint32_t d = ds[it] >> 16;
          rec[cnt[d] + (ds[it] & 0xffffu)] = make_uint4(key[it], idx[it], MASS ? __float_as_uint(m[it]) : 0u, d);
        }
      __syncthreads();
#pragma unroll
      for (int it = 0; it < IT; ++it)
        if (FULL || it * NT + tid < have) {
          const uint4 r = rec[it * NT + tid];
          const uint32_t b = gb[r.w];
          if (b != 0x80000000u) {
            const uint32_t g = b + it * NT + tid;
            kvo[g] = make_uint2(r.x, r.y);
            if (MASS) mo[g] = __uint_as_float(r.z);
          }
        }
    };
    if (full) place(std::true_type{});
    else place(std::false_type{});
    if (FIRST && MASS && (++done & 511u) == 0) msum.flush();
  }
  if (FIRST && MASS) {
    if (given_up) {  // fewer than 2^13 masses per thread
      const uint32_t step = nblk * NT;
      uint32_t i = blk * NT + tid;
      for (; i + 7u * step < n; i += 8u * step) {  // (n <= 2^30)
        float m[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) m[q] = min_[i + q * step];
#pragma unroll
        for (int q = 0; q < 8; ++q) msum.add(m[q], bad);
      }
      for (; i < n; i += step) msum.add(min_[i], bad);
    }
    msum.flush();
    u128 t = msum.slow;
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) t += shfl_down_u128(t, o);
    if (lane == 0) wmass[warp] = t;
    __syncthreads();
    if (tid == 0) {
      t = 0;
      for (int w = 0; w < NT / 32; ++w) t += wmass[w];
      a.cta_mass[2 * blk] = (unsigned long long)t;
      a.cta_mass[2 * blk + 1] = (unsigned long long)(t >> 64);
    }
  }
  if (FIRST && __any_sync(0xffffffffu, bad) && lane == 0)
    raise_status(a.status, MASS ? (AMBER_ERR_NONFINITE | AMBER_ERR_INVALID_MASS) : AMBER_ERR_NONFINITE);
}

template <int NT, int IT, bool FIRST, bool MASS>
__global__ void __launch_bounds__(NT, 1024 / NT) k_msd_split(const MsdArgs a) {
  pdl_begin();
  msd_split_body<NT, IT, FIRST, MASS>(a, blockIdx.x, gridDim.x);
}

template <bool FIRST>
__global__ void __launch_bounds__(512, 2) k_msd_split_multi(const MsdArgs* __restrict__ args) {
  __shared__ MsdArgs a;
  if (threadIdx.x == 0) a = args[blockIdx.y];
  __syncthreads();
  msd_split_body<512, kMsdTileA / 512, FIRST, true>(a, blockIdx.x, gridDim.x);
}

// A final bucket's sub-buckets: linear in (key, cell) over what it holds.
struct SubMap {
  int mode;  // 0: by key, 1: by key and cell, 2: by cell
  int ishift;
  uint32_t off, mul_k, mul_i, F;
  __device__ __forceinline__ uint32_t sub(uint32_t key, uint32_t idx) const {
    if (mode == 0) return __umulhi(key - off, mul_k);
    if (mode == 1) return (key - off) * F + __umulhi(idx << ishift, F);
    return mul_i ? __umulhi(idx - off, mul_i) : idx - off;
  }
  // of cells with one key: the place in their sub-bucket as a fraction of 2^32
  __device__ __forceinline__ uint32_t frac(uint32_t idx) const {
    return mode == 0 ? idx << ishift : mode == 1 ? (idx << ishift) * F : (idx - off) * mul_i;
  }
};

// A sub-bucket of more cells than kMsdTies, mostly ties, sends its bucket to
// sort_ties: counting each against all others is quadratic.  Up to kMsdTiesMost it
// may still be counted there.  (With 12 the tails of ordinary fields take it too
// often, 512^3 l = 3 5.47 -> 5.52 ms, with 16 5.48; ranking 1.0e7 cells with 20 a
// value 0.30 ms, with 24 0.37, with 64 0.36.)
constexpr uint32_t kMsdTies = 16, kMsdTiesMost = 64;

// The counts of S sub-buckets (packed 16-bit words) become starts, with the end
// behind the last one; true if one holds more than `limit`.  Called by the whole
// CTA, with a barrier at its end.
template <int NT, int S>
__device__ __forceinline__ bool counts_to_starts(uint32_t* sc, uint32_t* wsum, uint32_t limit) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  uint4* sc4 = reinterpret_cast<uint4*>(sc);
  constexpr int PER = S / 2 / NT;
  static_assert(PER % 4 == 0, "whole 16-byte words per thread");
  uint32_t w[PER], sum = 0;
#pragma unroll
  for (int q = 0; q < PER / 4; ++q) {
    const uint4 v = sc4[tid * (PER / 4) + q];
    w[4 * q] = v.x;
    w[4 * q + 1] = v.y;
    w[4 * q + 2] = v.z;
    w[4 * q + 3] = v.w;
  }
  uint32_t most = 0;
#pragma unroll
  for (int q = 0; q < PER; ++q) most = __vmaxu2(most, w[q]);
#pragma unroll
  for (int q = 0; q < PER; ++q) sum += w[q];  // both 16-bit halves at once (each below 2^13)
  sum = (sum & 0xffffu) + (sum >> 16);
  uint32_t x = sum;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) wsum[warp] = x;
  __syncthreads();
  uint32_t st = x - sum + warps_before(wsum, NT / 32, lane, warp);
#pragma unroll
  for (int q = 0; q < PER; ++q) {
    const uint32_t c0 = w[q] & 0xffffu, c1 = w[q] >> 16;
    w[q] = st | (st + c0) << 16;
    st += c0 + c1;
  }
#pragma unroll
  for (int q = 0; q < PER / 4; ++q)
    sc4[tid * (PER / 4) + q] = make_uint4(w[4 * q], w[4 * q + 1], w[4 * q + 2], w[4 * q + 3]);
  if (tid == NT - 1) sc[S / 2] = st;
  return __syncthreads_or((most & 0xffffu) > limit || (most >> 16) > limit);
}

// The rest of the local sort where a sub-bucket holds more than kMsdTies cells, from
// the starts and the `have` composites in shared memory.  Where the cells of each
// such sub-bucket share one key, they are counted once more, into as many places as
// they are by their cells' fractions.  Where that leaves more than kMsdTiesMost in
// one, or was not possible, the composites are merge sorted: a run of IT per thread in registers, then runs
// pairwise by merge path, pairs that follow on each other untouched; each cell then
// finds its rank by bisection.  Cells and masses end in sidx and smass (over the
// composites).  The cells are read again: kept over the call they would spill in
// every bucket.  Called by the whole CTA.
// Ranking seven octaves with 150 and 600 cells a value, counted against one another
// and now (no ties; digit passes): 2^22 cells 0.49 and 1.16 -> 0.15 ms (0.13;
// 0.19), 1.0e7 1.06 and 2.45 -> 0.28 (0.23; 0.32), 2^27 4.8 and 8.5 -> 3.0 (2.57;
// 2.9).
template <int NT, int IT, int S, bool MASS>
__device__ __noinline__ void sort_ties(uint32_t have, const uint2* __restrict__ kv, const float* __restrict__ mass,
                                       const SubMap* shared_map) {
  static_assert((NT & (NT - 1)) == 0, "runs double up to the whole array");
  extern __shared__ __align__(16) unsigned char smem_raw[];
  unsigned long long* comp = reinterpret_cast<unsigned long long*>(smem_raw);  // [NT IT]
  uint32_t* sc = reinterpret_cast<uint32_t*>(comp + NT * IT);                  // [S/2 + 4]
  const uint16_t* st16 = reinterpret_cast<const uint16_t*>(sc);
  __shared__ uint32_t wsum[NT / 32];
  const int tid = threadIdx.x;
  const SubMap sub = *shared_map;
  uint32_t idx[IT], rank[IT];
  bool sorted;
  {
    uint32_t key[IT];
    bool differ = false, most = false;
#pragma unroll
    for (int it = 0; it < IT; ++it) {
      const uint32_t p = it * NT + tid;
      if (p < have) {
        const uint2 c = kv[p];
        key[it] = c.x;
        idx[it] = c.y;
      }
    }
#pragma unroll
    for (int it = 0; it < IT; ++it) {
      const uint32_t p = it * NT + tid;
      if (p < have) {
        const uint32_t s = sub.sub(key[it], idx[it]), b0 = st16[s], c = st16[s + 1] - b0;
        rank[it] = b0;
        if (c > kMsdTies) {
          rank[it] += __umulhi(sub.frac(idx[it]), c);
          differ |= key[it] != (uint32_t)(comp[b0] >> 32);
          most |= c > kMsdTiesMost;
        }
      }
    }
    if (__syncthreads_or(differ)) {
      sorted = !__syncthreads_or(most);
#pragma unroll
      for (int it = 0; it < IT; ++it)
        if (it * NT + tid < have) rank[it] = sub.sub(key[it], idx[it]);
    } else {
#pragma unroll
      for (int i = 0; i < S / 8 / NT; ++i) reinterpret_cast<uint4*>(sc)[i * NT + tid] = make_uint4(0, 0, 0, 0);
      __syncthreads();
#pragma unroll
      for (int it = 0; it < IT; ++it) {
        const uint32_t p = it * NT + tid;
        if (p < have) {
          const uint32_t s = rank[it];  // below `have`
          const int sh = (s & 1u) * 16;
          rank[it] = s << 16 | ((atomicAdd(&sc[s >> 1], 1u << sh) >> sh) & 0xffffu);
        }
      }
      __syncthreads();
      sorted = !counts_to_starts<NT, S>(sc, wsum, kMsdTiesMost);
#pragma unroll
      for (int it = 0; it < IT; ++it) {
        const uint32_t p = it * NT + tid;
        if (p < have) {
          const uint32_t s = rank[it] >> 16;
          comp[st16[s] + (rank[it] & 0xffffu)] = (unsigned long long)key[it] << 32 | idx[it];
          rank[it] = s;
        }
      }
      __syncthreads();
    }
    if (sorted) {
#pragma unroll
      for (int it = 0; it < IT; ++it) {
        const uint32_t p = it * NT + tid;
        if (p < have) {
          const uint32_t b0 = st16[rank[it]], b1 = st16[rank[it] + 1];
          const unsigned long long me = (unsigned long long)key[it] << 32 | idx[it];
          uint32_t r = b0;
          if (b1 - b0 > 1u)
            for (uint32_t q = b0; q < b1; ++q) r += comp[q] < me;
          rank[it] = r;
        }
      }
    }
  }
  if (!sorted) {
    unsigned long long v[IT];
#pragma unroll
    for (int i = 0; i < IT; ++i) v[i] = (uint32_t)(tid * IT + i) < have ? comp[tid * IT + i] : ~0ull;
#pragma unroll
    for (int r = 0; r < IT; ++r)
#pragma unroll
      for (int i = r & 1; i + 1 < IT; i += 2) {
        const unsigned long long x = v[i], y = v[i + 1];
        v[i] = x < y ? x : y;
        v[i + 1] = x < y ? y : x;
      }
#pragma unroll
    for (int i = 0; i < IT; ++i) comp[tid * IT + i] = v[i];
    __syncthreads();
#pragma unroll 1
    for (int w = 1; w < NT; w *= 2) {
      const int la = w * IT, d = (tid & (2 * w - 1)) * IT;
      const unsigned long long *A = comp + (tid & ~(2 * w - 1)) * IT, *B = A + la;
      const bool apart = A[la - 1] <= B[0];
      if (!apart) {
        int lo = max(0, d - la), hi = min(d, la);  // before this thread's first output: lo of A, d - lo of B
        while (lo < hi) {
          const int mid = (lo + hi) >> 1;
          if (A[mid] <= B[d - 1 - mid]) lo = mid + 1;
          else hi = mid;
        }
        int b = d - lo;
#pragma unroll
        for (int i = 0; i < IT; ++i) {
          const bool from_a = b >= la || (lo < la && A[lo] <= B[b]);
          v[i] = from_a ? A[lo++] : B[b++];
        }
      }
      __syncthreads();
      if (!apart) {
#pragma unroll
        for (int i = 0; i < IT; ++i) comp[tid * IT + i] = v[i];
      }
      __syncthreads();
    }
#pragma unroll
    for (int it = 0; it < IT; ++it) {
      const uint32_t p = it * NT + tid;
      if (p < have) {
        const uint2 c = kv[p];
        const unsigned long long me = (unsigned long long)c.x << 32 | c.y;
        uint32_t lo = 0, hi = have - 1;
        while (lo < hi) {
          const uint32_t mid = (lo + hi) >> 1;
          if (comp[mid] < me) lo = mid + 1;
          else hi = mid;
        }
        idx[it] = c.y;
        rank[it] = lo;
      }
    }
  }
  uint32_t* sidx = reinterpret_cast<uint32_t*>(smem_raw);
  float* smass = reinterpret_cast<float*>(sidx + NT * IT);
  float m[IT];
  if (MASS) {
#pragma unroll
    for (int it = 0; it < IT; ++it)
      if (it * NT + tid < have) m[it] = mass[it * NT + tid];
  }
  __syncthreads();
#pragma unroll
  for (int it = 0; it < IT; ++it) {
    if (it * NT + tid < have) {
      sidx[rank[it]] = idx[it];
      if (MASS) smass[rank[it]] = m[it];
    }
  }
}

// SCAN: with the masses, matched here as well (LIN: see scan.cuh), each redshift
// stored in its place.
template <bool MASS, bool SCAN, bool LIN>
__device__ __forceinline__ void msd_local_body(const MsdArgs& a, const ScanArgs& sa) {
  constexpr int NT = kMsdLocalThreads, IT = kMsdLocalItems, CAP = kMsdCap, S = kMsdSub;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  unsigned long long* comp = reinterpret_cast<unsigned long long*>(smem_raw);  // [CAP]
  uint32_t* sidx = reinterpret_cast<uint32_t*>(smem_raw);                      // [CAP], after comp
  float* smass = reinterpret_cast<float*>(sidx + CAP);                         // [CAP]
  uint32_t* sc = reinterpret_cast<uint32_t*>(comp + CAP);                      // [S/2 + 4] packed 16-bit counts / starts
  ScanShared& SS = *reinterpret_cast<ScanShared*>(sc);                         // after sc
  static_assert(sizeof(ScanShared) <= S * 2, "the scan's shared words lie over the counters");
  __shared__ uint32_t wsum[NT / 32], wlo[NT / 32], whi[NT / 32], wbase[NT / 32];
  __shared__ unsigned long long wmass[NT / 32];
  __shared__ uint32_t s_tile;
  __shared__ SubMap s_map;
  const bool fell = *reinterpret_cast<volatile uint32_t*>(&a.mc->overflow) != 0;
  if (!SCAN && fell) return;  // the fallback has written the ranking
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  uint32_t b = blockIdx.x;
  if (SCAN) {  // buckets in ticket order: the look-back waits only for running CTAs
    if (tid == 0) s_tile = atomicAdd(sa.ticket, 1u);
    __syncthreads();
    b = s_tile;
  }
  uint32_t have, base = 0;
  const uint2* kv = nullptr;
  const float* mv_in = nullptr;
  if (SCAN && fell) {  // a slice of the fallback's ranking
    const uint32_t nb = a.nb1 * a.nb2, n = (uint32_t)a.n, per = (n + nb - 1) / nb;
    base = min(b * per, n);
    have = min(n - base, per);
  } else if (a.nb2 > 1) {
    const uint32_t d = b / a.nb2, e = b - d * a.nb2;
    have = a.cnt2[b];
    kv = a.kv2 + (size_t)b * CAP;
    mv_in = a.mass2 + (size_t)b * CAP;
    for (uint32_t i = tid; i < d; i += NT) base += a.mc->cnt1[i * msd_cnt1_step(a.nb1)];
    for (uint32_t i = tid; i < e; i += NT) base += a.cnt2[d * a.nb2 + i];
  } else {
    have = a.mc->cnt1[b * msd_cnt1_step(a.nb1)];
    kv = a.kv1 + (size_t)b * a.cap1;
    mv_in = a.mass1 + (size_t)b * a.cap1;
    for (uint32_t i = tid; i < b; i += NT) base += a.mc->cnt1[i * msd_cnt1_step(a.nb1)];
  }
  const float qs = SCAN ? __int_as_float((127 + *sa.qshift) << 23) : 0.f;
  LookBack lb;
  lb.done = true;
  if (SCAN && fell) {
    const int side = (a.ctrl->npasses - 1) & 1;
#pragma unroll
    for (int it = 0; it < IT; ++it) {
      const uint32_t p = it * NT + tid;
      if (p < have) {
        sidx[p] = a.fb_order[side][base + p];
        smass[p] = a.fb_mass[side][base + p];
      }
    }
  } else {
    uint4* sc4 = reinterpret_cast<uint4*>(sc);
#pragma unroll
    for (int i = 0; i < S / 8 / NT; ++i) sc4[i * NT + tid] = make_uint4(0, 0, 0, 0);
    uint32_t key[IT], idx[IT], ss[IT];
    float m[IT];
    uint32_t lo = 0xffffffffu, hi = 0;
    unsigned long long msum = 0;
#pragma unroll
    for (int it = 0; it < IT; ++it) {
      const uint32_t p = it * NT + tid;
      if (p < have) {
        const uint2 v = kv[p];
        key[it] = v.x;
        idx[it] = v.y;
        if (MASS) m[it] = mv_in[p];
      }
    }
#pragma unroll
    for (int it = 0; it < IT; ++it) {
      const uint32_t p = it * NT + tid;
      if (p < have) {
        lo = min(lo, key[it]);
        hi = max(hi, key[it]);
        if (SCAN) msum += mass_fix(m[it], qs);
      }
    }
    base = __reduce_add_sync(0xffffffffu, base);
    lo = __reduce_min_sync(0xffffffffu, lo);
    hi = __reduce_max_sync(0xffffffffu, hi);
    if (SCAN) {
#pragma unroll
      for (int o = 16; o >= 1; o >>= 1) msum += __shfl_down_sync(0xffffffffu, msum, o);
    }
    if (lane == 0) {
      wbase[warp] = base;
      wlo[warp] = lo;
      whi[warp] = hi;
      if (SCAN) wmass[warp] = msum;
    }
    __syncthreads();
    base = __reduce_add_sync(0xffffffffu, lane < NT / 32 ? wbase[lane] : 0u);
    lo = __reduce_min_sync(0xffffffffu, lane < NT / 32 ? wlo[lane] : 0xffffffffu);
    hi = __reduce_max_sync(0xffffffffu, lane < NT / 32 ? whi[lane] : 0u);
    if (SCAN && warp == 0) {
      // the bucket's mass is known before its order: successors can pass over
      // this bucket, and its own look-back runs beside the sort
      unsigned long long t = lane < NT / 32 ? wmass[lane] : 0ull;
#pragma unroll
      for (int o = 16; o >= 1; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
      lb.start(sa, b, t, lane);
    }
    const uint32_t span = hi - lo;
    SubMap sub{0, a.idx_shift, lo, 0, 0, 0};
    if (span >= (uint32_t)S - 1u) {
      sub.mul_k = __float2uint_rz((float)S * 4294967296.0f / ((float)span + 1.0f) * 0.9999f);
    } else if (span > 0) {
      sub.mode = 1;
      sub.F = (uint32_t)S / (span + 1u);
    } else {
      sub.mode = 2;
      uint32_t ilo = 0xffffffffu, ihi = 0;
#pragma unroll
      for (int it = 0; it < IT; ++it) {
        const uint32_t p = it * NT + tid;
        if (p < have) {
          ilo = min(ilo, idx[it]);
          ihi = max(ihi, idx[it]);
        }
      }
      ilo = __reduce_min_sync(0xffffffffu, ilo);
      ihi = __reduce_max_sync(0xffffffffu, ihi);
      __syncthreads();
      if (lane == 0) {
        wlo[warp] = ilo;
        whi[warp] = ihi;
      }
      __syncthreads();
      ilo = __reduce_min_sync(0xffffffffu, lane < NT / 32 ? wlo[lane] : 0xffffffffu);
      ihi = __reduce_max_sync(0xffffffffu, lane < NT / 32 ? whi[lane] : 0u);
      sub.off = ilo;
      const uint32_t isp = ihi - ilo;
      sub.mul_i = isp >= (uint32_t)S - 1u
                  ? __float2uint_rz((float)S * 4294967296.0f / ((float)isp + 1.0f) * 0.9999f)
                  : 0u;  // 0: the offset itself
    }
    if (tid == 0) s_map = sub;
#pragma unroll
    for (int it = 0; it < IT; ++it) {
      const uint32_t p = it * NT + tid;
      if (p < have) {
        const uint32_t s = sub.sub(key[it], idx[it]);
        const int sh = (s & 1u) * 16;
        ss[it] = s << 16 | ((atomicAdd(&sc[s >> 1], 1u << sh) >> sh) & 0xffffu);
      }
    }
    if (SCAN && warp == 0) lb.poll(sa, lane);
    __syncthreads();
    const bool ties = counts_to_starts<NT, S>(sc, wsum, kMsdTies);
    const uint16_t* st16 = reinterpret_cast<const uint16_t*>(sc);
#pragma unroll
    for (int it = 0; it < IT; ++it) {
      const uint32_t p = it * NT + tid;
      if (p < have) {
        const uint32_t s = ss[it] >> 16, b0 = st16[s];
        comp[b0 + (ss[it] & 0xffffu)] = (unsigned long long)key[it] << 32 | idx[it];
        ss[it] = s << 16 | b0;
      }
    }
    if (SCAN && warp == 0) lb.poll(sa, lane);
    __syncthreads();
    if (ties) {  // uniform
      sort_ties<NT, IT, S, MASS>(have, kv, mv_in, &s_map);
      if (SCAN && warp == 0) lb.poll(sa, lane);
    } else {
#pragma unroll
      for (int it = 0; it < IT; ++it) {
        const uint32_t p = it * NT + tid;
        if (p < have) {
          const uint32_t b0 = ss[it] & 0xffffu, b1 = st16[(ss[it] >> 16) + 1];
          uint32_t r = b0;
          if (b1 - b0 > 1u) {
            const unsigned long long me = (unsigned long long)key[it] << 32 | idx[it];
            for (uint32_t q = b0; q < b1; ++q) r += comp[q] < me;
          }
          ss[it] = r;
        }
      }
      if (SCAN && warp == 0) lb.poll(sa, lane);
      __syncthreads();
#pragma unroll
      for (int it = 0; it < IT; ++it) {
        const uint32_t p = it * NT + tid;
        if (p < have) {
          sidx[ss[it]] = idx[it];
          if (MASS) smass[ss[it]] = m[it];
        }
      }
    }
  }
  if (SCAN) scan_clear<NT>(SS, 0);  // the starts were read before the last barrier
  __syncthreads();
  if (!SCAN || a.order) {
#pragma unroll
    for (int it = 0; it < IT; ++it) {
      const uint32_t p = it * NT + tid;
      if (p < have) {
        a.order[base + p] = sidx[p];
        if (MASS) a.mass_out[base + p] = smass[p];
      }
    }
  }
  if constexpr (SCAN) {
    uint32_t cell[IT];
    float mv[IT];
    unsigned long long run = 0;
#pragma unroll
    for (int i = 0; i < IT; ++i) {
      const uint32_t p = tid * IT + i;
      cell[i] = p < have ? sidx[p] : 0u;
      mv[i] = p < have ? smass[p] : 0.f;
      run += mass_fix(mv[i], qs);
    }
    // (the fallback's slices have not started their look-back)
    if (fell)
      scan_tile<NT, IT, false, false, true, false, LIN>(sa, SS, lb, b, base, (int)have, cell, mv, run, qs, sidx, smass,
                                                        nullptr, nullptr);
    else
      scan_tile<NT, IT, false, true, true, false, LIN>(sa, SS, lb, b, base, (int)have, cell, mv, run, qs, sidx, smass,
                                                       nullptr, nullptr);
  }
}

template <bool MASS, bool SCAN, bool LIN>
__global__ void __launch_bounds__(kMsdLocalThreads, 2) k_msd_local(const MsdArgs a, const ScanArgs sa) {
  pdl_begin();
  msd_local_body<MASS, SCAN, LIN>(a, sa);
}

template <bool LIN>
__global__ void __launch_bounds__(kMsdLocalThreads, 2)
    k_msd_local_multi(const MsdArgs* __restrict__ args, const ScanArgs* __restrict__ scans) {
  __shared__ MsdArgs a;
  __shared__ ScanArgs sa;
  if (threadIdx.x == 0) a = args[blockIdx.y];
  if (threadIdx.x == 32) sa = scans[blockIdx.y];
  __syncthreads();
  msd_local_body<true, true, LIN>(a, sa);
}

// ---------------------------------------------------------------------------
// Host side.
// ---------------------------------------------------------------------------
MsdPlan msd_plan(int64_t n, bool with_mass, int num_sms) {
  MsdPlan p{};
  // small fields: at least a CTA of the local sort for each of its places
  const int64_t avg = std::min<int64_t>(kMsdAvg, std::max<int64_t>(kMsdMinAvg, n / (2 * num_sms)));
  const uint32_t nb = (uint32_t)((n + avg - 1) / avg);
  if (nb <= (uint32_t)kMsdMaxDigits) {
    p.nb1 = nb;
    p.nb2 = 1;
    p.cap1 = (uint32_t)std::min<int64_t>(kMsdCap, (avg + avg / 5 + 64 + 31) / 32 * 32);
  } else {
    uint32_t r = 1;
    while ((uint64_t)r * r < nb) ++r;
    p.nb1 = p.nb2 = r;
    const uint64_t per = (uint64_t)(n + r - 1) / r;
    p.cap1 = (uint32_t)((per + per / 32 + 1024 + 31) / 32 * 32);
  }
  int lg = 1;
  while (((int64_t)1 << lg) < n) ++lg;
  p.idx_shift = 32 - lg;
  p.fine = msd_fine(n);
  const int64_t c1 = (int64_t)p.nb1 * p.cap1, c2 = p.nb2 > 1 ? (int64_t)p.nb1 * p.nb2 * kMsdCap : 0;
  p.kv1 = 2 * c1;
  p.m1 = with_mass ? c1 : 0;
  p.kv2 = 2 * c2;
  p.m2 = with_mass ? c2 : 0;
  return p;
}

static int split_tile(uint32_t digits) { return digits > kMsdManyDigits ? kMsdTileB : kMsdTileA; }

// (A batch launches as many of its 4096-cell CTAs per ranking, with as many mass
// sums: 152 at 128^3, where twice that gave 5 items 0.446 instead of 0.455 ms and
// 32 items 2.50 instead of 2.46.)
int msd_split_ctas(int64_t n, const MsdPlan& p, int num_sms) {
  const int tile = split_tile(p.nb1);
  return (int)std::min<int64_t>((n + tile - 1) / tile, (int64_t)num_sms * (tile == kMsdTileB ? 1 : 2));
}

template <int NT, int IT, bool FIRST, bool MASS>
static void launch_split_v(const MsdArgs& a, int grid, cudaStream_t s) {
  constexpr size_t smem = (size_t)NT * IT * 16 + kMsdKnots * 8 + kMsdSpans * 4 + 2 * kMsdMaxDigits * 4;
  static PerDeviceOnce attr;  // per instantiation and device
  once_on_device(attr, [&](DeviceSetUp& u) {
    u.smem(k_msd_split<NT, IT, FIRST, MASS>, smem);
  });
  launch_pdl(k_msd_split<NT, IT, FIRST, MASS>, grid, NT, smem, s, a);
}
template <bool FIRST, bool MASS>
static void launch_split(const MsdArgs& a, int grid, cudaStream_t s) {
  // (nb2, if more than 1, is nb1: both splits take the same tiles)
  if (split_tile(a.nb1) == kMsdTileB) launch_split_v<1024, kMsdTileB / 1024, FIRST, MASS>(a, grid, s);
  else launch_split_v<512, kMsdTileA / 512, FIRST, MASS>(a, grid, s);
}

template <bool MASS, bool SCAN, bool LIN>
static void launch_local(const MsdArgs& a, const ScanArgs& sa, cudaStream_t s) {
  constexpr size_t smem = (size_t)kMsdCap * 8 + (kMsdSub / 2 + 4) * 4;
  static PerDeviceOnce attr;
  once_on_device(attr, [&](DeviceSetUp& u) {
    u.smem(k_msd_local<MASS, SCAN, LIN>, smem);
  });
  launch_pdl(k_msd_local<MASS, SCAN, LIN>, a.nb1 * a.nb2, kMsdLocalThreads, smem, s, a, sa);
}

template <int FINE> static void launch_map(const MsdArgs& a, int grid, cudaStream_t s) {
  constexpr size_t smem = (size_t)(kMsdSpans << FINE) * 4;
  static PerDeviceOnce attr;
  once_on_device(attr, [&](DeviceSetUp& u) {
    u.smem(k_msd_map<FINE>, smem);
  });
  launch_pdl(k_msd_map<FINE>, grid, 1024, smem, s, a);
}

cudaError_t msd_run(const MsdArgs& a, const FallbackArgs& f, int num_sms, const ThreshArgs* ta, const ScanArgs* sa,
                    cudaStream_t s, FftProfile* prof) {
  const int sg = (int)std::max<int64_t>(1, std::min<int64_t>(num_sms * 2, (a.n + 8191) / 8192));
  prof_begin(prof, PK_SORT_HIST, s);
  if (a.fine == 5) launch_map<5>(a, sg, s);
  else if (a.fine == 4) launch_map<4>(a, sg, s);
  else launch_map<3>(a, sg, s);
  prof_end(prof, PK_SORT_HIST, s);
  const int g1 = msd_split_ctas(a.n, MsdPlan{a.nb1, a.nb2, a.cap1}, num_sms);
  prof_begin(prof, PK_SORT_PASS, s);
  if (a.mass) launch_split<true, true>(a, g1, s);
  else launch_split<true, false>(a, g1, s);
  prof_end(prof, PK_SORT_PASS, s);
  if (a.nb2 > 1) {
    prof_begin(prof, PK_SORT_PASS, s);
    if (a.mass) launch_split<false, true>(a, g1, s);
    else launch_split<false, false>(a, g1, s);
    prof_end(prof, PK_SORT_PASS, s);
  }
  if (sa) {
    prof_begin(prof, PK_THRESHOLDS, s);
    thresholds_launch(*ta, s);
    prof_end(prof, PK_THRESHOLDS, s);
  }
  cudaError_t e = sort_fallback(f, a.mass != nullptr, num_sms, s);
  if (e != cudaSuccess) return e;
  if (sa) {
    prof_begin(prof, PK_SCAN_ASSIGN, s);
    if (sa->weighting != AMBER_WEIGHT_MASS) launch_local<true, true, true>(a, *sa, s);
    else launch_local<true, true, false>(a, *sa, s);
    prof_end(prof, PK_SCAN_ASSIGN, s);
  } else {
    prof_begin(prof, PK_SORT_PASS, s);
    if (a.mass) launch_local<true, false, false>(a, ScanArgs{}, s);
    else launch_local<false, false, false>(a, ScanArgs{}, s);
    prof_end(prof, PK_SORT_PASS, s);
  }
  return cudaGetLastError();
}

cudaError_t msd_multi(const MsdMulti& m, int num_sms, cudaStream_t s) {
  constexpr size_t msmem = (size_t)(kMsdSpans << kMsdMaxFine) * 4;
  constexpr size_t ssmem = (size_t)kMsdTileA * 16 + kMsdKnots * 8 + kMsdSpans * 4 + 2 * kMsdMaxDigits * 4;
  constexpr size_t lsmem = (size_t)kMsdCap * 8 + (kMsdSub / 2 + 4) * 4;
  static PerDeviceOnce attr;  // per device
  once_on_device(attr, [&](DeviceSetUp& u) {
    u.smem(k_msd_map_multi<5>, msmem);
    u.smem(k_msd_split_multi<true>, ssmem);
    u.smem(k_msd_split_multi<false>, ssmem);
    u.smem(k_msd_local_multi<true>, lsmem);
    u.smem(k_msd_local_multi<false>, lsmem);
  });
  const dim3 g((unsigned)m.split_ctas, (unsigned)m.M);
  const dim3 gm((unsigned)num_sms, (unsigned)m.M);
  if (m.fine == 5) k_msd_map_multi<5><<<gm, 1024, msmem, s>>>(m.args);
  else k_msd_map_multi<4><<<gm, 1024, msmem / 2, s>>>(m.args);  // (sizes from 64^3 up)
  k_msd_split_multi<true><<<g, 512, ssmem, s>>>(m.args);
  if (m.two_splits) k_msd_split_multi<false><<<g, 512, ssmem, s>>>(m.args);
  return sort_fallback_multi(m.fallback, m.M, m.tiles, num_sms, s);
}

void msd_multi_match(const MsdMulti& m, cudaStream_t s) {
  constexpr size_t lsmem = (size_t)kMsdCap * 8 + (kMsdSub / 2 + 4) * 4;
  for (int f = 0; f < 2; ++f) {
    if (!m.Mg[f]) continue;
    const dim3 g((unsigned)m.buckets, (unsigned)m.Mg[f]);
    const MsdArgs* a = m.args + (f ? m.Mg[0] : 0);
    const ScanArgs* sa = m.scans + (f ? m.Mg[0] : 0);
    if (f) k_msd_local_multi<true><<<g, kMsdLocalThreads, lsmem, s>>>(a, sa);
    else k_msd_local_multi<false><<<g, kMsdLocalThreads, lsmem, s>>>(a, sa);
  }
}

}  // namespace amber
