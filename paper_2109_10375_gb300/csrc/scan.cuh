// The scan of abundance matching over one tile of consecutive ranks (Sec.
// 3.4.2): prefix masses by decoupled look-back, table brackets, redshifts, and
// the tile's (cell, z) pairs grouped by bucket of cells.  Shared by the scan of
// a given ranking (assign.cu) and by the local sort that ends a ranking
// (msd.cu), which runs it on its sorted cells.
#pragma once

#include "assign.cuh"

namespace amber {

// Cell mass in the scan's 64-bit fixed point: floor(m 2^s), s chosen per call
// by k_thresholds so the total stays below 2^62.  Each cell loses less than
// 2^-s, so over n cells F_n is off by less than n 2^-s / T <= n 2^-62 (2e-10
// relative at 2^30 cells) -- far inside an FP64 running sum's own error.
// scale = 2^s: scaling by a power of two is exact, so this is floor_u64 of
// m 2^s (below 2^62 for every valid mass, since m <= T); masses the total pass
// flagged count as 0.
__device__ __forceinline__ unsigned long long mass_fix(float m, float scale) {
  return (m >= 0.0f && m < 1099511627776.0f) ? floor_u64(m * scale) : 0ull;
}

// u64 -> float from its two 32-bit halves (within two roundings; only the
// interpolation weight uses it)
__device__ __forceinline__ float u64_to_float(unsigned long long x) {
  return fmaf(__uint2float_rn((uint32_t)(x >> 32)), 4294967296.0f, __uint2float_rn((uint32_t)x));
}

// Look-back word of a scan tile: 2 flag bits over a 62-bit prefix.
constexpr unsigned long long kScanAgg = 1ull << 62;
constexpr unsigned long long kScanInc = 2ull << 62;
constexpr unsigned long long kScanMask = 3ull << 62;
constexpr unsigned long long kScanValue = (1ull << 62) - 1ull;

__device__ __forceinline__ unsigned long long ld_relaxed_u64(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_relaxed_u64(unsigned long long* p, unsigned long long v) {
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

// One round of a warp-wide 32-ary search for c = #{j : X_j >= v} (X
// non-increasing), c known to lie in [lo, hi]: lane k probes lo + k step; the
// probes that hold form a prefix, and the range shrinks below step.
__device__ __forceinline__ void count_ge_round(const unsigned long long* __restrict__ X, unsigned long long v,
                                               int& lo, int& hi, int lane) {
  if (lo >= hi) return;  // warp-uniform
  const int step = (hi - lo + 31) >> 5;
  const int q = lo + lane * step;
  const bool t = q < hi && X[q] >= v;
  const int c = __popc(__ballot_sync(0xffffffffu, t));
  const int nlo = c ? lo + (c - 1) * step + 1 : lo;
  const int nhi = min(hi, lo + c * step);
  lo = nlo;
  hi = nhi;
}

constexpr int kScanWin = 64;  // thresholds one tile may span, staged in shared memory

// Largest j in (jall, js] whose margin at (u, v) is not negative, jall if none,
// for the lanes that ask: lane after lane, the warp testing 32 points at once.
// (One lane stepping down 253 points for each of its cells took 120 us.)
static __device__ __noinline__ int lin_walk_far(const ScanArgs& a, bool head, float u, float v, int js, int jall,
                                                bool far) {
  const int lane = threadIdx.x & 31;
  unsigned need = __ballot_sync(0xffffffffu, far);
  while (need) {
    const int src = __ffs(need) - 1;
    need &= need - 1;
    const float us = __shfl_sync(0xffffffffu, u, src), vs = __shfl_sync(0xffffffffu, v, src);
    const float* C = __shfl_sync(0xffffffffu, (int)head, src) ? a.linP : a.linQ;
    int found = jall;
    for (int top = __shfl_sync(0xffffffffu, js, src); top > jall; top -= 32) {
      const int j = top - lane;
      const unsigned m = __ballot_sync(
          0xffffffffu, j > jall && fmaf(a.linb[max(j, 0)], vs, fmaf(a.lina[max(j, 0)], us, C[max(j, 0)])) >= 0.0f);
      if (m) {
        found = top - (__ffs(m) - 1);
        break;
      }
    }
    if (lane == src) js = found;
  }
  return js;
}

struct ScanShared {
  int s_jall, s_jtop;
  int s_cx[3];  // c(M_last), c(M_first), first staged threshold (-1: none)
  unsigned long long wtot[32];
  unsigned long long s_excl;
  unsigned long long sX[kScanWin];
  float sInv[kScanWin];
  uint32_t scnt[kMaxBuckets];
  uint32_t soff[kMaxBuckets + 1];
};

// Clears what scan_tile needs cleared (followed by a barrier before it).
template <int NT> __device__ __forceinline__ void scan_clear(ScanShared& S, int nbuckets) {
  if (threadIdx.x == 0) {
    S.s_jall = -1;
    S.s_jtop = -1;
  }
  for (int b = threadIdx.x; b < nbuckets; b += NT) S.scnt[b] = 0;
}

// Decoupled look-back of one tile, run by one warp: each lane holds one
// predecessor's word, so a round trip covers 32 tiles; aggregates are summed
// back to the nearest inclusive prefix.  A round can be tried without waiting
// (step), so that a tile with other work to do looks back meanwhile.
struct LookBack {
  unsigned long long word, excl;
  int64_t t;
  bool done;
  __device__ __forceinline__ void issue(const ScanArgs& a, int lane) {
    word = (t - lane >= 0) ? ld_relaxed_u64(a.state + t - lane) : kScanInc;
  }
  // publish this tile's aggregate and load the first predecessors' words
  __device__ __forceinline__ void start(const ScanArgs& a, uint32_t tile, unsigned long long tile_sum, int lane) {
    if (lane == 0) st_relaxed_u64(a.state + tile, (tile == 0 ? kScanInc : kScanAgg) | tile_sum);
    excl = 0;
    t = (int64_t)tile - 1;
    done = false;
    issue(a, lane);
  }
  // one round on the loaded words; false when no predecessor had published more
  __device__ __forceinline__ bool step(const ScanArgs& a, int lane) {
    const unsigned long long f = word & kScanMask;
    const unsigned inc_mask = __ballot_sync(0xffffffffu, f == kScanInc);
    const unsigned stop_mask = inc_mask | __ballot_sync(0xffffffffu, f == 0ull);
    const int first = stop_mask ? __ffs(stop_mask) - 1 : 32;
    done = first < 32 && ((inc_mask >> first) & 1u);
    unsigned long long part = (lane < first || (done && lane == first)) ? (word & kScanValue) : 0ull;
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) part += __shfl_down_sync(0xffffffffu, part, o);
    excl += __shfl_sync(0xffffffffu, part, 0);
    if (done) return true;
    t -= first;
    return first == 32;
  }
  __device__ __forceinline__ void poll(const ScanArgs& a, int lane) {
    if (done) return;
    step(a, lane);
    if (!done) issue(a, lane);
  }
  __device__ __forceinline__ unsigned long long finish(const ScanArgs& a, int lane) {
    unsigned spins = 0;
    while (!done) {
      const bool full = step(a, lane);
      if (done) break;
      if (!full) {
        if (++spins >= a.spin_limit) {
          if (lane == 0) raise_status(a.status, AMBER_ERR_DEVICE_TIMEOUT);
          break;
        }
        __nanosleep(20);
      }
      issue(a, lane);
    }
    return excl;
  }
};

// Ranks start .. start + cnt - 1: thread tid holds the cells and masses of
// ranks start + tid IT + i (i < IT) and `run`, the sum of their fixed-point
// masses.  scell, sz: NT IT (padded by PAD) staging words, free to be
// overwritten after the next barrier.  EARLY: warp 0's look-back lb has been
// started with the tile's sum; otherwise it is started here.
// The pairs go to bcell, bz + start.
// DIRECT: the redshifts go straight to a.zre in cell order instead (bcell, bz
// and the staging words unused): for fields that stay in L2.
// LIN: a linear weighting (growth or volume).  The exact-integer threshold
// test of the mass weighting is replaced by the margins h_j(n) in FP32: a
// cell takes the largest table point j with h_j >= 0.  A margin is linear in
// (n, M_n), so its extremes over the box that a run of ranks spans lie at the
// corners.  Per tile every point is classified: jall is the largest one that
// ionizes all of its cells, jtop the largest one that can ionize any.  From
// jtop each warp walks down 32 points at a time to the first one its own box
// allows, each thread from there to the first one its 16 ranks allow, and only
// then each cell tests margins.  (The first tile of 128^3 spans over 1000 of
// 2000 points; with every cell testing all of the tile's points it took 1.06 ms.)
template <int NT, int IT, bool PAD, bool EARLY, bool DIRECT, bool WANT_F, bool LIN>
__device__ __forceinline__ void scan_tile(const ScanArgs& a, ScanShared& S, LookBack& lb, uint32_t tile, uint32_t start,
                                          int cnt, const uint32_t* cell, const float* mv, unsigned long long run,
                                          float qs, uint32_t* scell, float* sz, uint32_t* bcell, float* bz) {
  static_assert(DIRECT || (IT % 2 == 0 && NT * IT <= 65536), "places are packed in pairs of 16 bits");
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t n = (uint32_t)a.n;
  const int M = a.n_table;
  auto at = [](int p) { return PAD ? p + (p >> 5) : p; };
  // block exclusive scan of the thread totals
  unsigned long long x = run;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned long long y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) S.wtot[warp] = x;
  __syncthreads();
  unsigned long long wpre = 0, tile_sum = 0;
#pragma unroll
  for (int w = 0; w < NT / 32; ++w) {
    if (w < warp) wpre += S.wtot[w];
    tile_sum += S.wtot[w];
  }
  const unsigned long long thr_excl = wpre + x - run;

  // warp 0 publishes the tile's aggregate and starts its look-back load; the
  // bucket slots of every cell (which need no prefix) are taken meanwhile
  if (!EARLY && warp == 0) lb.start(a, tile, tile_sum, lane);
  uint32_t slot[(IT + 1) / 2];  // two 16-bit places each: 16 words spilled (512^3 scan 0.77 ms)
  if constexpr (!DIRECT) {
    // one add per cell, or per thread where each thread of the warp holds
    // cells of one bucket only (an order that follows the cells would have
    // all lanes add to one counter cell after cell: identity order at 2^27
    // cells 2.44 ms)
    uint32_t differ = 0;
#pragma unroll
    for (int i = 1; i < IT; ++i) differ |= cell[i] ^ cell[0];
    if (__all_sync(0xffffffffu, (differ >> a.bucket_shift) == 0u && (tid + 1) * IT <= cnt)) {
      const uint32_t base = atomicAdd(&S.scnt[cell[0] >> a.bucket_shift], (uint32_t)IT);
#pragma unroll
      for (int k = 0; k < IT / 2; ++k) slot[k] = (base + 2u * k) * 0x10001u + 0x10000u;
    } else {
#pragma unroll
      for (int i = 0; i < IT; ++i) {
        const uint32_t t = (tid * IT + i < cnt) ? atomicAdd(&S.scnt[cell[i] >> a.bucket_shift], 1u) : 0u;
        slot[i / 2] = i % 2 ? slot[i / 2] | t << 16 : t;
      }
    }
  }
  __syncthreads();

  if (warp == 0) {
    const unsigned long long excl = lb.finish(a, lane);
    if (lane == 0) {
      if (tile != 0) st_relaxed_u64(a.state + tile, kScanInc | ((excl + tile_sum) & kScanValue));
      S.s_excl = excl;
    }
    // bracket the whole tile: c(M) = #{j : X_j >= M} at its first and last
    // prefix, both searched at once (three round trips for 2000 thresholds)
    int lo0 = 0, hi0 = LIN ? 0 : M, lo1 = 0, hi1 = LIN ? 0 : M;
    while (lo0 < hi0 || lo1 < hi1) {
      count_ge_round(a.Xq, excl, lo0, hi0, lane);
      count_ge_round(a.Xq, excl + tile_sum, lo1, hi1, lane);
    }
    // thresholds the tile's cells can touch: X_j for j in [c_last - 1, c_first]
    const int base = max(lo1 - 1, 0), L = min(lo0, M - 1) - base + 1;
    const bool stage = !LIN && L <= kScanWin;
    if (stage) {
      for (int i = lane; i < L; i += 32) {
        S.sX[i] = a.Xq[base + i];
        S.sInv[i] = (base + i < M - 1) ? a.inv_dx[base + i] : 0.0f;
      }
    }
    if (lane == 0) {
      S.s_cx[0] = lo1;
      S.s_cx[1] = lo0;
      S.s_cx[2] = stage ? base : -1;
    }
  } else if (!DIRECT && warp == 1) {
    // tile-local bucket starts (exclusive scan over the buckets) and this
    // tile's row of the offset table
    uint32_t carry = 0;
    uint16_t* row = a.btab + (int64_t)tile * (a.nbuckets + 1);
    for (int b0 = 0; b0 < a.nbuckets; b0 += 32) {
      const int b = b0 + lane;
      const uint32_t c = b < a.nbuckets ? S.scnt[b] : 0u;
      uint32_t y = c;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t z = __shfl_up_sync(0xffffffffu, y, o);
        if (lane >= o) y += z;
      }
      if (b < a.nbuckets) {
        S.soff[b] = carry + y - c;
        row[b] = (uint16_t)(carry + y - c);
      }
      carry += __shfl_sync(0xffffffffu, y, 31);
    }
    if (lane == 0) {
      S.soff[a.nbuckets] = carry;
      row[a.nbuckets] = (uint16_t)carry;
    }
  }
  __syncthreads();
  unsigned long long Mn = S.s_excl + thr_excl;
  const double invT = WANT_F ? 1.0 / (double)*a.qtotal : 0.0;
  const float qinv = __int_as_float((127 - *a.qshift) << 23);  // 2^-s: fixed point -> mass units
  const unsigned long long qT = LIN ? *a.qtotal : 0ull;  // total in the prefix's fixed point (>= every M_n)
  // head form (ranks in the first half) or tail form, for the tile's box:
  // h = C_j + sa alpha_j u + sa beta_j v with (C, u, v, sa) = (x W_N, n, M_n, -1)
  // or ((x - 1) W_N, N - n, T - M_n, +1)
  const bool head = start + (uint32_t)cnt / 2u <= n / 2u;
  const float* linC = head ? a.linP : a.linQ;
  const float sa = head ? -1.0f : 1.0f;
  // table point j over the box of ranks (r0, r1] (from 0) with prefix masses
  // in [m0, m1]: bounds of its margin and the rounding they are good to
  struct Box { float u0, u1, v0, v1; };
  auto box_of = [&](uint32_t r0, uint32_t r1, unsigned long long m0, unsigned long long m1) -> Box {
    if (head) return {(float)(r0 + 1u), (float)r1, u64_to_float(m0) * qinv, u64_to_float(m1) * qinv};
    return {(float)(n - r1), (float)(n - (r0 + 1u)), u64_to_float(qT - m1) * qinv, u64_to_float(qT - m0) * qinv};
  };
  auto classify = [&](const Box& x, int j, float& hmin, float& hmax, float& tol) {
    const float Cj = linC[j], al = sa * a.lina[j], be = sa * a.linb[j];
    const float au0 = al * x.u0, au1 = al * x.u1, bv0 = be * x.v0, bv1 = be * x.v1;
    hmin = Cj + fminf(au0, au1) + fminf(bv0, bv1);
    hmax = Cj + fmaxf(au0, au1) + fmaxf(bv0, bv1);
    tol = 4e-7f * (fabsf(Cj) + fmaxf(fabsf(au0), fabsf(au1)) + fmaxf(fabsf(bv0), fabsf(bv1)));
  };
  if constexpr (LIN) {
    const Box tb = box_of(start, start + (uint32_t)cnt, S.s_excl, S.s_excl + tile_sum);
    int ja = -1, jt = -1;
    for (int j = tid; j < M; j += NT) {
      float hmin, hmax, tol;
      classify(tb, j, hmin, hmax, tol);
      if (hmin >= tol) ja = j;
      if (hmax >= -tol) jt = j;
    }
    ja = __reduce_max_sync(0xffffffffu, ja);
    jt = __reduce_max_sync(0xffffffffu, jt);
    if (lane == 0) {
      if (ja >= 0) atomicMax(&S.s_jall, ja);
      if (jt >= 0) atomicMax(&S.s_jtop, jt);
    }
    __syncthreads();
  }
  const int cx_lo = S.s_cx[0], cx_hi = S.s_cx[1], wb = S.s_cx[2];
  // threshold j from the staged window when the tile fits it
  auto Xj = [&](int j) -> unsigned long long { return wb >= 0 ? S.sX[j - wb] : a.Xq[j]; };
  auto Ij = [&](int j) -> float { return wb >= 0 ? S.sInv[j - wb] : a.inv_dx[j]; };

  // a cell's redshift: to its bucket-ordered staging slot (order and masses
  // were consumed above), or straight to its place
  auto put = [&](int i, float z) {
    if constexpr (DIRECT) {
      a.zre[cell[i]] = z;
    } else {
      const uint32_t q = S.soff[cell[i] >> a.bucket_shift] + (i % 2 ? slot[i / 2] >> 16 : slot[i / 2] & 0xffffu);
      scell[at(q)] = cell[i];
      sz[at(q)] = z;
    }
  };
  // bracket: cx = #{j : X_j >= M_n}; X is non-increasing in j and M_n grows
  // with rank, so each thread searches the tile's range once, then walks
  // down.  Each (cell, z) goes straight to its bucket-ordered staging slot
  // (order and masses were consumed above, so their shared arrays are free).
  if (LIN && S.s_jtop <= S.s_jall) {
    // no table point above max{j : all ionized} can ionize any cell of the
    // tile: every cell takes j* = jall, whose two margin rows are held in
    // registers
    const int js = S.s_jall;
    const bool mid = js >= 0 && js < M - 1;
    float la0 = 0.f, lb0 = 0.f, P0 = 0.f, Q0 = 0.f, la1 = 0.f, lb1 = 0.f, P1 = 0.f, Q1 = 0.f;
    if (mid) {
      la0 = a.lina[js], lb0 = a.linb[js], P0 = a.linP[js], Q0 = a.linQ[js];
      la1 = a.lina[js + 1], lb1 = a.linb[js + 1], P1 = a.linP[js + 1], Q1 = a.linQ[js + 1];
    }
    const float zc = js < 0 ? a.z_lo : a.z_hi;
#pragma unroll
    for (int i = 0; i < IT; ++i) {
      const int p = tid * IT + i;
      if (p >= cnt) continue;
      Mn += mass_fix(mv[i], qs);
      float z = zc;
      if (mid) {
        const uint32_t rank1 = start + (uint32_t)p + 1u;
        const bool chead = rank1 <= n / 2u;
        const float cs = chead ? -1.0f : 1.0f;
        const float uu = cs * (chead ? (float)rank1 : (float)(n - rank1));
        const float vv = cs * (chead ? u64_to_float(Mn) * qinv : u64_to_float(qT - Mn) * qinv);
        const float h0 = fmaf(lb0, vv, fmaf(la0, uu, chead ? P0 : Q0));
        const float h1 = fmaf(lb1, vv, fmaf(la1, uu, chead ? P1 : Q1));
        float t = h0 / (h0 - h1);
        t = fminf(fmaxf(t, 0.0f), 0.99999994f);
        z = a.z_lo + ((float)js + t) * a.dzt;
      }
      if (WANT_F) a.F[start + p] = (double)Mn * invT;
      put(i, z);
    }
  } else if (!LIN && cx_lo == cx_hi) {
    // the whole tile between two thresholds (all but a few tiles): one
    // interval, its threshold and slope held in registers
    const int j = cx_lo - 1;
    const bool mid = j >= 0 && j < M - 1;
    const unsigned long long Xu = mid ? Xj(j) : 0ull;
    const float Iu = mid ? Ij(j) : 0.0f;
    const float zc = j < 0 ? a.z_lo : a.z_hi;
#pragma unroll
    for (int i = 0; i < IT; ++i) {
      const int p = tid * IT + i;
      if (p >= cnt) continue;
      Mn += mass_fix(mv[i], qs);
      float z = zc;
      if (mid) {
        float t = u64_to_float(Xu - Mn) * Iu;
        t = fminf(fmaxf(t, 0.0f), 0.99999994f);
        z = a.z_lo + ((float)j + t) * a.dzt;
      }
      if (WANT_F) a.F[start + p] = (double)Mn * invT;
      put(i, z);
    }
  } else if constexpr (LIN) {
    const int jall = S.s_jall;
    int jt = S.s_jtop;
    {
      // the warp's ranks: 32 points per round from the top down
      const uint32_t w0 = start + (uint32_t)min(warp * 32 * IT, cnt), w1 = start + (uint32_t)min((warp + 1) * 32 * IT, cnt);
      const Box wbx = box_of(w0, w1, S.s_excl + wpre, S.s_excl + wpre + S.wtot[warp]);
      unsigned hit = 0;
      if (w1 > w0) {
        for (; jt > jall; jt -= 32) {
          const int j = jt - lane;
          float hmin, hmax = -1.f, tol = 0.f;
          if (j > jall) classify(wbx, j, hmin, hmax, tol);
          hit = __ballot_sync(0xffffffffu, j > jall && hmax >= -tol);
          if (hit) break;
        }
      }
      jt = hit ? jt - (__ffs(hit) - 1) : jall;
    }
    if (tid * IT < cnt) {
      const Box cb = box_of(start + (uint32_t)(tid * IT), start + (uint32_t)min((tid + 1) * IT, cnt), Mn, Mn + run);
      // mostly a step or two; a long way down eight points at a time, so that
      // their loads overlap
      unsigned hit = 0;
      for (int steps = 0; jt > jall && steps < 6; ++steps, --jt) {
        float hmin, hmax, tol;
        classify(cb, jt, hmin, hmax, tol);
        if (hmax >= -tol) {
          hit = 1;
          break;
        }
      }
#pragma unroll 1
      for (; jt > jall && !hit; jt -= hit ? __ffs(hit) - 1 : 8) {
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          float hmin, hmax, tol;
          classify(cb, max(jt - k, 0), hmin, hmax, tol);
          hit |= (jt - k > jall && hmax >= -tol) ? 1u << k : 0u;
        }
      }
      jt = max(jt, jall);
    }
#pragma unroll
    for (int i = 0; i < IT; ++i) {
      const int p = tid * IT + i;
      const bool ok = p < cnt;
      if (ok) Mn += mass_fix(mv[i], qs);
      // the cell's own form (a tile can straddle the middle rank; the boxes'
      // classification above carries a tolerance for either form)
      const uint32_t rank1 = start + (uint32_t)p + 1u;
      const bool chead = rank1 <= n / 2u;
      const float cs = chead ? -1.0f : 1.0f;
      const float* cC = chead ? a.linP : a.linQ;
      const float uu = cs * (chead ? (float)rank1 : (float)(n - rank1));
      const float vv = cs * (chead ? u64_to_float(Mn) * qinv : u64_to_float(qT - Mn) * qinv);
      auto h = [&](int j) { return fmaf(a.linb[j], vv, fmaf(a.lina[j], uu, cC[j])); };
      int js = ok ? jt : jall, steps = 0;
      while (js > jall && steps < 24 && !(h(js) >= 0.0f)) --js, ++steps;
      // a long way down (the first ranks, and deep voids at the end): 32 points at once
      const bool far = steps == 24 && js > jall;
      if (__any_sync(0xffffffffu, far)) js = lin_walk_far(a, chead, uu, vv, js, jall, far);
      if (!ok) continue;
      float z;
      if (js < 0) z = a.z_lo;
      else if (js == M - 1) z = a.z_hi;
      else {
        const float h0 = h(js), h1 = h(js + 1);
        float t = h0 / (h0 - h1);
        t = fminf(fmaxf(t, 0.0f), 0.99999994f);
        z = a.z_lo + ((float)js + t) * a.dzt;
      }
      if (WANT_F) a.F[start + p] = (double)Mn * invT;
      put(i, z);
    }
  } else {
    int cx = -1;
#pragma unroll
    for (int i = 0; i < IT; ++i) {
      const int p = tid * IT + i;
      if (p >= cnt) continue;
      Mn += mass_fix(mv[i], qs);
      int lo = cx_lo, hi = cx_hi;
      if (cx >= 0) {
        // the prefix grew: gallop down from the last cell's bracket (in a
        // small grid's first tile neighbours lie hundreds of points apart, and
        // stepping through them one dependent load at a time took 63 us at 32^3)
        hi = cx;
        lo = cx;
        for (int step = 1; lo > cx_lo; step *= 2) {
          const int q = max(lo - step, cx_lo);
          if (Xj(q) >= Mn) {
            lo = q + 1;
            break;
          }
          hi = lo = q;
        }
      }
      while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (Xj(mid) >= Mn) lo = mid + 1; else hi = mid;
      }
      cx = lo;
      const int j = cx - 1;
      float z;
      if (j < 0) z = a.z_lo;
      else if (j == M - 1) z = a.z_hi;
      else {
        float t = u64_to_float(Xj(j) - Mn) * Ij(j);
        t = fminf(fmaxf(t, 0.0f), 0.99999994f);
        z = a.z_lo + ((float)j + t) * a.dzt;
      }
      if (WANT_F) a.F[start + p] = (double)Mn * invT;
      put(i, z);
    }
  }
  if constexpr (DIRECT) return;
  __syncthreads();
  // the pairs are read back only after the whole scan: keep them out of L2
  const unsigned long long pol = l2_evict_first();
#pragma unroll
  for (int k = 0; k < IT; ++k) {
    const int p = k * NT + tid;
    if (p < cnt) {
      st_hint(bcell + start + p, scell[at(p)], pol);
      st_hint(bz + start + p, sz[at(p)], pol);
    }
  }
}

}  // namespace amber
