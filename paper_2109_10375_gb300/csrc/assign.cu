// Abundance matching (Sec. 3.4.2): the rank-n cell is ionized at z_n where
// the cumulative mass fraction F_n = M_n / M_total equals the history x(z_n)
// (Sec. 3.1.2, Eq. weibull), with x(z) tabulated on uniform redshifts.
//
//   k_mass_reduce   : M_total = sum of all cell masses (order-free, exact)
//   k_thresholds    : table x_j = x(z_j) and integer thresholds
//                     X_j = floor(x_j * M_total) in the scan's fixed point,
//                     so "x_j >= F_n" is the integer test "X_j >= M_n";
//                     plus 1/(X_j - X_j+1)
//   k_scan_assign   : M_n by a decoupled-look-back prefix sum over ranks,
//                     bracket j* by a search in the thresholds amortised over
//                     each thread's run of ranks, interpolate to z_n, and
//                     write (cell, z_n) into buckets of consecutive cells
//   k_scatter_back  : per bucket, z_re[cell] = z_n; a bucket's cells span a
//                     region small enough to stay in L2, so the permuted
//                     writes reach HBM as whole sectors
//
// The total is summed exactly as 128-bit fixed point with 64 fraction bits.
// The running prefix uses 64-bit fixed point whose shift s is chosen from the
// total so it stays below 2^62: each mass is rounded down to a multiple of
// 2^-s, so F_n is off by at most n 2^-60 (1e-9 at 2^30 cells), and no sum
// depends on the order of addition.  Only the interpolation weight is FP32.
#include <cstdlib>
#include <type_traits>

#include "assign.cuh"
#include "fixed128.cuh"
#include "scan.cuh"
#include "sort.cuh"

namespace amber {

// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_mass_reduce(const float* __restrict__ mass, int64_t n,
                                                     unsigned long long* __restrict__ total,
                                                     unsigned int* __restrict__ status) {
  MassSum sum;
  bool bad = false;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  const int64_t gtid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  // 16-byte loads, four in flight, only from a 16-byte aligned array, else
  // element by element
  const int64_t nvec = (reinterpret_cast<uintptr_t>(mass) & 15) == 0 ? n / 4 : 0;
  const float4* mass4 = reinterpret_cast<const float4*>(mass);
  auto add4 = [&](float4 m) {
    sum.add(m.x, bad);
    sum.add(m.y, bad);
    sum.add(m.z, bad);
    sum.add(m.w, bad);
  };
  int64_t v = gtid;
  for (; v + 3 * stride < nvec; v += 4 * stride) {
    const float4 a = mass4[v], b = mass4[v + stride], c = mass4[v + 2 * stride], d = mass4[v + 3 * stride];
    add4(a);
    add4(b);
    add4(c);
    add4(d);
    sum.flush();
  }
  for (; v < nvec; v += stride) add4(mass4[v]);
  sum.flush();
  for (int64_t i = nvec * 4 + gtid; i < n; i += stride) {
    sum.add(mass[i], bad);
    sum.flush();
  }
  u128 acc = sum.slow;
#pragma unroll
  for (int o = 16; o >= 1; o >>= 1) acc += shfl_down_u128(acc, o);
  __shared__ u128 ws[8];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (lane == 0) ws[warp] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    u128 s = 0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += ws[w];
    if (s != 0) atomic_add_u128(total, s);
  }
  if (__any_sync(0xffffffffu, bad) && lane == 0) raise_status(status, AMBER_ERR_INVALID_MASS);
}

// floor(x * T) for x in [0, 1] and T < 2^128, exactly.
__device__ __forceinline__ u128 mul_floor(double x, u128 T) {
  if (!(x > 0.0)) return 0;
  if (x >= 1.0) return T;
  int ex;
  const double f = frexp(x, &ex);                                    // x = f 2^ex, f in [0.5, 1)
  const unsigned long long mant = (unsigned long long)ldexp(f, 53);  // exact 53-bit integer
  const int s = 53 - ex;                                             // x = mant 2^-s, s >= 53
  const unsigned long long tl = (unsigned long long)T, th = (unsigned long long)(T >> 64);
  const unsigned long long p0 = mant * tl, p0h = __umul64hi(mant, tl);
  const unsigned long long p1 = mant * th, p1h = __umul64hi(mant, th);
  const unsigned long long l1 = p0h + p1;
  const unsigned long long c1 = (l1 < p0h) ? 1ull : 0ull;
  const unsigned long long l2 = p1h + c1;
  // 192-bit product (l2:l1:p0) >> s
  if (s >= 192) return 0;
  const u128 top = ((u128)l2 << 64) | (u128)l1;
  if (s >= 64) return top >> (s - 64);
  return (top << (64 - s)) | (u128)(p0 >> s);
}

// Block sum of the per-tile mass sums first, first + step, ... (valid on thread 0).
__device__ __forceinline__ u128 sum_tile_mass(const unsigned long long* __restrict__ tile_mass, int64_t ntiles,
                                              int64_t first, int64_t step) {
  __shared__ u128 ws[32];
  u128 acc = 0;
  for (int64_t t = first; t < ntiles; t += step) {
    const ulonglong2 v = reinterpret_cast<const ulonglong2*>(tile_mass)[t];
    acc += ((u128)v.y << 64) | (u128)v.x;
  }
#pragma unroll
  for (int o = 16; o >= 1; o >>= 1) acc += shfl_down_u128(acc, o);
  if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = acc;
  __syncthreads();
  u128 s = 0;
  if (threadIdx.x == 0)
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += ws[w];
  return s;
}

// Linear growth factor D(a) of flat LCDM (Omega_m = om, Omega_L = 1 - om),
// normalised to D = a early on: D(a) = (5 om / 2) E(a) int_0^a da'/(a' E(a'))^3
// with E(a) = sqrt(om a^-3 + 1 - om).  In closed form D(a) = a 2F1(1/3, 1;
// 11/6; -x) with x = a^3 (1 - om)/om; its power series converges fast for
// x <= 1/2 (every z above ~0.7 at om = 0.3).  Beyond that the integral is
// taken by Simpson's rule after the substitution a' = s^2, which makes the
// integrand 2 s^4 / (om + (1 - om) s^6)^(3/2) smooth at 0.
__device__ double growth_D(double a, double om) {
  const double ol = 1.0 - om;
  const double x = a * a * a * ol / om;
  if (x <= 0.5) {
    double sum = 0.0, term = 1.0;
    for (int k = 0; k < 200 && fabs(term) > 1e-18 * fabs(sum + 1.0); ++k) {
      sum += term;
      term *= -x * (1.0 / 3.0 + k) / (11.0 / 6.0 + k);
    }
    return a * sum;
  }
  const int S = 2048;  // even
  const double s1 = sqrt(a), hs = s1 / S;
  auto f = [&](double sv) {
    const double s2 = sv * sv, s6 = s2 * s2 * s2;
    const double d = om + ol * s6;
    return 2.0 * s2 * s2 / (d * sqrt(d));
  };
  double acc = f(0.0) + f(s1);
  for (int i = 1; i < S; ++i) acc += (i & 1 ? 4.0 : 2.0) * f(i * hs);
  const double I = acc * hs / 3.0;
  const double E = sqrt(om / (a * a * a) + ol);
  return 2.5 * om * E * I;
}

// Exact total of the ranking's per-tile mass sums into total (zeroed): for
// many tiles, where reading them all in every thresholds CTA would cost more
// than this launch.  (1024^3: 262144 sums, 4 MB, over 64 CTAs.)
__global__ void __launch_bounds__(256) k_tile_total(const unsigned long long* __restrict__ tile_mass, int64_t ntiles,
                                                    unsigned long long* __restrict__ total) {
  const u128 s = sum_tile_mass(tile_mass, ntiles, (int64_t)blockIdx.x * blockDim.x + threadIdx.x,
                               (int64_t)gridDim.x * blockDim.x);
  if (threadIdx.x == 0 && s != 0) atomic_add_u128(total, s);
}

// From the exact total T (2^-64 units) the kernel picks the scan's
// fixed-point shift s (total below 2^62), and tabulates X_j = floor(x_j T
// 2^(s-64)) so "x_j >= F_n" is the integer test "X_j >= M_n", plus
// 1/(X_j - X_j+1) for the interpolation weight.  tile_mass (optional):
// per-tile partial sums from the ranking; every CTA adds them up itself
// (exact, order-free), so no launch is needed for the total.
// The table's exp, pow and growth series run on the FP64 pipe, which takes 16
// cycles per warp instruction here: one warp per CTA evaluates 31 points (and
// the next one, for the difference), so 2000 points spread over 65 SMs, and
// warps 1-7 read the partial sums meanwhile.  One CTA of 1024 threads for the
// whole table took 103 us (growth weighting 255 us); a 32^3 solve went from 256
// to 145 us with this and the scan's gallop, a 128^3 growth one from 1501 to 489.
constexpr int kThreshThreads = 256;
constexpr int kThreshPoints = 31;
// more tile sums than this take a launch of their own (k_tile_total): 4096
// sums are 64 KB read per CTA, about 1 us; 262144 would be 4 MB, over 30 us
constexpr int64_t kTileTotalMin = 4096;

__device__ __forceinline__ void thresholds_body(const ThreshArgs& A, int blk) {
  __shared__ u128 sT;
  const int lane = threadIdx.x & 31, M = A.M;
  const int j = blk * kThreshPoints + lane;
  const bool mine = threadIdx.x < 32 && j < M;
  double x = 0.0, alpha = 1.0, beta = 0.0;  // weight of a cell at z_j: alpha + beta mass (volume weighting: 1)
  if (mine) {
    const double z = A.z_lo + (A.z_hi - A.z_lo) * (double)j / (double)(M - 1);
    const double u = fmax((z - A.a_w) / A.b_w, 0.0);
    x = exp(-pow(u, A.c_w));
    if (A.weighting == AMBER_WEIGHT_MASS_GROWTH) {
      const double g = growth_D(1.0 / (1.0 + z), A.omega_m) / growth_D(1.0 / (1.0 + A.z_mid), A.omega_m);
      alpha = 1.0 - g;
      beta = g;
    }
  }
  pdl_begin();  // the table's values need nothing of the kernels before
  if (A.tile_mass) {
    const u128 s = sum_tile_mass(A.tile_mass, A.ntiles, threadIdx.x, blockDim.x);
    if (threadIdx.x == 0) sT = s;
  } else if (threadIdx.x == 0) {
    sT = ((u128)A.total[1] << 64) | (u128)A.total[0];
  }
  __syncthreads();
  if (threadIdx.x >= 32) return;
  const u128 T = sT;
  // bit length L of T; the real total is below 2^(L-64), so s = 126 - L
  // keeps it below 2^62 (s <= 64: no finer than the exact representation)
  const unsigned long long th = (unsigned long long)(T >> 64), tl = (unsigned long long)T;
  const int L = th ? 128 - __clzll((long long)th) : 64 - __clzll((long long)tl);
  const int s = 126 - L < 64 ? 126 - L : 64;
  const int sh = 64 - s;  // X in 2^-s units: floor(x T) >> (64 - s)
  if (blk == 0 && lane == 0) {
    *A.qshift = s;
    *A.qtotal = (unsigned long long)(sh >= 0 ? (T >> sh) : (T << (-sh)));
  }
  const u128 X = mul_floor(x, T);
  const unsigned long long Xq = mine ? (unsigned long long)(sh >= 0 ? (X >> sh) : (X << (-sh))) : 0ull;
  const unsigned long long next = __shfl_down_sync(0xffffffffu, Xq, 1);
  if (!mine || lane >= kThreshPoints) return;  // lane 31's point belongs to the next CTA
  A.Xq[j] = Xq;
  if (j < M - 1) {
    const unsigned long long d = Xq - next;
    A.inv_dx[j] = d > 0 ? 1.0f / __ull2float_rn(d) : 0.0f;
  }
  if (A.weighting != AMBER_WEIGHT_MASS) {
    // margin h_j(n) = x_j W_N - W_n.  Two equal forms keep the operands small
    // at either end of the ranking: the head form x_j W_N - alpha_j n - beta_j
    // M_n for the first half of the ranks, and the tail form (x_j - 1) W_N +
    // alpha_j (N - n) + beta_j (T - M_n) for the second, where the weight
    // after rank n (all that is left on the x = 1 plateau) comes from exact
    // differences
    const double Treal = u128_to_double(T) * 5.421010862427522e-20;  // 2^-64
    const double WN = alpha * (double)A.ncells + beta * Treal;
    A.lin[j] = (float)(x * WN);
    A.lin[kMaxTable + j] = (float)((x - 1.0) * WN);
    A.lin[2 * kMaxTable + j] = (float)alpha;
    A.lin[3 * kMaxTable + j] = (float)beta;
  }
}

__global__ void __launch_bounds__(kThreshThreads) k_thresholds(const ThreshArgs A) {
  thresholds_body(A, (int)blockIdx.x);
}

// CTA (x, y): points of CTA y of item x's table (a grid's y ends at 65535).
__global__ void __launch_bounds__(kThreshThreads) k_thresholds_multi(const ThreshArgs* __restrict__ args) {
  __shared__ ThreshArgs A;
  if (threadIdx.x == 0) A = args[blockIdx.x];
  __syncthreads();
  if ((int)blockIdx.y * kThreshPoints < A.M) thresholds_body(A, (int)blockIdx.y);
}

// ---------------------------------------------------------------------------
template <bool GATHER, bool WANT_F, bool LIN, bool DIRECT>
__device__ __forceinline__ void scan_assign_body(const ScanArgs& a) {
  constexpr int NT = kScanThreads, IT = kScanItems, TILE = kScanTile;
  __shared__ uint32_t sord[TILE + TILE / 32];
  __shared__ float smass[TILE + TILE / 32];
  __shared__ uint32_t s_tile;
  __shared__ ScanShared S;
  const int tid = threadIdx.x;
  if (tid == 0) s_tile = atomicAdd(a.ticket, 1u);
  scan_clear<NT>(S, a.nbuckets);
  __syncthreads();
  const uint32_t tile = s_tile;
  // n <= 2^30: positions fit 32 bits
  const uint32_t start = tile * (uint32_t)TILE;
  const uint32_t n = (uint32_t)a.n;
  const int cnt = (int)(n - start < (uint32_t)TILE ? n - start : (uint32_t)TILE);
  const bool fell = a.fell && *a.fell;
  const bool side_b = a.pick && fell == (a.fell != nullptr) && ((*a.pick - 1) & 1);
  const uint32_t* order = side_b ? a.order_b : fell ? a.order_a : a.order;
  const float* mass = side_b ? a.mass_b : fell ? a.mass_a : a.mass;
  if (tid == 0 && a.ahead) {
    // order and masses of the tile a.ahead tickets later into L2
    const uint32_t fs = (tile + a.ahead) * (uint32_t)TILE;
    if (fs < n) {
      const uint32_t fb = n - fs < (uint32_t)TILE ? n - fs : (uint32_t)TILE;
      prefetch_l2_bulk(order + fs, fb * 4u);
      if constexpr (!GATHER) prefetch_l2_bulk(mass + fs, fb * 4u);
    }
  }
  const float qs = __int_as_float((127 + *a.qshift) << 23);  // 2^s, s in [-2, 64]

  // order (and rank-order masses): coalesced striped loads -> padded shared
  // memory -> a blocked run of IT consecutive ranks per thread
#pragma unroll
  for (int k = 0; k < IT; ++k) {
    const int p = k * NT + tid;
    sord[p + (p >> 5)] = p < cnt ? order[start + p] : 0u;
    if constexpr (!GATHER) smass[p + (p >> 5)] = p < cnt ? mass[start + p] : 0.0f;
  }
  __syncthreads();
  uint32_t cell[IT];
  float mv[IT];
  unsigned long long run = 0;
#pragma unroll
  for (int i = 0; i < IT; ++i) {
    const int p = tid * IT + i;
    cell[i] = sord[p + (p >> 5)];
    mv[i] = 0.0f;
    if (p < cnt) mv[i] = GATHER ? mass[cell[i]] : smass[p + (p >> 5)];
    run += mass_fix(mv[i], qs);
  }
  LookBack lb;
  scan_tile<NT, IT, true, false, DIRECT, WANT_F, LIN>(a, S, lb, tile, start, cnt, cell, mv, run, qs, sord, smass, a.bcell,
                                              a.bz);
}

template <bool GATHER, bool WANT_F, bool LIN, bool DIRECT>
__global__ void __launch_bounds__(kScanThreads, AMBER_SCAN_MINB) k_scan_assign(const ScanArgs a) {
  pdl_begin();
  scan_assign_body<GATHER, WANT_F, LIN, DIRECT>(a);
}

// Several matchings at once: CTA b works on item find_item(prefix, M, b) (the
// prefix counts scan tiles), taking its tile from that item's own ticket.
template <bool LIN>
__global__ void __launch_bounds__(kScanThreads, AMBER_SCAN_MINB)
    k_scan_assign_multi(const ScanArgs* __restrict__ args, const uint32_t* __restrict__ prefix, int M) {
  __shared__ ScanArgs sa;
  if (threadIdx.x == 0) sa = args[find_item(prefix, M, blockIdx.x)];
  __syncthreads();
  scan_assign_body<false, false, LIN, false>(sa);
}

// z_re[cell] = z, bucket after bucket: CTA (bucket b, tile group g) copies
// bucket b's run of every tile in its group, a tile per warp.  A warp takes
// its run in rounds of four 32-pair chunks: all the round's loads (lanes read
// a run coalesced), then its stores, so the dependent load -> store chains
// overlap.  A
// bucket's cells span a bounded region of z_re, so the permuted writes of
// the CTAs working on it stay close together.
__device__ __forceinline__ void scatter_back_body(const ScatterArgs& x, uint32_t blk) {
  const uint32_t* __restrict__ bcell = x.bcell;
  const float* __restrict__ bz = x.bz;
  const uint16_t* __restrict__ btab = x.btab;
  float* __restrict__ zre = x.zre;
  const int nbuckets = x.nbuckets, groups = x.groups;
  const int64_t tiles = x.tiles;
  const int b = blk / groups;
  const int64_t g = blk - (int64_t)b * groups;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const unsigned long long stream_pol = l2_evict_first(), keep_pol = l2_evict_last();
  const int64_t t = g * kBackTilesPerCta + warp;
  if (t >= tiles) return;
  const uint16_t* row = btab + t * (nbuckets + 1);
  const int start = row[b], end = row[b + 1];
  const int64_t base = t * kScanTile;
  constexpr int G = 4;  // 32-pair chunks per round
#pragma unroll 1
  for (int j0 = start; j0 < end; j0 += 32 * G) {
    uint32_t c[G];
    float zz[G];
#pragma unroll
    for (int q = 0; q < G; ++q) {
      const int i = j0 + 32 * q + lane;
      c[q] = 0xffffffffu;
      if (i < end) {
        c[q] = ld_hint(bcell + base + i, stream_pol);
        zz[q] = ld_hint(bz + base + i, stream_pol);
      }
    }
#pragma unroll
    for (int q = 0; q < G; ++q)
      if (c[q] != 0xffffffffu) st_hint(zre + c[q], zz[q], keep_pol);
  }
}

__global__ void __launch_bounds__(256) k_scatter_back(const ScatterArgs x) {
  pdl_begin();
  scatter_back_body(x, blockIdx.x);
}

// Several scatters at once: CTA b works on item find_item(prefix, M, b).
__global__ void __launch_bounds__(256) k_scatter_back_multi(const ScatterArgs* __restrict__ args,
                                                            const uint32_t* __restrict__ prefix, int M) {
  const int it = find_item(prefix, M, blockIdx.x);
  scatter_back_body(args[it], blockIdx.x - prefix[it]);
}

// ---------------------------------------------------------------------------
// Tomographic matching helpers: z_re starts as NaN (neutral); before interval
// k's ranking the cells already ionized get intensity +inf so they rank first;
// after its matching a neutral cell takes the interval's redshift when it
// lies at or above the interval's lower bound (always in the last interval).
__global__ void __launch_bounds__(256) k_tomo_fill(float* __restrict__ z, int64_t n) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    z[i] = __int_as_float(0x7fc00000);  // quiet NaN
}

// Cells ionized in an earlier interval take the next float above the largest
// intensity of this interval (its key is one below the minimum key): they
// rank first, in cell order, exactly as +inf would, while the key range -- and
// so the number of digit passes -- grows by one key instead of to the top of
// the float range.
__global__ void __launch_bounds__(256) k_tomo_mask(float* __restrict__ J, const float* __restrict__ z, int64_t n,
                                                   const SortCtrl* __restrict__ ctrl) {
  const uint32_t k = (uint32_t)ctrl->kmin - 1u;  // kmin > 0 for finite intensities
  const uint32_t u = ~k;                          // undo the descending flip
  const float first = __uint_as_float((u & 0x80000000u) ? (u & 0x7fffffffu) : ~u);
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    if (!isnan(z[i])) J[i] = first;
}

__global__ void k_tomo_widen(SortCtrl* ctrl) {
  if (ctrl->kmin > 0) ctrl->kmin -= 1;
}

__global__ void __launch_bounds__(256) k_tomo_merge(float* __restrict__ z, const float* __restrict__ ztmp, int64_t n,
                                                    float z_low, bool last) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    if (isnan(z[i]) && (last || ztmp[i] >= z_low)) z[i] = ztmp[i];
}

static int elem_grid(int64_t n, int num_sms) {
  return (int)std::max<int64_t>(1, std::min<int64_t>((n + 255) / 256, (int64_t)num_sms * 16));
}

cudaError_t tomo_fill(float* z, int64_t n, int num_sms, cudaStream_t s) {
  k_tomo_fill<<<elem_grid(n, num_sms), 256, 0, s>>>(z, n);
  return cudaGetLastError();
}
cudaError_t tomo_mask(float* J, const float* z, int64_t n, SortCtrl* ctrl, int num_sms, cudaStream_t s) {
  k_tomo_mask<<<elem_grid(n, num_sms), 256, 0, s>>>(J, z, n, ctrl);
  k_tomo_widen<<<1, 1, 0, s>>>(ctrl);
  return cudaGetLastError();
}
cudaError_t tomo_merge(float* z, const float* ztmp, int64_t n, float z_low, bool last, int num_sms, cudaStream_t s) {
  k_tomo_merge<<<elem_grid(n, num_sms), 256, 0, s>>>(z, ztmp, n, z_low, last);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Buckets of consecutive cells: 33 to 64 of them, or (above 2^29 cells) up to
// 128 of 2^23 cells, 32 MB of z_re, so that the bucket being written stays in
// L2.  A tile's 8192 cells take their places by shared-memory adds on their
// buckets' counters, so few buckets collide, and a smaller bucket's sectors
// fill up sooner: with 2^23 cells per bucket at every size (16 buckets at
// 512^3, equal buckets of a warp found by a match first) the scan took 0.95 ms
// and the scatter 0.98 ms at 512^3, with 64 buckets 0.77 and 0.73.  128 buckets,
// with runs of 64 pairs for the scatter, are 2 % slower there; 30 and 60 million
// cells and 24 grids of 64^3 show the same optimum, and 1024^3 differs by 1.5 %
// between 64 and 256 buckets.
void bucket_plan(int64_t n, int* nbuckets, int* shift) {
  int bits = 0;
  while (((int64_t)1 << bits) < n) ++bits;
  *shift = std::min(std::max(bits - 6, 0), 23);
  *nbuckets = (int)((n + ((int64_t)1 << *shift) - 1) >> *shift);
}

void thresholds_launch(ThreshArgs ta, cudaStream_t s) {
  if (ta.ntiles > kTileTotalMin) {
    k_tile_total<<<(unsigned)std::min<int64_t>(64, (ta.ntiles + 1023) / 1024), 256, 0, s>>>(ta.tile_mass, ta.ntiles,
                                                                                         ta.total);
    ta.tile_mass = nullptr;
  }
  launch_pdl(k_thresholds, (ta.M + kThreshPoints - 1) / kThreshPoints, kThreshThreads, 0, s, ta);
}

void assign_args(const AssignWork& w, const uint32_t* order, const float* mass, const unsigned long long* tile_mass,
                 int64_t n, const HistoryCoeffs& hc, float* zre, double* F, unsigned int* status,
                 unsigned int spin_limit, const uint32_t* order_b, const float* mass_b, const int* pick,
                 ThreshArgs* ta, ScanArgs* sa, ScatterArgs* xa) {
  const int64_t tiles = (n + kScanTile - 1) / kScanTile;
  unsigned long long* total = reinterpret_cast<unsigned long long*>(w.ctrl);
  uint32_t* ticket = reinterpret_cast<uint32_t*>(w.ctrl + 16);
  int* qshift = reinterpret_cast<int*>(w.ctrl + 32);
  unsigned long long* qtotal = reinterpret_cast<unsigned long long*>(w.ctrl + 40);
  ThreshArgs& t = *ta;
  t.total = total;
  t.tile_mass = tile_mass;
  t.ntiles = tile_mass ? sort_tiles(n) : 0;
  t.M = hc.n_table;
  t.a_w = hc.a;
  t.b_w = hc.b;
  t.c_w = hc.c;
  t.z_lo = hc.z_lo;
  t.z_hi = hc.z_hi;
  t.Xq = w.Xq;
  t.inv_dx = w.inv_dx;
  t.qshift = qshift;
  t.qtotal = qtotal;
  t.weighting = hc.weighting;
  t.omega_m = hc.omega_m;
  t.z_mid = hc.z_mid;
  t.ncells = n;
  t.lin = w.lin;

  ScanArgs& a = *sa;
  a.order = order;
  a.mass = mass;
  a.order_b = order_b;
  a.mass_b = mass_b;
  a.pick = pick;
  a.fell = nullptr;
  a.order_a = nullptr;
  a.mass_a = nullptr;
  a.n = n;
  a.Xq = w.Xq;
  a.qshift = qshift;
  a.qtotal = qtotal;
  a.inv_dx = w.inv_dx;
  a.n_table = hc.n_table;
  a.weighting = hc.weighting;
  a.z_lo = (float)hc.z_lo;
  a.z_hi = (float)hc.z_hi;
  a.dzt = (float)((hc.z_hi - hc.z_lo) / (double)(hc.n_table - 1));
  a.F = F;
  a.state = w.state;
  a.ticket = ticket;
  bucket_plan(n, &a.nbuckets, &a.bucket_shift);
  a.zre = nullptr;
  a.bcell = w.bcell;
  a.bz = w.bz;
  a.btab = w.btab;
  a.status = status;
  a.spin_limit = spin_limit;
  a.ahead = (uint32_t)w.num_sms;  // half the resident wave (2 CTAs per SM): measured best
  a.linP = w.lin;
  a.linQ = w.lin + kMaxTable;
  a.lina = w.lin + 2 * kMaxTable;
  a.linb = w.lin + 3 * kMaxTable;

  ScatterArgs& x = *xa;
  x.bcell = w.bcell;
  x.bz = w.bz;
  x.btab = w.btab;
  x.nbuckets = a.nbuckets;
  x.tiles = tiles;
  x.groups = (int)((tiles + kBackTilesPerCta - 1) / kBackTilesPerCta);
  x.zre = zre;
}

template <typename A, typename B> static bool disjoint(const A* a, int64_t na, const B* b, int64_t nb) {
  return !b || reinterpret_cast<uintptr_t>(a + na) <= reinterpret_cast<uintptr_t>(b) ||
         reinterpret_cast<uintptr_t>(b + nb) <= reinterpret_cast<uintptr_t>(a);
}

cudaError_t assign_impl(const AssignWork& w, const uint32_t* order, const float* mass, bool mass_in_rank_order,
                        const unsigned long long* tile_mass, int64_t n, const HistoryCoeffs& hc, float* zre, double* F,
                        unsigned int* status, cudaStream_t s, FftProfile* prof, unsigned int spin_limit,
                        const uint32_t* order_b, const float* mass_b, const int* pick, int64_t nsums,
                        const FellArgs* fell) {
  const int64_t tiles = (n + kScanTile - 1) / kScanTile;
  ThreshArgs ta;
  ScanArgs a;
  ScatterArgs xa;
  assign_args(w, order, mass, tile_mass, n, hc, zre, F, status, spin_limit, order_b, mass_b, pick, &ta, &a, &xa);
  if (tile_mass && nsums >= 0) ta.ntiles = nsums;
  if (fell) {
    a.fell = fell->fell;
    a.order_a = fell->order_a;
    a.mass_a = fell->mass_a;
  }
  cudaError_t e = cudaMemsetAsync(w.ctrl, 0, kAssignCtrlBytes, s);
  if (e != cudaSuccess) return e;
  e = cudaMemsetAsync(w.state, 0, (size_t)tiles * sizeof(unsigned long long), s);
  if (e != cudaSuccess) return e;

  if (!tile_mass) {  // masses in cell order: one exact reduction pass
    prof_begin(prof, PK_MASS_REDUCE, s);
    int grid = (int)std::min<int64_t>((n / 4 + 255) / 256, (int64_t)w.num_sms * 8);
    if (grid < 1) grid = 1;
    k_mass_reduce<<<grid, 256, 0, s>>>(mass, n, ta.total, status);
    prof_end(prof, PK_MASS_REDUCE, s);
  }

  prof_begin(prof, PK_THRESHOLDS, s);
  thresholds_launch(ta, s);
  prof_end(prof, PK_THRESHOLDS, s);

  prof_begin(prof, PK_SCAN_ASSIGN, s);
  const unsigned g = (unsigned)tiles;
  const bool gather = !mass_in_rank_order, lin = hc.weighting != AMBER_WEIGHT_MASS;
  // Up to 2^24 cells the field (64 MB) stays in L2 while it is written, so the
  // scan stores each redshift in its place (ranked matching: 256^3 301 -> 216
  // us, 128^3 72 -> 56, 32^3 64 -> 52); above that the stores would reach HBM
  // one sector per cell, so the pairs go through the buckets.  With the masses
  // gathered as well the two kinds of scattered access share the pipe: ranking
  // and matching 1.0e6 cells 154 -> 145 us, 3.0e6 274 -> 272, 1.0e7 610 -> 618.
  // (Also when the result may overwrite what the scan reads.)
  const bool direct = n <= (gather ? kDirectGatherMaxCells : kDirectMaxCells) && disjoint(zre, n, order, n) && disjoint(zre, n, mass, n) &&
                      disjoint(zre, n, order_b, n) && disjoint(zre, n, mass_b, n) && disjoint(zre, n, a.order_a, n) && disjoint(zre, n, a.mass_a, n) &&
                      disjoint(zre, n, F, n);
  if (direct) a.zre = zre;
  auto launch = [&](auto gt, auto ft, auto lt, auto dt) {
    launch_pdl(k_scan_assign<decltype(gt)::value, decltype(ft)::value, decltype(lt)::value, decltype(dt)::value>, g,
               kScanThreads, 0, s, a);
  };
  auto pick4 = [&](auto gt, auto ft, auto lt) {
    if (direct) launch(gt, ft, lt, std::true_type{});
    else launch(gt, ft, lt, std::false_type{});
  };
  auto pick3 = [&](auto gt, auto ft) {
    if (lin) pick4(gt, ft, std::true_type{});
    else pick4(gt, ft, std::false_type{});
  };
  auto pick2 = [&](auto gt) {
    if (F) pick3(gt, std::true_type{});
    else pick3(gt, std::false_type{});
  };
  if (gather) pick2(std::true_type{});
  else pick2(std::false_type{});
  prof_end(prof, PK_SCAN_ASSIGN, s);
  if (direct) return cudaGetLastError();
  prof_begin(prof, PK_SCATTER_BACK, s);
  launch_pdl(k_scatter_back, (unsigned)(xa.groups * xa.nbuckets), 256, 0, s, xa);
  prof_end(prof, PK_SCATTER_BACK, s);
  return cudaGetLastError();
}

cudaError_t assign_multi(const AssignMulti& m, cudaStream_t s) {
  k_thresholds_multi<<<dim3((unsigned)m.M, (unsigned)((m.max_table + kThreshPoints - 1) / kThreshPoints)),
                       kThreshThreads, 0, s>>>(m.thresh);
  if (m.scan_tiles[0]) k_scan_assign_multi<false><<<m.scan_tiles[0], kScanThreads, 0, s>>>(m.scan[0], m.scan_prefix[0], m.Mg[0]);
  if (m.scan_tiles[1]) k_scan_assign_multi<true><<<m.scan_tiles[1], kScanThreads, 0, s>>>(m.scan[1], m.scan_prefix[1], m.Mg[1]);
  if (m.scatter_blocks) k_scatter_back_multi<<<m.scatter_blocks, 256, 0, s>>>(m.scatter, m.scatter_prefix, m.Ms);
  return cudaGetLastError();
}

}  // namespace amber
