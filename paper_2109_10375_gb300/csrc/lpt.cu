// Source-field pipeline on the GPU (Sec. 3.2, Eq. xlpt; Sec. 3.2.1, Eqs.
// interlace and Wofk; Sec. 3.3, Eq. fcoll).
//
//   k_assign      : NGP / CIC / TSC assignment of one particle per lattice
//                   point (FP32 sums, in any order)
//   k_scale_mesh  : plain assignment's normalisation
//
// The operators on spectra (second derivatives, inverse gradients, filters,
// the interlaced combination) and the products of their results are fused into
// the transform passes (fft_ops.cuh).
#include <cmath>

#include <algorithm>
#include <type_traits>

#include "fft_ops.cuh"
#include "lpt.cuh"

namespace amber {

// Window of order P of a particle at pos (cells) on one axis: the first mesh
// point it reaches and its P weights.  The nearest mesh point is
// floor(pos + 1/2), d = pos - that point in [-1/2, 1/2).
template <int P> __device__ __forceinline__ int window(float pos, float w[P]) {
  const float b = floorf(pos + 0.5f);
  const float d = pos - b;
  if constexpr (P == 1) {
    w[0] = 1.f;
    return (int)b;
  } else if constexpr (P == 2) {
    const float ad = fabsf(d);
    w[0] = d < 0.f ? ad : 1.f - ad;
    w[1] = d < 0.f ? 1.f - ad : ad;
    return d < 0.f ? (int)b - 1 : (int)b;
  } else {
    w[0] = 0.5f * (0.5f - d) * (0.5f - d);
    w[1] = 0.75f - d * d;
    w[2] = 0.5f * (0.5f + d) * (0.5f + d);
    return (int)b - 1;
  }
}

// Straight to the mesh: one global atomic per mesh point the particle reaches
// (n is a power of two, so a coordinate wraps by its low bits).  Points of weight
// 0 are not reached: a mass that is not finite stays where its window is.
template <int P>
__device__ __forceinline__ void deposit_global(float* __restrict__ mesh, const float pos[3], float m, int n) {
  float w[3][P];
  int b[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) b[a] = window<P>(pos[a], w[a]);
  const unsigned mask = (unsigned)n - 1u;
#pragma unroll
  for (int oz = 0; oz < P; ++oz) {
    if (w[2][oz] == 0.f) continue;
    const int64_t zo = (int64_t)(((unsigned)b[2] + oz) & mask) * n;
#pragma unroll
    for (int oy = 0; oy < P; ++oy) {
      if (w[1][oy] == 0.f) continue;
      float* row = mesh + (zo + (((unsigned)b[1] + oy) & mask)) * n;
      const float wzy = m * w[2][oz] * w[1][oy];
#pragma unroll
      for (int ox = 0; ox < P; ++ox)
        if (w[0][ox] != 0.f) atomicAdd(&row[((unsigned)b[0] + ox) & mask], wzy * w[0][ox]);
    }
  }
}

// Grids below one block, and plain nearest-point meshes, whose one mesh point per
// particle leaves nothing to gather (512^3 0.85 ms, by blocks 1.43): one particle
// per thread; lattice point (ix, iy, iz) displaced by psi (box units, inv_dx
// cells per unit) plus `shift` cells on every axis.
template <int P>
__global__ void __launch_bounds__(256) k_assign_direct(const float* __restrict__ px, const float* __restrict__ py,
                                                      const float* __restrict__ pz, const float* __restrict__ mass,
                                                      int n, int lg, float inv_dx, float shift,
                                                      float* __restrict__ mesh) {
  const int np = n * n * n;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < np; i += gridDim.x * blockDim.x) {
    const int ix = i & (n - 1), iy = (i >> lg) & (n - 1), iz = i >> (2 * lg);
    const float pos[3] = {ix + px[i] * inv_dx + shift, iy + py[i] * inv_dx + shift, iz + pz[i] * inv_dx + shift};
    deposit_global<P>(mesh, pos, mass ? mass[i] : 1.0f, n);
  }
}

// A CTA takes a block of 32 x 8 x 8 lattice points (lanes along x, 8 y and two
// halves of z over the warps, four z per thread).  Neighbouring particles stay
// neighbours, so the mesh points the block reaches fit a box of 2-4 points per
// particle: its sums are formed there, in shared memory, and each box point
// goes to the mesh with one coalesced global atomic.  Global atomics for every
// window point, 27 per particle for TSC, were bound by the packets they send to
// L2 (two 512^3 TSC meshes 9.84 ms); float atomics in shared memory are a
// compare-and-swap loop here (9.7 wavefronts per warp, 9.28 ms).  Integer ones
// take 2, so the box holds 32-bit fixed-point words, two per point or one.  With
// two, S the scale of the first and 2^-k the unit of the second, a contribution
// c adds round(c S) to the first and the rest, at most 1/2, to the second.
//
// An interlaced density (PLAIN false: both meshes, the second's particles half
// a cell on, from one read of psi) goes through transforms that mix all mesh
// points, so what counts is an error against the field's own scale.  S brings
// the block's mass total M below 2^30 (no sum can overflow), k is 20 (2048 rests
// of at most 1/2 fit): a resolution between 2^-49 and 2^-48 of M.  Particles of
// equal mass take one word where no mesh point is the nearest of more than 8 of
// them (counted first): a point's window weights then sum to less than 8 (CIC;
// 5.4 for TSC) times that count, so that a resolution of 2^-25 or finer fits,
// under float's rounding of a mean density of 1.  Two 512^3 TSC meshes take 4.00
// ms (5.40 with two words), bound by the shared-memory pipe (69 % busy; 83 %).
//
// A plain mesh (PLAIN) is itself the result, and its points differ by many
// orders: in a void a point may hold only the far tail of one window.  It always
// takes two words, as fine as they go: with c the most particles that any mesh
// point is the nearest of (2^lc >= c) and 2^e above every mass, S = 2^(27 - lc -
// e), and k = 23 up to c = 16 (27 c rests fit), 20 above: a resolution of 2^-48
// of a particle for c <= 4.  It has to lie 40 bits below the lightest mass, which
// leaves the masses of a block 8 bits to differ by (c <= 4): collapsed fractions,
// which span many orders, go straight to the mesh.  Against 64-bit sums the
// errors are then those of float atomics or less at every density (256^3 CIC of
// particles 2 cells off their places, FP32-exact positions: 3e-8 rms at density 1
// against 4e-8, both exact below 0.1; with one word of 2^-25 2e-6 at 1e-2, 1e-4
// at 1e-4).  512^3 TSC 2.61 -> 3.31 ms (float atomics 5.27).
//
// A block whose box does not fit, or whose masses are all 0, not finite or out
// of the scale's range, or that has a position that is not finite, deposits
// straight to the mesh.
constexpr int kAsgX = 32, kAsgY = 8, kAsgZ = 8, kAsgPer = 4;
constexpr int kAsgThreads = kAsgX * kAsgY * kAsgZ / kAsgPer;
constexpr int kAsgBox = 14000;  // mesh points a block's box may hold (two CTAs per SM)

__device__ __forceinline__ float pow2f(int e) { return __int_as_float((127 + e) << 23); }  // |e| <= 126

template <int P, bool PLAIN>
__global__ void __launch_bounds__(kAsgThreads, 2)
    k_assign(const float* __restrict__ px, const float* __restrict__ py, const float* __restrict__ pz,
             const float* __restrict__ mass, int n, float inv_dx, float* __restrict__ mesh0,
             float* __restrict__ mesh1) {
  constexpr int NW = kAsgThreads / 32;
  extern __shared__ __align__(16) int box_hi[];  // [kAsgBox], then the second words
  int* box_lo = box_hi + kAsgBox;
  __shared__ int s_lo[3][NW], s_hi[3][NW], s_most[NW];
  __shared__ float s_mass[NW];
  __shared__ unsigned s_heavy[NW], s_light[NW];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int nx = n / kAsgX, ny = n / kAsgY;
  const int bx = blockIdx.x % nx, by = (blockIdx.x / nx) % ny, bz = blockIdx.x / (nx * ny);
  const int ix = bx * kAsgX + lane, iy = by * kAsgY + (warp & 7), iz0 = bz * kAsgZ + (warp >> 3) * kAsgPer;
  float pos[kAsgPer][3], m[kAsgPer];
#pragma unroll
  for (int q = 0; q < kAsgPer; ++q) {
    const int64_t i = ((int64_t)(iz0 + q) * n + iy) * n + ix;
    pos[q][0] = px[i];
    pos[q][1] = py[i];
    pos[q][2] = pz[i];
    m[q] = mass ? mass[i] : 1.0f;
  }
  float msum = 0.f;
  unsigned heavy = 0, light = 0xffffffffu;  // bits of the largest and the smallest |m| > 0
#pragma unroll
  for (int q = 0; q < kAsgPer; ++q) {
    pos[q][0] = ix + pos[q][0] * inv_dx;
    pos[q][1] = iy + pos[q][1] * inv_dx;
    pos[q][2] = iz0 + q + pos[q][2] * inv_dx;
    // a position that is not finite makes the sum NaN (straight to the mesh)
    msum += fabsf(m[q]) + 0.f * (pos[q][0] + pos[q][1] + pos[q][2]);
    if (PLAIN) {
      const unsigned u = __float_as_uint(fabsf(m[q]));
      heavy = max(heavy, u);
      light = min(light, u - 1u);  // (0 becomes the largest)
    }
  }
#pragma unroll
  for (int o = 16; o >= 1; o >>= 1) msum += __shfl_xor_sync(0xffffffffu, msum, o);
  if (PLAIN) {
    heavy = __reduce_max_sync(0xffffffffu, heavy);
    light = __reduce_min_sync(0xffffffffu, light);
  }
  if (lane == 0) {
    s_mass[warp] = msum;
    if (PLAIN) {
      s_heavy[warp] = heavy;
      s_light[warp] = light;
    }
  }
  float scale = 0.f, unscale = 0.f;
  for (int pass = 0; pass < (PLAIN ? 1 : 2); ++pass) {
    float* __restrict__ mesh = pass ? mesh1 : mesh0;
    const float shift = pass ? 0.5f : 0.f;
    // the box of mesh points the block's windows reach
    int ext[3], org[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      int lo = 0x7fffffff, hi = -0x7fffffff;
#pragma unroll
      for (int q = 0; q < kAsgPer; ++q) {
        float w[P];
        const int b = window<P>(pos[q][a] + shift, w);
        lo = min(lo, b);
        hi = max(hi, b);
      }
      lo = __reduce_min_sync(0xffffffffu, lo);
      hi = __reduce_max_sync(0xffffffffu, hi);
      if (lane == 0) {
        s_lo[a][warp] = lo;
        s_hi[a][warp] = hi;
      }
    }
    __syncthreads();
    int mexp = 0;      // PLAIN: every |m| is below 2^mexp
    float lightest = 0.f;
    if (pass == 0) {
      float t = s_mass[lane % NW];  // NW = 16: every sum twice
#pragma unroll
      for (int o = NW / 2; o >= 1; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
      // t < 2^(e - 126) (one more bit for the rounding of this sum)
      const int e = (__float_as_int(t) >> 23) + 1;
      if (PLAIN) {
        mexp = (int)(__reduce_max_sync(0xffffffffu, s_heavy[lane % NW]) >> 23) - 126;
        lightest = __uint_as_float(__reduce_min_sync(0xffffffffu, s_light[lane % NW]) + 1u);
        // (a first guess, for one particle per point; replaced when they are counted)
        if (t > 0.f && e < 250 && mexp > -80 && mexp < 100 && lightest >= pow2f(40 - 23 - 27 + mexp)) scale = 1.f;
      } else if (t > 0.f && e > 40 && e < 250 && 30 - (e - 126) < 120) {
        scale = pow2f(30 - (e - 126));
        unscale = pow2f(e - 126 - 30);
      }
    }
    bool fits = scale != 0.f;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      org[a] = __reduce_min_sync(0xffffffffu, s_lo[a][lane % NW]);
      const int hi = __reduce_max_sync(0xffffffffu, s_hi[a][lane % NW]);
      // (float: the spread of far-flung particles can exceed an int)
      fits = fits && (float)hi - (float)org[a] < 256.f;
      ext[a] = fits ? hi - org[a] + P : 0;
    }
    const int plane = ext[0] * ext[1], cells = plane * ext[2];
    fits = fits && cells <= kAsgBox;  // the same on every thread
    float one = 0.f;  // the scale of a single word, or 0: two words
    int k = 20;
    if (fits) {
      for (int c = tid * 4; c < cells; c += kAsgThreads * 4) {
        *reinterpret_cast<int4*>(box_hi + c) = make_int4(0, 0, 0, 0);
        *reinterpret_cast<int4*>(box_lo + c) = make_int4(0, 0, 0, 0);
      }
      __syncthreads();
      if (PLAIN || !mass) {
#pragma unroll
        for (int q = 0; q < kAsgPer; ++q) {
          int b[3];
#pragma unroll
          for (int a = 0; a < 3; ++a) b[a] = (int)floorf(pos[q][a] + shift + 0.5f) - org[a];
          atomicAdd(box_lo + b[2] * plane + b[1] * ext[0] + b[0], 1);
        }
        __syncthreads();
        int most = 0;
        for (int c = tid * 4; c < cells; c += kAsgThreads * 4) {
          int4* at = reinterpret_cast<int4*>(box_lo + c);
          const int4 v = *at;
          most = max(most, max(max(v.x, v.y), max(v.z, v.w)));
          *at = make_int4(0, 0, 0, 0);
        }
        if (PLAIN) {
          most = __reduce_max_sync(0xffffffffu, most);
          if (lane == 0) s_most[warp] = most;
          __syncthreads();
          most = __reduce_max_sync(0xffffffffu, s_most[lane % NW]);
          const int lc = 32 - __clz(most - 1);  // 2^lc >= most
          if (lc <= 4) k = 23;
          // unit of the second word: 2^(lc + mexp - 27 - k)
          fits = lightest >= pow2f(40 + lc + mexp - 27 - k);
          scale = pow2f(27 - lc - mexp);
          unscale = pow2f(lc + mexp - 27);
        } else if (!__syncthreads_or(most > (P == 2 ? 7 : 8))) {  // (8 x 8 x 2^25 would be 2^31)
          one = __syncthreads_or(most > 4) ? 33554432.f : 67108864.f;  // 2^25, 2^26
        }
      }
    }
    if (!fits) {
#pragma unroll 1
      for (int q = 0; q < kAsgPer; ++q) {
        const float at[3] = {pos[q][0] + shift, pos[q][1] + shift, pos[q][2] + shift};
        deposit_global<P>(mesh, at, m[q], n);
      }
      __syncthreads();  // s_lo, s_hi are read
      continue;
    }
    const float rest = (float)(1 << k);
    auto deposit = [&](auto words) {
#pragma unroll
      for (int q = 0; q < kAsgPer; ++q) {
        float w[3][P];
        int b[3];
#pragma unroll
        for (int a = 0; a < 3; ++a) b[a] = window<P>(pos[q][a] + shift, w[a]) - org[a];
        const float ms = decltype(words)::value == 1 ? one : m[q] * scale;
        int* at = box_hi + b[2] * plane + b[1] * ext[0] + b[0];
#pragma unroll
        for (int oz = 0; oz < P; ++oz) {
#pragma unroll
          for (int oy = 0; oy < P; ++oy) {
            const float wzy = ms * w[2][oz] * w[1][oy];
            int* row = at + oz * plane + oy * ext[0];
#pragma unroll
            for (int ox = 0; ox < P; ++ox) {
              const float c = wzy * w[0][ox];
              const int h = __float2int_rn(c);
              atomicAdd(row + ox, h);
              if (decltype(words)::value == 2)
                atomicAdd(row + ox + kAsgBox, __float2int_rn((c - (float)h) * rest));
            }
          }
        }
      }
    };
    if (!PLAIN && one != 0.f) deposit(std::integral_constant<int, 1>{});
    else deposit(std::integral_constant<int, 2>{});
    __syncthreads();
    const float back = !PLAIN && one != 0.f ? 1.f / one : unscale, unit = 1.f / rest;
    const unsigned mask = (unsigned)n - 1u;
    const unsigned mx = 0xffffffffu / (unsigned)ext[0] + 1u, my = 0xffffffffu / (unsigned)ext[1] + 1u;
    for (int c = tid; c < cells; c += kAsgThreads) {
      const int l = box_lo[c], h = box_hi[c] + (l >> k);
      const float v = ((float)h + (float)(l & ((1 << k) - 1)) * unit) * back;
      if (v != 0.f) {
        // c = (z ext1 + y) ext0 + x; the reciprocals are exact for c < 2^16
        const unsigned yz = ext[0] == 1 ? (unsigned)c : __umulhi((unsigned)c, mx), x = c - yz * ext[0];
        const unsigned z = ext[1] == 1 ? yz : __umulhi(yz, my), y = yz - z * ext[1];
        const unsigned gx = (org[0] + x) & mask, gy = (org[1] + y) & mask, gz = (org[2] + z) & mask;
        atomicAdd(&mesh[((int64_t)gz * n + gy) * n + gx], v);
      }
    }
    __syncthreads();  // the box is read: the next mesh may use it
  }
}

__global__ void __launch_bounds__(256) k_scale_mesh(float* __restrict__ rho, int64_t n3, const double* __restrict__ total) {
  const float f = (float)((double)n3 / *total);
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n3; i += (int64_t)gridDim.x * blockDim.x)
    rho[i] *= f;
}

__global__ void __launch_bounds__(256) k_set_total(double* __restrict__ total, double v) { *total = v; }

// ---------------------------------------------------------------------------
static int grid_of(int64_t work, int num_sms) {
  return (int)std::max<int64_t>(1, std::min<int64_t>((work + 255) / 256, (int64_t)num_sms * 16));
}

cudaError_t lpt_impl(const LptWork& w, int n, double box, double D1, double D2, const float* delta, float* psi_x,
                     float* psi_y, float* psi_z, cudaStream_t s) {
  LinOp op{};
  op.A = reinterpret_cast<const cpx<float>*>(w.H0);
  op.c1 = 1.f;
  op.kf = (float)(2.0 * 3.14159265358979323846 / box);
  op.scale = (float)(1.0 / ((double)n * n * n));
  cudaError_t e = forward_spectrum_f32(n, delta, w.H0, w.tw, s);
  // second derivatives of phi1 (k_a k_b delta / k^2): xx and yy into psi as
  // scratch, their products with zz into F0, less the mixed ones squared
  const int term[6][3] = {{0, 0, LIN_STORE}, {1, 1, LIN_STORE}, {2, 2, LIN_DIAG},
                          {0, 1, LIN_SUB_SQUARE}, {0, 2, LIN_SUB_SQUARE}, {1, 2, LIN_SUB_SQUARE}};
  float* to[6] = {psi_x, psi_y, w.F0, w.F0, w.F0, w.F0};
  for (int q = 0; q < 6 && e == cudaSuccess; ++q) {
    op.a = term[q][0];
    op.b = term[q][1];
    e = inverse_lin_f32(n, op, term[q][2], psi_x, psi_y, w.H2, to[q], w.tw, w.status, s);
  }
  if (e == cudaSuccess) e = forward_spectrum_f32(n, w.F0, w.H1, w.tw, s);
  // psi_a = -D1 grad_a phi1 + D2 grad_a phi2 = (-i k_a / k^2)(-D1 delta + D2 S2)
  op.B = reinterpret_cast<const cpx<float>*>(w.H1);
  op.b = -1;
  op.c1 = (float)(-D1);
  op.c2 = (float)D2;
  float* out[3] = {psi_x, psi_y, psi_z};
  for (int a = 0; a < 3 && e == cudaSuccess; ++a) {
    op.a = a;
    e = inverse_lin_f32(n, op, LIN_STORE, nullptr, nullptr, w.H2, out[a], w.tw, w.status, s);
  }
  return e;
}

template <int P>
static cudaError_t assign_p(int n, float inv_dx, const float* px, const float* py, const float* pz, const float* mass,
                            float* mesh0, float* mesh1, int num_sms, cudaStream_t s) {
  const int64_t n3 = (int64_t)n * n * n;
  if (n >= kAsgX && (P > 1 || mesh1)) {
    constexpr size_t smem = 2 * kAsgBox * sizeof(int);
    static PerDeviceOnce attr;  // per instantiation and device
    once_on_device(attr, [&](DeviceSetUp& u) {
      if constexpr (P > 1) u.smem(k_assign<P, true>, smem);
      u.smem(k_assign<P, false>, smem);
    });
    const unsigned grid = (unsigned)(n3 / (kAsgX * kAsgY * kAsgZ));
    if (mesh1) k_assign<P, false><<<grid, kAsgThreads, smem, s>>>(px, py, pz, mass, n, inv_dx, mesh0, mesh1);
    else if constexpr (P > 1) k_assign<P, true><<<grid, kAsgThreads, smem, s>>>(px, py, pz, mass, n, inv_dx, mesh0, nullptr);
  } else {
    int lg = 0;
    while ((1 << lg) < n) ++lg;
    for (int pass = 0; pass < 2; ++pass)
      if (pass ? mesh1 : mesh0)
        k_assign_direct<P><<<grid_of(n3, num_sms), 256, 0, s>>>(px, py, pz, mass, n, lg, inv_dx, pass ? 0.5f : 0.f,
                                                               pass ? mesh1 : mesh0);
  }
  return cudaGetLastError();
}

// mesh0 (and mesh1, shifted by half a cell, unless null) = sums of the masses
static cudaError_t assign(int order, int n, double box, const float* px, const float* py, const float* pz,
                          const float* mass, float* mesh0, float* mesh1, int num_sms, cudaStream_t s) {
  const size_t bytes = (size_t)n * n * n * sizeof(float);
  cudaError_t e = cudaMemsetAsync(mesh0, 0, bytes, s);
  if (e == cudaSuccess && mesh1) e = cudaMemsetAsync(mesh1, 0, bytes, s);
  if (e != cudaSuccess) return e;
  const float inv_dx = (float)(n / box);
  if (order == 1) return assign_p<1>(n, inv_dx, px, py, pz, mass, mesh0, mesh1, num_sms, s);
  if (order == 2) return assign_p<2>(n, inv_dx, px, py, pz, mass, mesh0, mesh1, num_sms, s);
  return assign_p<3>(n, inv_dx, px, py, pz, mass, mesh0, mesh1, num_sms, s);
}

cudaError_t mesh_impl(const LptWork& w, int n, double box, int order, bool interlace, const float* psi_x,
                      const float* psi_y, const float* psi_z, const float* mass, float* rho, cudaStream_t s) {
  const int64_t n3 = (int64_t)n * n * n;
  cudaError_t e;
  if (mass) {
    e = sum_f64_impl(mass, n3, w.acc, w.num_sms, s);
  } else {
    k_set_total<<<1, 1, 0, s>>>(w.acc, (double)n3);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess)
    e = assign(order, n, box, psi_x, psi_y, psi_z, mass, rho, interlace ? w.F0 : nullptr, w.num_sms, s);
  if (e != cudaSuccess) return e;
  if (!interlace) {
    k_scale_mesh<<<grid_of(n3, w.num_sms), 256, 0, s>>>(rho, n3, w.acc);
    return cudaGetLastError();
  }
  e = forward_spectrum_f32(n, rho, w.H0, w.tw, s);
  if (e == cudaSuccess) e = forward_spectrum_f32(n, w.F0, w.H1, w.tw, s);
  if (e == cudaSuccess) {
    // 1/total: mean 1 and the inverse transform's 1/n^3 together
    const InterlaceOp op{reinterpret_cast<const cpx<float>*>(w.H0), reinterpret_cast<const cpx<float>*>(w.H1), w.acc,
                         order};
    e = inverse_interlace_f32(n, op, w.H2, rho, w.tw, w.status, s);
  }
  return e;
}

cudaError_t fcoll_impl(const LptWork& w, int n, double box, double R, int filter, double delta_c, double dsigma2,
                       const float* delta, float* out, cudaStream_t s) {
  const double kfR = 2.0 * 3.14159265358979323846 / box * R;
  FilterOp op{};
  op.tophat = filter;
  op.m2max = (int)std::min(std::floor(1.0 / (kfR * kfR)), 2e9);  // keep |m|^2 with k R <= 1
  op.kf = (float)(2.0 * 3.14159265358979323846 / box);
  op.R = (float)R;
  return filter_fcoll_f32(n, op, (float)delta_c, (float)(1.0 / std::sqrt(2.0 * dsigma2)), delta, w.H0, out, w.tw,
                          w.status, s);
}

}  // namespace amber
