// Source-field pipeline on the GPU (Sec. 3.2, Eq. xlpt; Sec. 3.2.1, Eqs.
// interlace and Wofk; Sec. 3.3, Eq. fcoll).
//
//   k_assign<P>   : NGP / CIC / TSC assignment of one particle per lattice
//                   point (FP32 atomics on the mesh)
//   k_scale_mesh  : plain assignment's normalisation
//
// The operators on spectra (second derivatives, inverse gradients, filters,
// the interlaced combination) and the products of their results are fused into
// the transform passes (fft_ops.cuh).
#include <cmath>

#include <algorithm>

#include "fft_ops.cuh"
#include "lpt.cuh"

namespace amber {

__device__ __forceinline__ int wrap(int v, int n) {
  v %= n;
  return v < 0 ? v + n : v;
}

// One particle per thread: lattice point (ix, iy, iz) displaced by psi
// (box units, inv_dx cells per unit) plus `shift` cells on every axis; the
// nearest mesh point is floor(pos + 1/2), d = pos - that point in [-1/2, 1/2).
template <int P>
__global__ void __launch_bounds__(256) k_assign(const float* __restrict__ px, const float* __restrict__ py,
                                                const float* __restrict__ pz, const float* __restrict__ mass, int n,
                                                float inv_dx, float shift, float* __restrict__ mesh) {
  const int64_t np = (int64_t)n * n * n;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < np; i += (int64_t)gridDim.x * blockDim.x) {
    const int ix = (int)(i % n), iy = (int)((i / n) % n), iz = (int)(i / ((int64_t)n * n));
    const float pos[3] = {ix + px[i] * inv_dx + shift, iy + py[i] * inv_dx + shift, iz + pz[i] * inv_dx + shift};
    int base[3];
    float w[3][3];  // offsets -1, 0, +1
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const float b = floorf(pos[a] + 0.5f);
      const float d = pos[a] - b;
      base[a] = (int)b;
      if (P == 1) {
        w[a][0] = 0.f; w[a][1] = 1.f; w[a][2] = 0.f;
      } else if (P == 2) {
        const float ad = fabsf(d);
        w[a][1] = 1.f - ad;
        w[a][0] = d < 0.f ? ad : 0.f;
        w[a][2] = d >= 0.f ? ad : 0.f;
      } else {
        w[a][0] = 0.5f * (0.5f - d) * (0.5f - d);
        w[a][1] = 0.75f - d * d;
        w[a][2] = 0.5f * (0.5f + d) * (0.5f + d);
      }
    }
    const float m = mass ? mass[i] : 1.0f;
#pragma unroll
    for (int oz = 0; oz < 3; ++oz) {
      if (w[2][oz] == 0.f) continue;
      const int64_t zo = (int64_t)wrap(base[2] + oz - 1, n) * n * n;
#pragma unroll
      for (int oy = 0; oy < 3; ++oy) {
        if (w[1][oy] == 0.f) continue;
        const int64_t yo = zo + (int64_t)wrap(base[1] + oy - 1, n) * n;
        const float wzy = m * w[2][oz] * w[1][oy];
#pragma unroll
        for (int ox = 0; ox < 3; ++ox) {
          if (w[0][ox] == 0.f) continue;
          atomicAdd(&mesh[yo + wrap(base[0] + ox - 1, n)], wzy * w[0][ox]);
        }
      }
    }
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

static cudaError_t assign(int order, int n, double box, float shift, const float* px, const float* py,
                          const float* pz, const float* mass, float* mesh, int num_sms, cudaStream_t s) {
  const int64_t n3 = (int64_t)n * n * n;
  cudaError_t e = cudaMemsetAsync(mesh, 0, (size_t)n3 * sizeof(float), s);
  if (e != cudaSuccess) return e;
  const float inv_dx = (float)(n / box);
  const int g = grid_of(n3, num_sms);
  if (order == 1) k_assign<1><<<g, 256, 0, s>>>(px, py, pz, mass, n, inv_dx, shift, mesh);
  else if (order == 2) k_assign<2><<<g, 256, 0, s>>>(px, py, pz, mass, n, inv_dx, shift, mesh);
  else k_assign<3><<<g, 256, 0, s>>>(px, py, pz, mass, n, inv_dx, shift, mesh);
  return cudaGetLastError();
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
  if (e == cudaSuccess) e = assign(order, n, box, 0.f, psi_x, psi_y, psi_z, mass, rho, w.num_sms, s);
  if (e != cudaSuccess) return e;
  if (!interlace) {
    k_scale_mesh<<<grid_of(n3, w.num_sms), 256, 0, s>>>(rho, n3, w.acc);
    return cudaGetLastError();
  }
  e = assign(order, n, box, 0.5f, psi_x, psi_y, psi_z, mass, w.F0, w.num_sms, s);
  if (e == cudaSuccess) e = forward_spectrum_f32(n, rho, w.H0, w.tw, s);
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
