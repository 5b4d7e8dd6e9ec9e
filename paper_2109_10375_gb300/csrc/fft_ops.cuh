// Spectral operators fused into the inverse transform's passes (source-field
// pipeline, Sec. 3.2, 3.2.1, 3.3): an operator is applied where the z pass
// loads (or, for filters, multiplies) the spectrum, and the elementwise work on
// the result where the x pass writes it, so neither costs a pass over memory.
// As kernels of their own the operators took 3.05 ms of a 512^3 2LPT
// displacement's 11.1 ms and the products of second derivatives 1.25 ms.
#pragma once

#include "fft.cuh"

namespace amber {

// v = c1 A + c2 B (B optional) times k_a k_b / k^2 (b >= 0; a <= b) or
// -i k_a / k^2 (b < 0), times scale; zero at k = 0.  An odd derivative along an
// axis whose wave number is the Nyquist one is 0.
// Table: the real factor for kz = 0..n/2 of the tile's columns (half the
// divisions, and none between the loads); at -kz it is the same, or its
// negative for an odd derivative along z.
struct LinOp {
  static constexpr bool kLoad = true, kFilter = false;
  const cpx<float>* A;
  const cpx<float>* B;
  int a, b;  // axes 0 = x, 1 = y, 2 = z
  float c1, c2;
  float kf;  // 2 pi / box
  float scale;

  template <int N, int SB> static constexpr size_t table_bytes() { return (size_t)(N / 2 + 1) * SB * 4; }
  __device__ __forceinline__ bool odd_z() const { return b < 0 ? a == 2 : b == 2 && a != 2; }
  template <int N, int SB, int NT> __device__ __forceinline__ void fill(void* table, int tid, int kx0, int yi) const {
    float* t = reinterpret_cast<float*>(table);
    const int my = signed_freq(yi, N), oy = yi == N / 2 ? 0 : my;
#pragma unroll 1
    for (int i = tid; i < (N / 2 + 1) * SB; i += NT) {
      const int mz = i / SB, mx = kx0 + (i - mz * SB), ox = mx == N / 2 ? 0 : mx, oz = mz == N / 2 ? 0 : mz;
      const int m2 = mx * mx + my * my + mz * mz;
      int num;
      if (b < 0) num = a == 0 ? ox : a == 1 ? oy : oz;
      else if (a == b) num = a == 0 ? mx * mx : a == 1 ? my * my : mz * mz;
      else num = (a == 0 ? ox : oy) * (b == 1 ? oy : oz);
      const float den = b < 0 ? (float)m2 * kf : (float)m2;
      t[i] = num == 0 ? 0.f : (float)num / den;
    }
  }
  // v[r] = the operator at kz index j + r N/R0 (spectrum offset `at` + index * es)
  template <int N, int SB, int R0>
  __device__ __forceinline__ void load(cpx<float>* v, const void* table, bool ok, int, int col, int, int64_t at,
                                       int64_t es, int j) const {
#pragma unroll
    for (int r = 0; r < R0; ++r) v[r] = ok ? A[at + (int64_t)(j + r * (N / R0)) * es] : mk<float>(0.f, 0.f);
    if (B) {
      constexpr int G = R0 < 8 ? R0 : 8;
#pragma unroll
      for (int r0 = 0; r0 < R0; r0 += G) {
        cpx<float> w[G];
#pragma unroll
        for (int g = 0; g < G; ++g)
          w[g] = ok ? B[at + (int64_t)(j + (r0 + g) * (N / R0)) * es] : mk<float>(0.f, 0.f);
#pragma unroll
        for (int g = 0; g < G; ++g)
          v[r0 + g] = mk<float>(fmaf(c2, w[g].x, c1 * v[r0 + g].x), fmaf(c2, w[g].y, c1 * v[r0 + g].y));
      }
    }
    const float* t = reinterpret_cast<const float*>(table) + col;
    const bool grad = b < 0;
    const float neg = odd_z() ? -scale : scale;
#pragma unroll
    for (int r = 0; r < R0; ++r) {
      const int n = j + r * (N / R0);
      const float f = n <= N / 2 ? t[n * SB] * scale : t[(N - n) * SB] * neg;  // scale: a power of two
      v[r] = grad ? mk<float>(f * v[r].y, -f * v[r].x) : mk<float>(f * v[r].x, f * v[r].y);
    }
  }
};

// [A + e^{i k.dX} B] / 2 / W(k)^p / *total, dX = (dx/2)(1,1,1), W the window's
// transform prod sin(k_a dx/2)/(k_a dx/2); zero where a component is Nyquist.
// Table: e^{i pi s / n} for the sums s = kx + ky + kz of the tile, the axis
// windows of |m| < n/2 and 1/total (one FP64 division per tile).
struct InterlaceOp {
  static constexpr bool kLoad = true, kFilter = false;
  const cpx<float>* A;
  const cpx<float>* B;
  const double* total;
  int p;

  template <int N, int SB> static constexpr size_t table_bytes() {
    return (size_t)(N + SB) * 8 + (size_t)(N / 2) * 4 + 8;
  }
  template <int N, int SB, int NT> __device__ __forceinline__ void fill(void* table, int tid, int kx0, int yi) const {
    cpx<float>* t = reinterpret_cast<cpx<float>*>(table);
    const int s0 = kx0 + signed_freq(yi, N) - N / 2;
#pragma unroll 1
    for (int e = tid; e < N + SB; e += NT) {
      float sn, cs;
      sincospif((float)(s0 + e) / (float)N, &sn, &cs);
      t[e] = mk<float>(cs, sn);
    }
    float* w = reinterpret_cast<float*>(t + N + SB);
#pragma unroll 1
    for (int m = tid; m < N / 2; m += NT) {
      const float x = (float)m / (float)N;  // k dx / 2 in units of pi
      w[m] = m == 0 ? 1.f : sinpif(x) / (3.14159265358979f * x);
    }
    if (tid == 0) w[N / 2] = (float)(1.0 / *total);
  }
  template <int N, int SB, int R0>
  __device__ __forceinline__ void load(cpx<float>* v, const void* table, bool ok, int kx, int col, int yi, int64_t at,
                                       int64_t es, int j) const {
    const cpx<float>* t = reinterpret_cast<const cpx<float>*>(table);
    const float* w = reinterpret_cast<const float*>(t + N + SB);
    const int my = signed_freq(yi, N);
    const bool live = ok && kx < N / 2 && yi != N / 2;
    const float wxy = live ? w[kx] * w[my < 0 ? -my : my] : 1.f, scale = 0.5f * w[N / 2];
#pragma unroll
    for (int r = 0; r < R0; ++r) v[r] = live ? A[at + (int64_t)(j + r * (N / R0)) * es] : mk<float>(0.f, 0.f);
    constexpr int G = R0 < 8 ? R0 : 8;
#pragma unroll
    for (int r0 = 0; r0 < R0; r0 += G) {
      cpx<float> y[G];
#pragma unroll
      for (int g = 0; g < G; ++g)
        y[g] = live ? B[at + (int64_t)(j + (r0 + g) * (N / R0)) * es] : mk<float>(0.f, 0.f);
#pragma unroll
      for (int g = 0; g < G; ++g) {
        const int n = j + (r0 + g) * (N / R0), mz = signed_freq(n, N), az = mz < 0 ? -mz : mz;
        const float W = wxy * w[az < N / 2 ? az : 0];
        float Wp = W;
        if (p > 1) Wp *= W;
        if (p > 2) Wp *= W;
        const cpx<float> e = t[mz + N / 2 + col];
        const float f = n == N / 2 ? 0.f : scale / Wp;
        const cpx<float> x = v[r0 + g];
        v[r0 + g] = mk<float>(f * (x.x + e.x * y[g].x - e.y * y[g].y), f * (x.y + e.x * y[g].y + e.y * y[g].x));
      }
    }
  }
};

__device__ __forceinline__ float tophat_w(float x) {
  if (x < 0.5f) {  // series: the closed form cancels for small x
    const float x2 = x * x;
    return 1.0f - x2 * (0.1f - x2 * (1.0f / 280.0f - x2 * (1.0f / 15120.0f)));
  }
  float sn, cs;
  sincosf(x, &sn, &cs);
  return 3.0f * (sn - x * cs) / (x * x * x);
}

// Window of the filtered linear field by the integer |m|^2: sharp in k
// (kept for |m|^2 <= m2max) or a spherical top hat of radius R.
struct FilterOp {
  static constexpr bool kLoad = false, kFilter = true;
  int tophat;
  int m2max;
  float kf, R;
  __device__ __forceinline__ float window(int m2) const {
    if (tophat) return tophat_w(kf * sqrtf((float)m2) * R);
    return m2 <= m2max ? 1.f : 0.f;
  }
};

// What the x pass does with a value v of element i of `out`.
struct EpiStore {
  static constexpr bool kKeys = false;
  struct Aux {};
  __device__ __forceinline__ Aux fetch(const float*, int64_t) const { return {}; }
  __device__ __forceinline__ float value(Aux, float v) const { return v; }
};
// xx yy + xx v + yy v: the diagonal terms of the second-order source
struct EpiDiag {
  static constexpr bool kKeys = false;
  const float* xx;
  const float* yy;
  struct Aux {
    float x, y;
  };
  __device__ __forceinline__ Aux fetch(const float*, int64_t i) const { return {xx[i], yy[i]}; }
  __device__ __forceinline__ float value(Aux a, float v) const { return fmaf(a.x, a.y, fmaf(a.x, v, a.y * v)); }
};
// out - v^2: the mixed terms
struct EpiSubSquare {
  static constexpr bool kKeys = false;
  struct Aux {
    float s;
  };
  __device__ __forceinline__ Aux fetch(const float* out, int64_t i) const { return {out[i]}; }
  __device__ __forceinline__ float value(Aux a, float v) const { return fmaf(-v, v, a.s); }
};
// erfc((dc - v) inv): the collapsed fraction
struct EpiErfc {
  static constexpr bool kKeys = false;
  float dc, inv;
  struct Aux {};
  __device__ __forceinline__ Aux fetch(const float*, int64_t) const { return {}; }
  __device__ __forceinline__ float value(Aux, float v) const { return erfcf((dc - v) * inv); }
};

enum LinOut { LIN_STORE = 0, LIN_DIAG, LIN_SUB_SQUARE };

// Host entries (FP32, n a power of two in [4, 1024]); tmp: a half spectrum the
// passes may use (not one of the operator's inputs).
// out = inverse transform of op's spectrum; LIN_DIAG: combined with the fields
// xx, yy (EpiDiag); LIN_SUB_SQUARE: out -= (it)^2.
cudaError_t inverse_lin_f32(int n, const LinOp& op, int what, const float* xx, const float* yy, void* tmp, float* out,
                            const void* tw, unsigned int* status, cudaStream_t s);
cudaError_t inverse_interlace_f32(int n, const InterlaceOp& op, void* tmp, float* out, const void* tw,
                                  unsigned int* status, cudaStream_t s);
// out = erfc((dc - (src filtered by op)) inv)
cudaError_t filter_fcoll_f32(int n, const FilterOp& op, float dc, float inv, const float* src, void* tmp, float* out,
                             const void* tw, unsigned int* status, cudaStream_t s);

}  // namespace amber
