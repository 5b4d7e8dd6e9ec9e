// Inverse transforms with fused spectral operators, FP32 (see fft_ops.cuh).
#include "fft_ops.cuh"

namespace amber {

namespace {

template <int N> struct Geom {
  using C = FftCfg<N>;
  static constexpr int RS = N / 2 + 2, ncol = N / 2 + 1;
  static constexpr int ntx = (ncol + C::SB - 1) / C::SB, sgrid = N * ntx;
  static constexpr int64_t nrows = (int64_t)N * N;
  static constexpr int xgrid = (int)((nrows / 2 + C::XP - 1) / C::XP);
  static constexpr size_t xs = XSmem<float, N>::elems * sizeof(cpx<float>);
  static constexpr size_t ss = StridedSmem<float, N>::elems * sizeof(cpx<float>);
};

// z pass with op into tmp, then the inverse y pass in place
template <int N, int MODE, class OP>
cudaError_t zy_passes(const OP& op, size_t table, cpx<float>* tmp, const cpx<float>* tw, float norm, cudaStream_t s) {
  using G = Geom<N>;
  static PerDeviceOnce attr;  // per instantiation and device
  once_on_device(attr, [&](DeviceSetUp& u) {
    u.smem(k_fft_strided<float, N, MODE, 0, false, false, OP>, G::ss + table);
    u.smem(k_fft_strided<float, N, PASS_INV>, G::ss);
  });
  run_strided<float, N, MODE, 0, false, false, OP>(G::sgrid, G::ss + table, s, tmp, (int64_t)N * G::RS, G::RS, G::ncol, G::ntx, tw, 0.f, 0.f, norm, nullptr, 0, nullptr, op);
  run_strided<float, N, PASS_INV>(G::sgrid, G::ss, s, tmp, G::RS, (int64_t)N * G::RS,
                                                                                G::ncol, G::ntx, tw, 0.f, 0.f, 0.f);
  return cudaGetLastError();
}

template <int N, class EPI>
cudaError_t x_pass(const EPI& epi, const cpx<float>* tmp, float* out, const cpx<float>* tw, unsigned int* status,
                   cudaStream_t s) {
  using G = Geom<N>;
  static PerDeviceOnce attr;
  once_on_device(attr, [&](DeviceSetUp& u) {
    u.smem(k_fft_c2r_x<float, N, 0, false, false, EPI>, G::xs);
  });
  run_c2r<float, N, 0, false, false, EPI>(G::xgrid, G::xs, s, tmp, out, G::nrows, G::RS, tw, status, nullptr, 0, epi);
  return cudaGetLastError();
}

template <int N>
cudaError_t inverse_lin_n(const LinOp& op, int what, const float* xx, const float* yy, cpx<float>* tmp, float* out,
                          const cpx<float>* tw, unsigned int* status, cudaStream_t s) {
  cudaError_t e = zy_passes<N, PASS_INV>(op, LinOp::table_bytes<N, FftCfg<N>::SB>(), tmp, tw, 0.f, s);
  if (e != cudaSuccess) return e;
  if (what == LIN_DIAG) return x_pass<N>(EpiDiag{xx, yy}, tmp, out, tw, status, s);
  if (what == LIN_SUB_SQUARE) return x_pass<N>(EpiSubSquare{}, tmp, out, tw, status, s);
  return x_pass<N>(EpiStore{}, tmp, out, tw, status, s);
}

template <int N>
cudaError_t inverse_interlace_n(const InterlaceOp& op, cpx<float>* tmp, float* out, const cpx<float>* tw,
                                unsigned int* status, cudaStream_t s) {
  cudaError_t e = zy_passes<N, PASS_INV>(op, InterlaceOp::table_bytes<N, FftCfg<N>::SB>(), tmp, tw, 0.f, s);
  return e != cudaSuccess ? e : x_pass<N>(EpiStore{}, tmp, out, tw, status, s);
}

template <int N>
cudaError_t filter_fcoll_n(const FilterOp& op, float dc, float inv, const float* src, cpx<float>* tmp, float* out,
                           const cpx<float>* tw, unsigned int* status, cudaStream_t s) {
  cudaError_t e = source_spectrum_n<float, N>(src, tmp, tw, s, nullptr);
  if (e == cudaSuccess)
    e = zy_passes<N, PASS_CONV>(op, (size_t)(N / 2 + 1) * FftCfg<N>::SB * sizeof(float), tmp, tw,
                                (float)(1.0 / ((double)N * N * N)), s);
  return e != cudaSuccess ? e : x_pass<N>(EpiErfc{dc, inv}, tmp, out, tw, status, s);
}

}  // namespace

#define AMBER_BY_SIZE(F, ...)              \
  switch (n) {                             \
    case 4: return F<4>(__VA_ARGS__);      \
    case 8: return F<8>(__VA_ARGS__);      \
    case 16: return F<16>(__VA_ARGS__);    \
    case 32: return F<32>(__VA_ARGS__);    \
    case 64: return F<64>(__VA_ARGS__);    \
    case 128: return F<128>(__VA_ARGS__);  \
    case 256: return F<256>(__VA_ARGS__);  \
    case 512: return F<512>(__VA_ARGS__);  \
    case 1024: return F<1024>(__VA_ARGS__);\
    default: return cudaErrorInvalidValue; \
  }

cudaError_t inverse_lin_f32(int n, const LinOp& op, int what, const float* xx, const float* yy, void* tmp, float* out,
                            const void* tw, unsigned int* status, cudaStream_t s) {
  auto* h = reinterpret_cast<cpx<float>*>(tmp);
  auto* w = reinterpret_cast<const cpx<float>*>(tw);
  AMBER_BY_SIZE(inverse_lin_n, op, what, xx, yy, h, out, w, status, s)
}

cudaError_t inverse_interlace_f32(int n, const InterlaceOp& op, void* tmp, float* out, const void* tw,
                                  unsigned int* status, cudaStream_t s) {
  auto* h = reinterpret_cast<cpx<float>*>(tmp);
  auto* w = reinterpret_cast<const cpx<float>*>(tw);
  AMBER_BY_SIZE(inverse_interlace_n, op, h, out, w, status, s)
}

cudaError_t filter_fcoll_f32(int n, const FilterOp& op, float dc, float inv, const float* src, void* tmp, float* out,
                             const void* tw, unsigned int* status, cudaStream_t s) {
  auto* h = reinterpret_cast<cpx<float>*>(tmp);
  auto* w = reinterpret_cast<const cpx<float>*>(tw);
  AMBER_BY_SIZE(filter_fcoll_n, op, dc, inv, src, h, out, w, status, s)
}

}  // namespace amber
