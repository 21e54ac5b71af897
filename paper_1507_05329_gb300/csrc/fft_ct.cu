// The FFT kernels of the compiled lengths (fft_ct.cuh).  This file is compiled COLA_CT_PARTS times, part
// COLA_CT_PART holding every COLA_CT_PARTS-th length, so that the parts build in parallel.
#include "fft_ct.cuh"
#include "fft_ops.h"

#include <utility>

namespace cola {
namespace ct {
namespace {

template <class K, class... A>
void go(K kern, dim3 grid, int threads, int smem, cudaStream_t st, A... args) {
  if (smem > 48 * 1024) ensure_smem(kern);
  kern<<<grid, threads, smem, st>>>(args...);
}

template <int N>
struct Launch {
  using C = PenCfg<N>;
  using R = RowCfg<N>;
  static constexpr long long kPairs = (long long)N * N / 2;
  static constexpr unsigned kRowBlocks = (unsigned)((kPairs + R::pairs - 1) / R::pairs);

  static void r2c(int kind, const void* src, long long rs, float scale, float2* dst, const FftTables& t,
                  unsigned long long* acc, cudaStream_t st) {
    if (kind == kSrcFixedPoint)
      go(k_r2c<N, kSrcFixedPoint>, kRowBlocks, R::T, R2cCfg<N>::smem, st, src, rs, scale, dst, kPairs, t.fwd, acc);
    else
      go(k_r2c<N, kSrcFloat>, kRowBlocks, R::T, R2cCfg<N>::smem, st, src, rs, scale, dst, kPairs, t.fwd,
         (unsigned long long*)nullptr);
  }
  static void c2r(float2* const* data, int fields, const FftTables& t, cudaStream_t st) {
    Ptr3 p{};
    for (int i = 0; i < fields; ++i) p.p[i] = data[i];
    go(k_c2r<N, false>, dim3(kRowBlocks, fields), R::T, C2rCfg<N>::smem, st, p, kPairs, t.fwd, (float*)nullptr, 1.0f);
  }
  static void c2r_dense(const float2* data, float scale, float* out, const FftTables& t, cudaStream_t st) {
    Ptr3 p{{const_cast<float2*>(data), nullptr, nullptr}};   // only read
    go(k_c2r<N, true>, dim3(kRowBlocks, 1), R::T, C2rCfg<N>::smem, st, p, kPairs, t.fwd, out, scale);
  }
  static void pencils(int axis, int dir, float2* const* data, int fields, const FftTables& t, cudaStream_t st) {
    Ptr3 p{};
    for (int i = 0; i < fields; ++i) p.p[i] = data[i];
    const dim3 grid(C::chunks, N, fields);
    if (axis == 1) {
      if (dir < 0) go(k_pen<N, 1, -1>, grid, C::T, C::smem, st, p, t.fwd);
      else go(k_pen<N, 1, +1>, grid, C::T, C::smem, st, p, t.fwd);
    } else {
      if (dir < 0) go(k_pen<N, 0, -1>, grid, C::T, C::smem, st, p, t.fwd);
      else go(k_pen<N, 0, +1>, grid, C::T, C::smem, st, p, t.fwd);
    }
  }
  static void x_mul(const float2* src, const IcMul& mul, float2* dst, const FftTables& t, cudaStream_t st) {
    go(k_pen_mul<N>, dim3(C::chunks, N), C::T, C::smem, st, src, dst, mul, t.fwd);
  }
  static void green(const float2* in, float2* out_f, float2* out_h, const float* dtab, float g_scale,
                    const FftTables& t, float2* spec_out, cudaStream_t st) {
    go(k_green<N>, dim3(C::chunks, N), C::T, PairCfg<N>::smem, st, in, out_f, out_h, dtab, g_scale, t.fwd, t.rev,
       spec_out);
  }
  static void pencils_yz(const float2* h, float2* out_y, float2* out_z, const float* dtab, const FftTables& t,
                         cudaStream_t st) {
    go(k_pen_yz<N>, dim3(C::chunks, N), C::T, PairCfg<N>::smem, st, h, out_y, out_z, dtab, t.fwd);
  }
};

// whether part COLA_CT_PART holds size i, and the part's table
template <int I>
constexpr FftOps ops_of() {
  constexpr int N = kCtSizes[I];
  using L = Launch<N>;
  return FftOps{N, L::r2c, L::c2r, L::c2r_dense, L::pencils, L::x_mul, L::green, L::pencils_yz};
}
constexpr int kMine = (kCtCount - COLA_CT_PART + COLA_CT_PARTS - 1) / COLA_CT_PARTS;
template <int... K>
const FftOps* find(int n, std::integer_sequence<int, K...>) {
  static const FftOps table[] = {ops_of<COLA_CT_PART + K * COLA_CT_PARTS>()...};
  for (const FftOps& o : table)
    if (o.n == n) return &o;
  return nullptr;
}

}  // namespace

template <>
const FftOps* ops_in_part<COLA_CT_PART>(int n) {
  return find(n, std::make_integer_sequence<int, kMine>{});
}

}  // namespace ct
}  // namespace cola
