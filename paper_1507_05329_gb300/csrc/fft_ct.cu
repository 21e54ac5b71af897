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
  launch_after(kern, grid, threads, smem, st, args...);
}

template <int N>
struct Launch {
  using C = PenCfg<N>;
  using R = RowCfg<N>;
  static constexpr long long kPairs = (long long)N * N / 2;
  static constexpr unsigned kRowBlocks = (unsigned)((kPairs + R::pairs - 1) / R::pairs);

  static void r2c(int kind, const void* const* src, int fields, long long rs, float scale, float2* const* dst,
                  const FftTables& t, unsigned long long* acc, cudaStream_t st) {
    Src3 s{};
    Ptr3 d{};
    for (int i = 0; i < fields; ++i) {
      s.p[i] = src[i];
      d.p[i] = dst[i];
    }
    const dim3 grid(kRowBlocks, fields);
    if (kind == kSrcFixedPoint)
      go(k_r2c<N, kSrcFixedPoint>, grid, R::T, R2cCfg<N>::smem, st, s, rs, scale, d, kPairs, t.fwd, acc);
    else
      go(k_r2c<N, kSrcFloat>, grid, R::T, R2cCfg<N>::smem, st, s, rs, scale, d, kPairs, t.fwd,
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
  // lattices up to 1024 (three tiles fit a CTA) have the fused 2LPT passes; only longer ones multiply field by field
  static constexpr bool kIc = N <= 1024;
  static_assert(!kIc || MultiCfg<N, 3>::smem <= 227 * 1024, "three tiles in a CTA");
  static void x_mul(const float2* src, const IcMul& mul, float2* dst, const FftTables& t, cudaStream_t st) {
    if constexpr (!kIc) go(k_pen_mul<N>, dim3(C::chunks, N), C::T, C::smem, st, src, dst, mul, t.fwd);
  }
  static void green(const float2* in, float2* out_f, float2* out_h, const float* dtab, float g_scale,
                    const FftTables& t, float2* spec_out, cudaStream_t st) {
    go(k_green<N>, dim3(C::chunks, N), C::T, MultiCfg<N, 2>::smem, st, in, out_f, out_h, dtab, g_scale, t.fwd, t.rev,
       spec_out);
  }
  static void pencils_yz(const float2* h, float2* out_y, float2* out_z, const float* dtab, const FftTables& t,
                         cudaStream_t st) {
    go(k_pen_yz<N>, dim3(C::chunks, N), C::T, MultiCfg<N, 2>::smem, st, h, out_y, out_z, dtab, t.fwd);
  }

  static void ic_x(const float2* in, float2* const* out, int fields, float scale, const float* amp_m2,
                   const FftTables& t, cudaStream_t st) {
    if constexpr (kIc) {
      const dim3 grid(C::chunks, N);
      if (fields == 3)
        go(k_ic_x<N, 3, true>, grid, C::T, MultiCfg<N, 3>::smem, st, in, Ptr3{{out[0], out[1], out[2]}}, scale, amp_m2,
           t.fwd, t.rev);
      else
        go(k_ic_x<N, 2, false>, grid, C::T, MultiCfg<N, 2>::smem, st, in, Ptr3{{out[0], out[1], nullptr}}, scale,
           (const float*)nullptr, t.fwd, t.rev);
    }
  }
  static void ic_y(const float2* in, float2* const* out, int fields, const int* zp, const FftTables& t,
                   cudaStream_t st) {
    if constexpr (kIc) {
      const dim3 grid(C::chunks, N);
      Pow3 z{};
      for (int i = 0; zp && i < fields; ++i) z.p[i] = zp[i];
      if (fields == 3)
        go(k_ic_y<N, 3>, grid, C::T, MultiCfg<N, 3>::smem, st, in, Ptr3{{out[0], out[1], out[2]}}, z,
           t.fwd);
      else
        go(k_ic_y<N, 2>, grid, C::T, MultiCfg<N, 2>::smem, st, in, Ptr3{{out[0], out[1], nullptr}}, z,
           t.fwd);
    }
  }
  static void ic_z1(float2* const* f, float2* src_k, float* psi1, float r_scale, const FftTables& t, cudaStream_t st) {
    if constexpr (kIc)
      go(k_ic_z1<N>, kRowBlocks, R::T, IcRowCfg<N>::smem, st, IcRows{{f[0], f[1], f[2], f[3], f[4], f[5]}}, src_k, psi1,
         (long long)N * N * N, r_scale, kPairs, t.fwd);
  }
  static void ic_z2(float2* const* f, const float* psi1, float* psi2, float* s, float* v, float r_scale, float d1,
                    float d2, const FftTables& t, cudaStream_t st) {
    if constexpr (kIc)
      go(k_ic_z2<N>, dim3(kRowBlocks, 3), R::T, C2rCfg<N>::smem, st, Ptr3{{f[0], f[1], f[2]}}, psi1, psi2, s, v,
         (long long)N * N * N, r_scale, d1, d2, kPairs, t.fwd);
  }
  static void lpt_adj(const float2* const* h, const float2* const* p, float2* out, float r_scale, const float* amp_m2,
                      const FftTables& t, cudaStream_t st) {
    if constexpr (kIc)
      go(k_lpt_adj<N>, dim3(C::chunks, N), C::T, MultiCfg<N, 3>::smem, st,
         Lpt9{{h[0], h[1], h[2], h[3], h[4], h[5]}, {p[0], p[1], p[2]}}, out, r_scale, amp_m2, t.fwd, t.rev);
  }
  static void grad_adj(float2* const* l, float2* out, const float* dtab, float g_scale, const FftTables& t,
                       cudaStream_t st) {
    go(k_grad_adj<N>, dim3(C::chunks, N), C::T, MultiCfg<N, 2>::smem, st, (const float2*)l[0], (const float2*)l[1],
       (const float2*)l[2], out, dtab, g_scale, t.fwd, t.rev);
  }
};

// the launches of size I, and the table of this part's sizes
template <int I>
constexpr FftOps ops_of() {
  constexpr int N = kCtSizes[I];
  using L = Launch<N>;
  return FftOps{N, L::r2c, L::c2r, L::c2r_dense, L::pencils, L::kIc ? nullptr : L::x_mul, L::green,
                L::kIc ? L::ic_x : nullptr, L::ic_y, L::ic_z1, L::ic_z2, L::lpt_adj, L::grad_adj, L::pencils_yz};
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
