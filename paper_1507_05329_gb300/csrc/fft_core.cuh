// Device building blocks of the hand-written mixed-radix 3D FFT passes (sm_103a), shared by the
// kernels compiled per length (fft_ct.cuh) and the run-time plans (fft_generic.cu).
//
// The paper's PM force spends 66% of its time in FFTW (§2.3, Table 1).  Here each 1D pass of the
// 3D transform is one kernel that reads a tile of W pencils from HBM once, transforms it in shared
// memory with Stockham autosort stages of radix 16/8/6/5/4/3/2, and writes it once:
//   * contiguous axis (z): pairs of real rows packed as one complex row (R2C / C2R);
//   * strided axes (y, x): W adjacent complex columns per tile, so each row segment is a
//     contiguous W*8-byte run;
//   * the last forward pass (x) is fused with the Poisson Green function, the 4-point gradient
//     kernel and the inverse x transforms of the force components (§2.2 Poisson equation): F_x
//     has its own, F_y and F_z share one (their gradient factors are constant along x).
// Shared-memory layout of a tile: element (j, w) at ((j + j/16) * W + w); the skew of one W-row
// every 16 rows keeps the stride-R writes of the first Stockham stages off a single bank group.
#pragma once
#include "cola_internal.h"

#include <cmath>
#include <cstdio>

namespace cola {
namespace fftk {

constexpr int kEpt = 16;   // complex elements per thread (register staging of a stage)
constexpr int kMaxThreads = 384;   // largest tile (6144 elements) / kEpt

__device__ __forceinline__ float2 operator+(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 operator-(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ float2 operator*(float s, float2 a) { return make_float2(s * a.x, s * a.y); }
__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
  return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
// multiply by -i (forward, DIR < 0) or +i (inverse, DIR > 0)
template <int DIR>
__device__ __forceinline__ float2 mul_i(float2 a) {
  return DIR < 0 ? make_float2(a.y, -a.x) : make_float2(-a.y, a.x);
}
template <int DIR>
__device__ __forceinline__ float2 rot(float2 a, float c, float s) {   // a * (c + i*DIR*s)
  return DIR < 0 ? make_float2(a.x * c + a.y * s, a.y * c - a.x * s)
                 : make_float2(a.x * c - a.y * s, a.y * c + a.x * s);
}

// ---- small DFTs in registers, natural order in and out; sign of the exponent = DIR ----------
template <int R, int DIR> struct Dft;

template <int DIR> struct Dft<2, DIR> {
  __device__ __forceinline__ static void run(float2* v) {
    const float2 t = v[0];
    v[0] = t + v[1];
    v[1] = t - v[1];
  }
};

template <int DIR> struct Dft<4, DIR> {
  __device__ __forceinline__ static void run(float2* v) {
    const float2 t0 = v[0] + v[2], t1 = v[0] - v[2], t2 = v[1] + v[3];
    const float2 t3 = mul_i<DIR>(v[1] - v[3]);
    v[0] = t0 + t2;
    v[2] = t0 - t2;
    v[1] = t1 + t3;
    v[3] = t1 - t3;
  }
};

template <int DIR> struct Dft<8, DIR> {
  __device__ __forceinline__ static void run(float2* v) {
    const float c = 0.70710678118654752f;
    float2 e[4] = {v[0], v[2], v[4], v[6]};
    float2 o[4] = {v[1], v[3], v[5], v[7]};
    Dft<4, DIR>::run(e);
    Dft<4, DIR>::run(o);
    o[1] = rot<DIR>(o[1], c, c);
    o[2] = mul_i<DIR>(o[2]);
    o[3] = rot<DIR>(o[3], -c, c);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      v[k] = e[k] + o[k];
      v[k + 4] = e[k] - o[k];
    }
  }
};

template <int DIR> struct Dft<16, DIR> {
  __device__ __forceinline__ static void run(float2* v) {
    // w16^k = cos(pi k / 8) + i DIR sin(pi k / 8), k = 0..7
    const float cs[8] = {1.0f, 0.92387953251128674f, 0.70710678118654752f, 0.38268343236508977f,
                         0.0f, -0.38268343236508977f, -0.70710678118654752f, -0.92387953251128674f};
    const float sn[8] = {0.0f, 0.38268343236508977f, 0.70710678118654752f, 0.92387953251128674f,
                         1.0f, 0.92387953251128674f, 0.70710678118654752f, 0.38268343236508977f};
    float2 e[8], o[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      e[k] = v[2 * k];
      o[k] = v[2 * k + 1];
    }
    Dft<8, DIR>::run(e);
    Dft<8, DIR>::run(o);
#pragma unroll
    for (int k = 1; k < 8; ++k) o[k] = rot<DIR>(o[k], cs[k], sn[k]);
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      v[k] = e[k] + o[k];
      v[k + 8] = e[k] - o[k];
    }
  }
};

template <int DIR> struct Dft<3, DIR> {
  __device__ __forceinline__ static void run(float2* v) {
    const float h = 0.86602540378443865f;   // sqrt(3)/2
    const float2 s = v[1] + v[2], d = v[1] - v[2];
    const float2 m = v[0] - 0.5f * s;
    const float2 t = h * mul_i<DIR>(d);
    v[0] = v[0] + s;
    v[1] = m + t;
    v[2] = m - t;
  }
};

// 6 = 2 x 3: radix 2 first, a_j = x_j + x_{j+3} and b_j = (x_j - x_{j+3}) w6^j, then a 3-point DFT of
// each; the even outputs come from a, the odd from b.
template <int DIR> struct Dft<6, DIR> {
  __device__ __forceinline__ static void run(float2* v) {
    const float h = 0.86602540378443865f;   // sqrt(3)/2
    float2 a[3] = {v[0] + v[3], v[1] + v[4], v[2] + v[5]};
    float2 b[3] = {v[0] - v[3], v[1] - v[4], v[2] - v[5]};
    b[1] = cmul(b[1], make_float2(0.5f, DIR * h));
    b[2] = cmul(b[2], make_float2(-0.5f, DIR * h));
    Dft<3, DIR>::run(a);
    Dft<3, DIR>::run(b);
    v[0] = a[0];
    v[1] = b[0];
    v[2] = a[1];
    v[3] = b[1];
    v[4] = a[2];
    v[5] = b[2];
  }
};

template <int DIR> struct Dft<5, DIR> {
  __device__ __forceinline__ static void run(float2* v) {
    const float c1 = 0.30901699437494742f, c2 = -0.80901699437494742f;
    const float s1 = 0.95105651629515357f, s2 = 0.58778525229247313f;
    const float2 a1 = v[1] + v[4], b1 = v[1] - v[4], a2 = v[2] + v[3], b2 = v[2] - v[3];
    const float2 m1 = v[0] + c1 * a1 + c2 * a2;
    const float2 m2 = v[0] + c2 * a1 + c1 * a2;
    const float2 t1 = mul_i<DIR>(s1 * b1 + s2 * b2);
    const float2 t2 = mul_i<DIR>(s2 * b1 - s1 * b2);
    v[0] = v[0] + a1 + a2;
    v[1] = m1 + t1;
    v[4] = m1 - t1;
    v[2] = m2 + t2;
    v[3] = m2 - t2;
  }
};

__device__ __forceinline__ int saddr(int j, int w, int lw) { return ((j + (j >> 4)) << lw) + w; }

// One Stockham stage on W pencils of length n (Govindaraju et al. 2008 formulation): butterfly b
// reads x[b + r n/R], twiddles by w_n^(r k n/(Ns R)) with k = b mod Ns, and writes
// y[(b - k) R + k + r Ns].  Ping-pong between two shared buffers, one barrier per stage.
template <int R, int DIR>
__device__ __forceinline__ void fft_stage(const float2* x, float2* y, int n, int lw,
                                          int ns, const float2* __restrict__ tw, int tid, int nthreads) {
  const int nb = n / R;
  const int total = nb << lw;
  const int tstride = n / (ns * R);
  const int wmask = (1 << lw) - 1;
  for (int idx = tid; idx < total; idx += nthreads) {
    const int w = idx & wmask, b = idx >> lw;
    const int k = b % ns;
    float2 v[R];
#pragma unroll
    for (int r = 0; r < R; ++r) v[r] = x[saddr(b + r * nb, w, lw)];
    if (ns > 1) {
#pragma unroll
      for (int r = 1; r < R; ++r) {
        float2 t = __ldg(&tw[r * k * tstride]);
        if (DIR > 0) t.y = -t.y;
        v[r] = cmul(v[r], t);
      }
    }
    Dft<R, DIR>::run(v);
    const int base = (b - k) * R + k;
#pragma unroll
    for (int r = 0; r < R; ++r) y[saddr(base + r * ns, w, lw)] = v[r];
  }
  __syncthreads();
}

// All stages of the plan; the data starts in buffer a and the returned pointer holds the result.
template <int DIR>
__device__ float2* fft_smem(float2* a, float2* b, const FftDev& p, int lw, int tid, int nthreads) {
  int ns = 1;
  for (int st = 0; st < p.nstages; ++st) {
    const int r = p.radix[st];
    switch (r) {
      case 16: fft_stage<16, DIR>(a, b, p.n, lw, ns, p.tw, tid, nthreads); break;
      case 8: fft_stage<8, DIR>(a, b, p.n, lw, ns, p.tw, tid, nthreads); break;
      case 6: fft_stage<6, DIR>(a, b, p.n, lw, ns, p.tw, tid, nthreads); break;
      case 5: fft_stage<5, DIR>(a, b, p.n, lw, ns, p.tw, tid, nthreads); break;
      case 4: fft_stage<4, DIR>(a, b, p.n, lw, ns, p.tw, tid, nthreads); break;
      case 3: fft_stage<3, DIR>(a, b, p.n, lw, ns, p.tw, tid, nthreads); break;
      default: fft_stage<2, DIR>(a, b, p.n, lw, ns, p.tw, tid, nthreads); break;
    }
    float2* t = a;
    a = b;
    b = t;
    ns *= r;
  }
  return a;
}

__device__ __forceinline__ int tile_elems(int n, int lw) { return (n + n / 16 + 1) << lw; }

// Raises a kernel's dynamic shared-memory limit the first time it is launched on the current
// device (host side; the attribute is per device).
template <class K>
inline void ensure_smem(K kernel) {
  once_on_device(reinterpret_cast<const void*>(kernel), [](const void* k) {
    cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
  });
}

}  // namespace fftk

// Launchers of the run-time plans (fft_generic.cu).
void generic_r2c_launch(const FftDev& d, int lw, unsigned blocks, int threads, size_t smem, int kind, const void* src,
                        long long rs, float scale, float2* dst, int pc, long long nrows, unsigned long long* acc,
                        cudaStream_t st);
void generic_c2r_launch(const FftDev& d, int lw, unsigned blocks, int threads, size_t smem, float2* data, int pc,
                        long long nrows, cudaStream_t st);
void generic_pencils_launch(const FftDev& d, int lw, dim3 grid, int threads, size_t smem, int dir, float2* data,
                            long long jstride, long long ostride, int nc, cudaStream_t st);
void generic_green_launch(const FftDev& d, int lw, dim3 grid, int threads, size_t smem, const float2* in,
                          float2* const out[3], int pc, int nc, const float* dtab, float g_scale, cudaStream_t st);
void generic_set_smem_limits();

}  // namespace cola
