// FFT pass kernels compiled for one length N each: radices, strides, tile shapes and twiddle offsets are
// compile-time constants, so a butterfly costs its arithmetic, its loads and stores with immediate
// offsets and one index computation.
//
// Every pass reads a tile of pencils from HBM once, runs the groups of the length's plan (fft_plan.h) on
// it through shared memory and writes it once; the first group loads straight from HBM and the last
// stores straight to it.  Strided passes (y, x) take tiles of 8 adjacent columns (64-byte row segments; 4 beyond 1536),
// lanes running over the columns first; the contiguous passes (z) take pairs of real rows as complex
// rows, lanes running along the row, so that their global accesses are whole 128-byte lines.
#pragma once
#include "fft_core.cuh"
#include "fft_plan.h"

namespace cola {
namespace ct {

using namespace fftk;

constexpr int round_up(int v, int m) { return (v + m - 1) / m * m; }
constexpr int imin(int a, int b) { return a < b ? a : b; }
constexpr int imax(int a, int b) { return a > b ? a : b; }

template <int N, bool REV>
struct PlanOf {
  static constexpr Groups g = make_groups(N, REV);
  static constexpr int m = g.m;
};

// One group of a plan on the values v[r] = x[b + r N/R] of butterfly b, k = b mod ns; on return
// v[r] belongs at (b - k) R + k + r ns.
template <int N, bool REV, int G, int DIR>
struct Group {
  static constexpr Groups P = make_groups(N, REV);
  static constexpr int R1 = P.r1[G], R2 = P.r2[G], R = R1 * R2, NS = P.ns[G], NB = N / R, O1 = P.off1[G], O2 = P.off2[G];

  __device__ __forceinline__ static float2 tw(const float2* __restrict__ t) {
    float2 w = __ldg(t);
    if (DIR > 0) w.y = -w.y;
    return w;
  }
  __device__ __forceinline__ static void run(float2 (&v)[R], const float2* __restrict__ table, int k) {
    const float2* t1 = table + O1 + k;
    if constexpr (R2 == 1) {
      if constexpr (NS > 1) {
#pragma unroll
        for (int r = 1; r < R1; ++r) v[r] = cmul(v[r], tw(t1 + (r - 1) * NS));
      }
      Dft<R1, DIR>::run(v);
    } else {
      // stage r1 on the R2 sub-butterflies b + i N/R, then stage r2 on the R1 butterflies their
      // outputs r share
#pragma unroll
      for (int i = 0; i < R2; ++i) {
        float2 t[R1];
#pragma unroll
        for (int r = 0; r < R1; ++r) t[r] = v[i + r * R2];
        if constexpr (NS > 1) {
#pragma unroll
          for (int r = 1; r < R1; ++r) t[r] = cmul(t[r], tw(t1 + (r - 1) * NS));
        }
        Dft<R1, DIR>::run(t);
#pragma unroll
        for (int r = 0; r < R1; ++r) v[i + r * R2] = t[r];
      }
      const float2* t2 = table + O2 + k;
      float2 o[R];
#pragma unroll
      for (int r = 0; r < R1; ++r) {
        float2 u[R2];
#pragma unroll
        for (int i = 0; i < R2; ++i) u[i] = v[i + r * R2];
        if (NS > 1 || r > 0) {
#pragma unroll
          for (int i = 1; i < R2; ++i) u[i] = cmul(u[i], tw(t2 + (i - 1) * NS * R1 + r * NS));
        }
        Dft<R2, DIR>::run(u);
#pragma unroll
        for (int i = 0; i < R2; ++i) o[r + i * R1] = u[i];
      }
#pragma unroll
      for (int r = 0; r < R; ++r) v[r] = o[r];
    }
  }
  __device__ __forceinline__ static int k_of(int b) {
    if constexpr (NS == 1) return 0;
    else if constexpr (NS == NB) return b;
    else return b % NS;
  }
  __device__ __forceinline__ static int out_row(int b, int k) { return (b - k) * R + k; }
};

// ---- tiles of W columns (strided passes) ---------------------------------------------------------
// element (j, w) at (j << LW) + w.  Rows are 64 bytes: only the stores of a first group of even radix
// meet two rows on the same banks (a pair of wavefronts for one), which costs less than a padded index.
template <int N>
struct PenCfg {
  static constexpr int lw = N <= 1536 ? 3 : 2;             // two tiles (the Green pass) fit a CTA
  static constexpr int W = 1 << lw;
  static constexpr Groups P = make_groups(N, false);
  static constexpr int ept = P.max_radix > 10 ? 16 : 8;   // values a thread holds in a group
  static constexpr int T = imin(1024, round_up((N * W + ept - 1) / ept, 32));
  static constexpr int PC = ((N / 2 + 1) + 1) & ~1;
  static constexpr int NC = N / 2 + 1;
  static constexpr int chunks = (NC + W - 1) / W;
  static constexpr int tile = N * W;                       // complex elements
  // one work buffer that the middle groups overwrite (each thread's values in registers over a barrier);
  // two where two still leave as many CTAs per SM as the registers do
  static constexpr int regs = ept == 16 ? 64 : 40;
  static constexpr int by_regs = imax(1, imin(2048, 65536 / regs) / T);
  static constexpr bool pp = P.m > 2 && 2 * tile * 8 * by_regs <= 220 * 1024;
  static constexpr int bufs = pp ? 2 : 1;
  static constexpr int smem = bufs * tile * 8;
  static constexpr int minb = imax(1, imin(imin(by_regs, 24), (224 * 1024) / (smem + 1024)));
};

template <int N>
struct TileR {
  const float2* s;
  __device__ __forceinline__ float2 operator()(int j, int w) const { return s[(j << PenCfg<N>::lw) + w]; }
};
template <int N>
struct TileW {
  float2* s;
  __device__ __forceinline__ void operator()(int j, int w, float2 v) const { s[(j << PenCfg<N>::lw) + w] = v; }
};

// W adjacent columns of a strided pencil of row stride JS; columns beyond the row's valid entries read 0
template <long long JS>
struct ColG {
  float2* base;   // column col0 + w of row 0
  bool ok;        // the thread's column exists
  __device__ __forceinline__ float2 operator()(int j, int) const { return ok ? base[j * JS] : make_float2(0.f, 0.f); }
  __device__ __forceinline__ void operator()(int j, int, float2 v) const {
    if (ok) base[j * JS] = v;
  }
};

template <int N, bool REV, int G, int DIR, int T, class Src, class Dst>
__device__ __forceinline__ void pen_stage(const Src& src, const Dst& dst, const float2* __restrict__ tw, int tid) {
  using Q = Group<N, REV, G, DIR>;
  constexpr int TOT = Q::NB << PenCfg<N>::lw, IT = (TOT + T - 1) / T;
#pragma unroll(IT <= 2 ? IT : 1)
  for (int it = 0; it < IT; ++it) {
    const int idx = tid + it * T;
    if (TOT % T == 0 || idx < TOT) {
      const int w = idx & (PenCfg<N>::W - 1), b = idx >> PenCfg<N>::lw, k = Q::k_of(b);
      float2 v[Q::R];
#pragma unroll
      for (int r = 0; r < Q::R; ++r) v[r] = src(b + r * Q::NB, w);
      Q::run(v, tw, k);
      const int o = Q::out_row(b, k);
#pragma unroll
      for (int r = 0; r < Q::R; ++r) dst(o + r * Q::NS, w, v[r]);
    }
  }
}

// a middle group that overwrites its buffer; the caller synchronises before the next group reads
template <int N, bool REV, int G, int DIR, int T>
__device__ __forceinline__ void pen_inplace(float2* buf, const float2* __restrict__ tw, int tid) {
  using Q = Group<N, REV, G, DIR>;
  constexpr int TOT = Q::NB << PenCfg<N>::lw, IT = (TOT + T - 1) / T;
  float2 v[IT][Q::R];
#pragma unroll
  for (int it = 0; it < IT; ++it) {
    const int idx = tid + it * T;
    if (TOT % T == 0 || idx < TOT) {
#pragma unroll
      for (int r = 0; r < Q::R; ++r) v[it][r] = buf[idx + r * (Q::NB << PenCfg<N>::lw)];
    }
  }
  __syncthreads();
#pragma unroll
  for (int it = 0; it < IT; ++it) {
    const int idx = tid + it * T;
    if (TOT % T == 0 || idx < TOT) {
      const int w = idx & (PenCfg<N>::W - 1), b = idx >> PenCfg<N>::lw, k = Q::k_of(b);
      Q::run(v[it], tw, k);
      const int o = (Q::out_row(b, k) << PenCfg<N>::lw) + w;
#pragma unroll
      for (int r = 0; r < Q::R; ++r) buf[o + r * (Q::NS << PenCfg<N>::lw)] = v[it][r];
    }
  }
}

// groups 1 .. m-2 from a (ping-pong with b, or in place); returns the buffer that holds the result,
// synchronised
template <int N, bool REV, int DIR, int T, bool PP, int G = 1>
__device__ __forceinline__ float2* pen_middle(float2* a, float2* b, const float2* __restrict__ tw, int tid) {
  if constexpr (G + 1 < PlanOf<N, REV>::m) {
    if constexpr (PP) {
      pen_stage<N, REV, G, DIR, T>(TileR<N>{a}, TileW<N>{b}, tw, tid);
      __syncthreads();
      return pen_middle<N, REV, DIR, T, PP, G + 1>(b, a, tw, tid);
    } else {
      pen_inplace<N, REV, G, DIR, T>(a, tw, tid);
      __syncthreads();
      return pen_middle<N, REV, DIR, T, PP, G + 1>(a, b, tw, tid);
    }
  } else {
    return a;
  }
}

struct Ptr3 {
  float2* p[3];
};
struct Src3 {
  const void* p[3];
};

// C2C along y (AXIS 1) or x (AXIS 0), in place, of the fields data.p[blockIdx.z]
template <int N, int AXIS, int DIR>
__global__ void __launch_bounds__(PenCfg<N>::T, PenCfg<N>::minb) k_pen(Ptr3 data, const float2* __restrict__ tw) {
  extern __shared__ float2 sm[];
  using C = PenCfg<N>;
  constexpr long long JS = AXIS == 1 ? C::PC : (long long)N * C::PC, OS = AXIS == 1 ? (long long)N * C::PC : C::PC;
  const int tid = threadIdx.x, col = blockIdx.x * PenCfg<N>::W + (tid & (PenCfg<N>::W - 1));
  const ColG<JS> g{data.p[blockIdx.z] + blockIdx.y * OS + col, col < C::NC};
  pen_stage<N, false, 0, DIR, C::T>(g, TileW<N>{sm}, tw, tid);
  __syncthreads();
  float2* cur = pen_middle<N, false, DIR, C::T, C::pp>(sm, sm + C::tile, tw, tid);
  pen_stage<N, false, PlanOf<N, false>::m - 1, DIR, C::T>(TileR<N>{cur}, g, tw, tid);
}

// The inverse x pass of the 2LPT multiplier mp times the lattice spectrum src, into dst
template <long long JS>
struct ColMul {
  const float2* base;
  bool ok;
  int n, my, mz;
  IcMul mp;
  __device__ __forceinline__ float2 operator()(int j, int) const {
    if (!ok) return make_float2(0.f, 0.f);
    const int m[3] = {signed_mode(j, n), my, mz};
    return ic_multiply_mode(base[j * JS], m, n, mp);
  }
};
template <int N>
__global__ void __launch_bounds__(PenCfg<N>::T, PenCfg<N>::minb) k_pen_mul(const float2* __restrict__ src, float2* dst,
                                                                           IcMul mp, const float2* __restrict__ tw) {
  extern __shared__ float2 sm[];
  using C = PenCfg<N>;
  constexpr long long JS = (long long)N * C::PC;
  const int tid = threadIdx.x, col = blockIdx.x * PenCfg<N>::W + (tid & (PenCfg<N>::W - 1)), y = blockIdx.y;
  const bool ok = col < C::NC;
  const ColMul<JS> g{src + (long long)y * C::PC + col, ok, N, signed_mode(y, N), col, mp};
  pen_stage<N, false, 0, +1, C::T>(g, TileW<N>{sm}, tw, tid);
  __syncthreads();
  float2* cur = pen_middle<N, false, +1, C::T, C::pp>(sm, sm + C::tile, tw, tid);
  pen_stage<N, false, PlanOf<N, false>::m - 1, +1, C::T>(TileR<N>{cur}, ColG<JS>{dst + (long long)y * C::PC + col, ok}, tw, tid);
}

// NT transforms at once from here on, in the tiles s, s + tile, ...: middle groups in place, last groups
// to d[0], d[1], ...
template <int N, bool REV, int DIR, int T, int G, int NT, class D>
__device__ __forceinline__ void multi_finish(float2* s, const D (&d)[NT], const float2* __restrict__ tw, int tid) {
  constexpr int M = PlanOf<N, REV>::m;
  if constexpr (G + 1 < M) {
#pragma unroll
    for (int i = 0; i < NT; ++i) pen_inplace<N, REV, G, DIR, T>(s + i * PenCfg<N>::tile, tw, tid);
    __syncthreads();
    multi_finish<N, REV, DIR, T, G + 1>(s, d, tw, tid);
  } else {
#pragma unroll
    for (int i = 0; i < NT; ++i) pen_stage<N, REV, G, DIR, T>(TileR<N>{s + i * PenCfg<N>::tile}, d[i], tw, tid);
  }
}

// Configuration of the passes that hold NT tiles
template <int N, int NT>
struct MultiCfg {
  using C = PenCfg<N>;
  static constexpr int smem = NT * C::tile * 8;
  static constexpr int regs = C::ept == 16 ? 80 : 64;
  static constexpr int minb = imax(1, imin(imin(imax(1, imin(2048, 65536 / regs) / C::T), 16), (224 * 1024) / (smem + 1024)));
};

// Forward x pass, times g_scale / |m|^2 (H(k), the common factor of the force components
// F_j = i D(k_j) H), inverse x transforms of F_x into out_f and of H into out_h (F_y and F_z are i D H
// with D constant along x: the y pass makes both from H).  out_h may be in.  spec_out (or null)
// receives the forward spectrum.
template <int N>
__global__ void __launch_bounds__(PenCfg<N>::T, MultiCfg<N, 2>::minb) k_green(const float2* in, float2* out_f, float2* out_h,
                                                                           const float* __restrict__ dtab, float g_scale,
                                                                           const float2* __restrict__ twf,
                                                                           const float2* __restrict__ twr,
                                                                           float2* spec_out) {
  extern __shared__ float2 sm[];
  using C = PenCfg<N>;
  constexpr int T = C::T, M = PlanOf<N, false>::m;
  constexpr long long JS = (long long)N * C::PC;
  const int tid = threadIdx.x, col = blockIdx.x * PenCfg<N>::W + (tid & (PenCfg<N>::W - 1)), y = blockIdx.y;
  const bool ok = col < C::NC;
  const long long off = (long long)y * C::PC + col;
  float2* a = sm;
  float2* b = sm + C::tile;
  pen_stage<N, false, 0, -1, T>(ColG<JS>{const_cast<float2*>(in) + off, ok}, TileW<N>{a}, twf, tid);
  __syncthreads();
  const float2* cur = pen_middle<N, false, -1, T, true>(a, b, twf, tid);
  using L = Group<N, false, M - 1, -1>;
  using F = Group<N, true, 0, +1>;
  static_assert(L::R == F::R && L::NS == L::NB && F::NS == 1, "the inverse starts from the forward's registers");
  constexpr int TOT = L::NB << PenCfg<N>::lw, IT = (TOT + T - 1) / T;
  float2 spec[IT][L::R];
  const int my = y < N / 2 ? y : y - N;
#pragma unroll
  for (int it = 0; it < IT; ++it) {
    const int idx = tid + it * T;
    if (TOT % T == 0 || idx < TOT) {
      const int bb = idx >> PenCfg<N>::lw;
#pragma unroll
      for (int r = 0; r < L::R; ++r) spec[it][r] = cur[idx + r * (L::NB << PenCfg<N>::lw)];
      L::run(spec[it], twf, bb);
      if (spec_out && ok) {
#pragma unroll
        for (int r = 0; r < L::R; ++r) spec_out[off + (bb + r * L::NS) * JS] = spec[it][r];
      }
      const int myz = my * my + col * col;
#pragma unroll
      for (int r = 0; r < L::R; ++r) {
        const int j = bb + r * L::NS;
        const int mx = j < N / 2 ? j : j - N;
        const int m2 = mx * mx + myz;
        spec[it][r] = (m2 > 0 ? g_scale / (float)m2 : 0.0f) * spec[it][r];
      }
    }
  }
  __syncthreads();   // the forward's buffers are free
#pragma unroll
  for (int it = 0; it < IT; ++it) {
    const int idx = tid + it * T;
    if (TOT % T == 0 || idx < TOT) {
      const int w = idx & (PenCfg<N>::W - 1), bb = idx >> PenCfg<N>::lw;
      float2 v[L::R];
#pragma unroll
      for (int r = 0; r < L::R; ++r) {
        const float d = __ldg(dtab + bb + r * L::NS);
        v[r] = make_float2(-d * spec[it][r].y, d * spec[it][r].x);   // i D H
      }
      F::run(v, twr, 0);
#pragma unroll
      for (int r = 0; r < L::R; ++r) a[((bb * L::R + r) << PenCfg<N>::lw) + w] = v[r];
      F::run(spec[it], twr, 0);
#pragma unroll
      for (int r = 0; r < L::R; ++r) b[((bb * L::R + r) << PenCfg<N>::lw) + w] = spec[it][r];
    }
  }
  __syncthreads();
  const ColG<JS> d[2] = {{out_f + off, ok}, {out_h + off, ok}};
  multi_finish<N, true, +1, T, 1>(sm, d, twr, tid);
}

// Inverse y pass of H into the y and z components: i D(k_y) H to out_y and i D(k_z) H to out_z (which
// may be h: a tile is read whole before it is written)
template <int N>
__global__ void __launch_bounds__(PenCfg<N>::T, MultiCfg<N, 2>::minb) k_pen_yz(const float2* h, float2* out_y, float2* out_z,
                                                                            const float* __restrict__ dtab,
                                                                            const float2* __restrict__ tw) {
  extern __shared__ float2 sm[];
  using C = PenCfg<N>;
  constexpr int T = C::T;
  constexpr long long JS = C::PC, OS = (long long)N * C::PC;
  const int tid = threadIdx.x, col = blockIdx.x * PenCfg<N>::W + (tid & (PenCfg<N>::W - 1));
  const bool ok = col < C::NC;
  const long long off = blockIdx.y * OS + col;
  float2* a = sm;
  float2* b = sm + C::tile;
  const ColG<JS> src{const_cast<float2*>(h) + off, ok};
  const float dz = ok ? __ldg(dtab + col) : 0.0f;
  using Q = Group<N, false, 0, +1>;
  constexpr int TOT = Q::NB << PenCfg<N>::lw, IT = (TOT + T - 1) / T;
#pragma unroll(IT <= 2 ? IT : 1)
  for (int it = 0; it < IT; ++it) {
    const int idx = tid + it * T;
    if (TOT % T == 0 || idx < TOT) {
      const int w = idx & (PenCfg<N>::W - 1), bb = idx >> PenCfg<N>::lw;
      float2 z[Q::R], v[Q::R];
#pragma unroll
      for (int r = 0; r < Q::R; ++r) z[r] = src(bb + r * Q::NB, w);
#pragma unroll
      for (int r = 0; r < Q::R; ++r) {
        const float d = __ldg(dtab + bb + r * Q::NB);
        v[r] = make_float2(-d * z[r].y, d * z[r].x);
      }
      Q::run(v, tw, 0);
#pragma unroll
      for (int r = 0; r < Q::R; ++r) a[((bb * Q::R + r) << PenCfg<N>::lw) + w] = v[r];
#pragma unroll
      for (int r = 0; r < Q::R; ++r) z[r] = make_float2(-dz * z[r].y, dz * z[r].x);
      Q::run(z, tw, 0);
#pragma unroll
      for (int r = 0; r < Q::R; ++r) b[((bb * Q::R + r) << PenCfg<N>::lw) + w] = z[r];
    }
  }
  __syncthreads();
  const ColG<JS> d[2] = {{out_y + off, ok}, {out_z + off, ok}};
  multi_finish<N, false, +1, T, 1>(sm, d, tw, tid);
}

// ---- 2LPT (x and y passes) ----------------------------------------------------------------------
// The 2LPT fields are delta_L(k) / k^2 times products of at most two wave numbers.  A wave number of an
// axis is constant along the other axes' pencils, so one forward x pass makes the inverse x transforms of
// delta/k^2 times 1, k_x and k_x^2, and each y pass those times 1, k_y and k_y^2 as far as they are
// needed; k_z waits for the row pass.  3 x and 6 y transforms then serve the nine first-order fields,
// where a transform of its own for each takes nine and nine (and a multiply each).  The factor of a single
// derivative is 0 on its Nyquist plane, a square keeps it; factors i are left to the row pass.
// With the row passes below (Hessians and source on chip, first positions written with Psi2) a call is 12
// launches and moves 52 field-sized reads and writes where 45 launches moved 120: 256^3 lattice 1706 -> 917
// us (0.51 ms for the 52 at the copy rate), 32^3 271 -> 82 us.

// z times k^p, p = 0, 1, 2, k = 2 pi m / n of storage index j
template <int N, int PW>
__device__ __forceinline__ float2 times_k(float2 z, int j) {
  constexpr float kf = 6.283185307179586f / N;
  const int m = j < N / 2 ? j : j - N;
  if constexpr (PW == 0) return z;
  else if constexpr (PW == 1) return (2 * j == N ? 0.0f : m * kf) * z;
  else return (m * kf) * (m * kf) * z;
}
// first group of the inverse transforms of v times 1, k, .., k^(NT-1) into the tiles s, s + tile, ..
template <int N, bool REV, int NT, int PW = 0, int R>
__device__ __forceinline__ void powers_stage(const float2 (&z)[R], int b, int w, float2* s, const float2* __restrict__ tw) {
  if constexpr (PW < NT) {
    using Q = Group<N, REV, 0, +1>;
    static_assert(Q::R == R, "a first group's butterfly");
    float2 v[R];
#pragma unroll
    for (int r = 0; r < R; ++r) v[r] = times_k<N, PW>(z[r], b + r * Q::NB);
    Q::run(v, tw, 0);
#pragma unroll
    for (int r = 0; r < R; ++r) s[PW * PenCfg<N>::tile + ((b * R + r) << PenCfg<N>::lw) + w] = v[r];
    powers_stage<N, REV, NT, PW + 1>(z, b, w, s, tw);
  }
}

// Forward x transform of in, times scale / k^2 (and the amplitude amp_m2[|m|^2] when AMP), and the inverse
// x transforms of that times 1, k_x, .. (NT of them) into out.p[0..NT-1]; out.p[0] may be in.
template <int N, int NT, bool AMP>
__global__ void __launch_bounds__(PenCfg<N>::T, MultiCfg<N, NT>::minb) k_ic_x(const float2* in, Ptr3 out, float scale,
                                                                              const float* __restrict__ amp_m2,
                                                                              const float2* __restrict__ twf,
                                                                              const float2* __restrict__ twr) {
  extern __shared__ float2 sm[];
  using C = PenCfg<N>;
  constexpr int T = C::T, M = PlanOf<N, false>::m;
  constexpr long long JS = (long long)N * C::PC;
  const int tid = threadIdx.x, col = blockIdx.x * C::W + (tid & (C::W - 1)), y = blockIdx.y;
  const bool ok = col < C::NC;
  const long long off = (long long)y * C::PC + col;
  pen_stage<N, false, 0, -1, T>(ColG<JS>{const_cast<float2*>(in) + off, ok}, TileW<N>{sm}, twf, tid);
  __syncthreads();
  const float2* cur = pen_middle<N, false, -1, T, true>(sm, sm + C::tile, twf, tid);
  using L = Group<N, false, M - 1, -1>;
  constexpr int TOT = L::NB << C::lw, IT = (TOT + T - 1) / T;
  constexpr float kf = 6.283185307179586f / N;
  float2 spec[IT][L::R];
  const int my = y < N / 2 ? y : y - N;
#pragma unroll
  for (int it = 0; it < IT; ++it) {
    const int idx = tid + it * T;
    if (TOT % T == 0 || idx < TOT) {
      const int bb = idx >> C::lw;
#pragma unroll
      for (int r = 0; r < L::R; ++r) spec[it][r] = cur[idx + r * (L::NB << C::lw)];
      L::run(spec[it], twf, bb);
      const int myz = my * my + col * col;
#pragma unroll
      for (int r = 0; r < L::R; ++r) {
        const int j = bb + r * L::NS;
        const int mx = j < N / 2 ? j : j - N;
        const int m2 = mx * mx + myz;
        float g = m2 > 0 ? scale / ((float)m2 * kf * kf) : 0.0f;
        if (AMP && ok) g *= __ldg(amp_m2 + m2);
        spec[it][r] = g * spec[it][r];
      }
    }
  }
  __syncthreads();   // the forward's buffers are free
#pragma unroll
  for (int it = 0; it < IT; ++it) {
    const int idx = tid + it * T;
    if (TOT % T == 0 || idx < TOT) powers_stage<N, true, NT>(spec[it], idx >> C::lw, idx & (C::W - 1), sm, twr);
  }
  __syncthreads();
  ColG<JS> d[NT];
#pragma unroll
  for (int i = 0; i < NT; ++i) d[i] = ColG<JS>{out.p[i] + off, ok};
  multi_finish<N, true, +1, T, 1>(sm, d, twr, tid);
}

struct Pow3 {
  int p[3];   // powers 0, 1, 2
};
// column store times a factor
template <long long JS>
struct ColScaled {
  ColG<JS> g;
  float f;
  __device__ __forceinline__ void operator()(int j, int w, float2 v) const { g(j, w, f * v); }
};

// Inverse y transforms of in times 1, k_y, .. (NT of them), times k_z^zp.p[i], into out.p[0..NT-1];
// out.p[0] may be in.
template <int N, int NT>
__global__ void __launch_bounds__(PenCfg<N>::T, MultiCfg<N, NT>::minb) k_ic_y(const float2* in, Ptr3 out, Pow3 zp,
                                                                              const float2* __restrict__ tw) {
  extern __shared__ float2 sm[];
  using C = PenCfg<N>;
  using Q = Group<N, false, 0, +1>;
  constexpr int T = C::T;
  constexpr long long JS = C::PC, OS = (long long)N * C::PC;
  const int tid = threadIdx.x, col = blockIdx.x * C::W + (tid & (C::W - 1));
  const bool ok = col < C::NC;
  const long long off = blockIdx.y * OS + col;
  const ColG<JS> src{const_cast<float2*>(in) + off, ok};
  constexpr int TOT = Q::NB << C::lw, IT = (TOT + T - 1) / T;
#pragma unroll(IT <= 2 ? IT : 1)
  for (int it = 0; it < IT; ++it) {
    const int idx = tid + it * T;
    if (TOT % T == 0 || idx < TOT) {
      const int w = idx & (C::W - 1), bb = idx >> C::lw;
      float2 z[Q::R];
#pragma unroll
      for (int r = 0; r < Q::R; ++r) z[r] = src(bb + r * Q::NB, w);
      powers_stage<N, false, NT>(z, bb, w, sm, tw);
    }
  }
  __syncthreads();
  constexpr float kf = 6.283185307179586f / N;
  const float kz = col * kf, kz_odd = 2 * col == N ? 0.0f : kz;
  ColScaled<JS> d[NT];
#pragma unroll
  for (int i = 0; i < NT; ++i)
    d[i] = ColScaled<JS>{{out.p[i] + off, ok}, zp.p[i] == 0 ? 1.0f : (zp.p[i] == 1 ? kz_odd : kz * kz)};
  multi_finish<N, false, +1, T, 1>(sm, d, tw, tid);
}

// ---- transposed gradients (the adjoint's x passes) ------------------------------------------------
// NT forward transforms of the tiles s, s + tile, .. whose first groups are done, but for the last groups
template <int N, int T, int NT, int G = 1>
__device__ __forceinline__ void multi_forward(float2* s, const float2* __restrict__ tw, int tid) {
  if constexpr (G + 1 < PlanOf<N, false>::m) {
#pragma unroll
    for (int i = 0; i < NT; ++i) pen_inplace<N, false, G, -1, T>(s + i * PenCfg<N>::tile, tw, tid);
    __syncthreads();
    multi_forward<N, T, NT, G + 1>(s, tw, tid);
  }
}

// The inverse x transform of -i g sum_j D(k_j) L_j(k), g = g_scale / |m|^2, of three spectra over k_y, k_z
// (x still in real space); out may be one of them.  D(k_y) and D(k_z) are constant along x, so two forward
// transforms serve the three components.
template <int N>
__global__ void __launch_bounds__(PenCfg<N>::T, MultiCfg<N, 2>::minb) k_grad_adj(const float2* l0, const float2* l1,
                                                                                 const float2* l2, float2* out,
                                                                                 const float* __restrict__ dtab, float g_scale,
                                                                                 const float2* __restrict__ twf,
                                                                                 const float2* __restrict__ twr) {
  extern __shared__ float2 sm[];
  using C = PenCfg<N>;
  using A = Group<N, false, 0, -1>;
  using L = Group<N, false, PlanOf<N, false>::m - 1, -1>;
  using F = Group<N, true, 0, +1>;
  constexpr int T = C::T;
  constexpr long long JS = (long long)N * C::PC;
  const int tid = threadIdx.x, col = blockIdx.x * C::W + (tid & (C::W - 1)), y = blockIdx.y;
  const bool ok = col < C::NC;
  const long long off = (long long)y * C::PC + col;
  const float dy = __ldg(dtab + y), dz = ok ? __ldg(dtab + col) : 0.0f;
  {
    constexpr int TOT = A::NB << C::lw, IT = (TOT + T - 1) / T;
#pragma unroll(IT <= 2 ? IT : 1)
    for (int it = 0; it < IT; ++it) {
      const int idx = tid + it * T;
      if (TOT % T == 0 || idx < TOT) {
        const int w = idx & (C::W - 1), bb = idx >> C::lw;
        float2 v[A::R], u[A::R];
#pragma unroll
        for (int r = 0; r < A::R; ++r) {
          const long long e = off + (bb + r * A::NB) * JS;
          v[r] = u[r] = make_float2(0.f, 0.f);
          if (ok) {
            v[r] = l0[e];
            u[r] = dy * l1[e] + dz * l2[e];
          }
        }
        A::run(v, twf, 0);
        A::run(u, twf, 0);
#pragma unroll
        for (int r = 0; r < A::R; ++r) {
          sm[((bb * A::R + r) << C::lw) + w] = v[r];
          sm[C::tile + ((bb * A::R + r) << C::lw) + w] = u[r];
        }
      }
    }
  }
  __syncthreads();
  multi_forward<N, T, 2>(sm, twf, tid);
  constexpr int TOT = L::NB << C::lw, IT = (TOT + T - 1) / T;
  float2 spec[IT][L::R];
  const int my = y < N / 2 ? y : y - N;
#pragma unroll
  for (int it = 0; it < IT; ++it) {
    const int idx = tid + it * T;
    if (TOT % T == 0 || idx < TOT) {
      const int bb = idx >> C::lw;
      float2 v[L::R], u[L::R];
#pragma unroll
      for (int r = 0; r < L::R; ++r) {
        v[r] = sm[idx + r * (L::NB << C::lw)];
        u[r] = sm[C::tile + idx + r * (L::NB << C::lw)];
      }
      L::run(v, twf, bb);
      L::run(u, twf, bb);
      const int myz = my * my + col * col;
#pragma unroll
      for (int r = 0; r < L::R; ++r) {
        const int j = bb + r * L::NS, mx = j < N / 2 ? j : j - N, m2 = mx * mx + myz;
        const float g = m2 > 0 ? g_scale / (float)m2 : 0.0f, dx = __ldg(dtab + j);
        const float2 z = dx * v[r] + u[r];
        spec[it][r] = make_float2(g * z.y, -g * z.x);
      }
    }
  }
  __syncthreads();   // the forward's tiles are free
#pragma unroll
  for (int it = 0; it < IT; ++it) {
    const int idx = tid + it * T;
    if (TOT % T == 0 || idx < TOT) {
      const int w = idx & (C::W - 1), bb = idx >> C::lw;
      F::run(spec[it], twr, 0);
#pragma unroll
      for (int r = 0; r < L::R; ++r) sm[((bb * L::R + r) << C::lw) + w] = spec[it][r];
    }
  }
  __syncthreads();
  const ColG<JS> d[1] = {{out + off, ok}};
  multi_finish<N, true, +1, T, 1>(sm, d, twr, tid);
}

// Transpose of the first-order 2LPT maps: the inverse x transform of
//   amp(|m|^2) / k^2 [ sum_ij k_i k_j h_ij - i r sum_j k_j p_j ]
// of the six Hessian cotangents h (xx, yy, zz, xy, xz, yz) and the three displacement cotangents p, all
// spectra over k_y, k_z with x in real space; out may be one of them.  Powers of k_y and k_z are constant
// along x: three forward transforms, of the factors of 1, k_x and k_x^2, serve all nine.
struct Lpt9 {
  const float2* h[6];
  const float2* p[3];
};
template <int N>
__global__ void __launch_bounds__(PenCfg<N>::T, MultiCfg<N, 3>::minb) k_lpt_adj(Lpt9 in, float2* out, float r_scale,
                                                                               const float* __restrict__ amp_m2,
                                                                               const float2* __restrict__ twf,
                                                                               const float2* __restrict__ twr) {
  extern __shared__ float2 sm[];
  using C = PenCfg<N>;
  using A = Group<N, false, 0, -1>;
  using L = Group<N, false, PlanOf<N, false>::m - 1, -1>;
  using F = Group<N, true, 0, +1>;
  constexpr int T = C::T;
  constexpr long long JS = (long long)N * C::PC;
  constexpr float kf = 6.283185307179586f / N;
  const int tid = threadIdx.x, col = blockIdx.x * C::W + (tid & (C::W - 1)), y = blockIdx.y;
  const bool ok = col < C::NC;
  const long long off = (long long)y * C::PC + col;
  const int my = y < N / 2 ? y : y - N;
  const float ky = my * kf, kz = col * kf, oy = 2 * y == N ? 0.0f : ky, oz = 2 * col == N ? 0.0f : kz;
  {
    constexpr int TOT = A::NB << C::lw, IT = (TOT + T - 1) / T;
#pragma unroll 1
    for (int it = 0; it < IT; ++it) {
      const int idx = tid + it * T;
      if (TOT % T == 0 || idx < TOT) {
        const int w = idx & (C::W - 1), bb = idx >> C::lw;
#pragma unroll
        for (int q = 0; q < 3; ++q) {   // factors of 1, k_x, k_x^2
          float2 v[A::R];
#pragma unroll
          for (int r = 0; r < A::R; ++r) {
            const long long e = off + (bb + r * A::NB) * JS;
            v[r] = make_float2(0.f, 0.f);
            if (ok) {
              if (q == 0) {
                const float2 g = r_scale * (oy * in.p[1][e] + oz * in.p[2][e]);
                v[r] = (ky * ky) * in.h[1][e] + (kz * kz) * in.h[2][e] + (oy * oz) * in.h[5][e] + make_float2(g.y, -g.x);
              } else if (q == 1) {
                const float2 g = r_scale * in.p[0][e];
                v[r] = oy * in.h[3][e] + oz * in.h[4][e] + make_float2(g.y, -g.x);
              } else {
                v[r] = in.h[0][e];
              }
            }
          }
          A::run(v, twf, 0);
#pragma unroll
          for (int r = 0; r < A::R; ++r) sm[q * C::tile + ((bb * A::R + r) << C::lw) + w] = v[r];
        }
      }
    }
  }
  __syncthreads();
  multi_forward<N, T, 3>(sm, twf, tid);
  constexpr int TOT = L::NB << C::lw, IT = (TOT + T - 1) / T;
  float2 spec[IT][L::R];
#pragma unroll
  for (int it = 0; it < IT; ++it) {
    const int idx = tid + it * T;
    if (TOT % T == 0 || idx < TOT) {
      const int bb = idx >> C::lw;
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        float2 v[L::R];
#pragma unroll
        for (int r = 0; r < L::R; ++r) v[r] = sm[q * C::tile + idx + r * (L::NB << C::lw)];
        L::run(v, twf, bb);
#pragma unroll
        for (int r = 0; r < L::R; ++r) {
          const int j = bb + r * L::NS, mx = j < N / 2 ? j : j - N;
          const float kx = mx * kf;
          const float f = q == 0 ? 1.0f : (q == 1 ? (2 * j == N ? 0.0f : kx) : kx * kx);
          spec[it][r] = q == 0 ? v[r] : spec[it][r] + f * v[r];
        }
      }
      const int myz = my * my + col * col;
#pragma unroll
      for (int r = 0; r < L::R; ++r) {
        const int j = bb + r * L::NS, mx = j < N / 2 ? j : j - N, m2 = mx * mx + myz;
        const float g = m2 > 0 && ok ? __ldg(amp_m2 + m2) / ((float)m2 * kf * kf) : 0.0f;
        spec[it][r] = g * spec[it][r];
      }
    }
  }
  __syncthreads();   // the forward's tiles are free
#pragma unroll
  for (int it = 0; it < IT; ++it) {
    const int idx = tid + it * T;
    if (TOT % T == 0 || idx < TOT) {
      const int w = idx & (C::W - 1), bb = idx >> C::lw;
      F::run(spec[it], twr, 0);
#pragma unroll
      for (int r = 0; r < L::R; ++r) sm[((bb * L::R + r) << C::lw) + w] = spec[it][r];
    }
  }
  __syncthreads();
  const ColG<JS> d[1] = {{out + off, ok}};
  multi_finish<N, true, +1, T, 1>(sm, d, twr, tid);
}

// ---- row pairs (the contiguous axis) -------------------------------------------------------------
// P row pairs per CTA, element j of pair p at p RS + j + j/16: the skew spreads a first group's strided
// stores over the banks.
template <int N>
struct RowCfg {
  static constexpr Groups P = make_groups(N, false);
  static constexpr int ept = P.max_radix > 10 ? 16 : 8;
  static constexpr int pairs_total = N * N / 2;
  // about 256 threads per CTA, and at least two CTAs per SM on small meshes
  static constexpr int pairs = imax(1, imin(256 * ept / N, pairs_total / 304));
  static constexpr int T = imin(1024, round_up((pairs * N + ept - 1) / ept, 32));
  static constexpr int PC = ((N / 2 + 1) + 1) & ~1;
  static constexpr int RS = N + N / 16 + 1;
  static constexpr int buf = pairs * RS;
  static constexpr int regs = ept == 16 ? 64 : 40;
  static constexpr int by_regs = imax(1, imin(2048, 65536 / regs) / T);
  static constexpr int minb(int bufs) { return imax(1, imin(imin(by_regs, 24), (224 * 1024) / (bufs * buf * 8 + 1024))); }
};
__device__ __forceinline__ int rpos(int j) { return j + (j >> 4); }

template <int N>
struct RowSm {
  float2* s;
  // rows j0 + r STEP of pair p; BLOCK: j0 .. lie in one aligned block of 16
  template <int STEP, bool BLOCK, int R>
  __device__ __forceinline__ void load(int p, int j0, float2 (&v)[R]) const {
    if constexpr (STEP % 16 == 0 || BLOCK) {
      constexpr int st = STEP % 16 == 0 ? STEP + STEP / 16 : STEP;
      const float2* q = s + p * RowCfg<N>::RS + rpos(j0);
#pragma unroll
      for (int r = 0; r < R; ++r) v[r] = q[r * st];
    } else {
#pragma unroll
      for (int r = 0; r < R; ++r) v[r] = s[p * RowCfg<N>::RS + rpos(j0 + r * STEP)];
    }
  }
  template <int STEP, bool BLOCK, int R>
  __device__ __forceinline__ void store(int p, int j0, const float2 (&v)[R]) const {
    if constexpr (STEP % 16 == 0 || BLOCK) {
      constexpr int st = STEP % 16 == 0 ? STEP + STEP / 16 : STEP;
      float2* q = s + p * RowCfg<N>::RS + rpos(j0);
#pragma unroll
      for (int r = 0; r < R; ++r) q[r * st] = v[r];
    } else {
#pragma unroll
      for (int r = 0; r < R; ++r) s[p * RowCfg<N>::RS + rpos(j0 + r * STEP)] = v[r];
    }
  }
};

template <int N, int G, int DIR, class Src, class Dst>
__device__ __forceinline__ void row_stage(const Src& src, const Dst& dst, const float2* __restrict__ tw, int tid) {
  using Q = Group<N, false, G, DIR>;
  using C = RowCfg<N>;
  constexpr int TOT = C::pairs * Q::NB, IT = (TOT + C::T - 1) / C::T;
#pragma unroll(IT <= 2 ? IT : 1)
  for (int it = 0; it < IT; ++it) {
    const int idx = tid + it * C::T;
    if (TOT % C::T == 0 || idx < TOT) {
      const int p = idx / Q::NB, b = idx - p * Q::NB, k = Q::k_of(b);
      float2 v[Q::R];
      src.template load<Q::NB, false>(p, b, v);
      Q::run(v, tw, k);
      dst.template store<Q::NS, (16 % (Q::NS * Q::R) == 0)>(p, Q::out_row(b, k), v);
    }
  }
}
template <int N, int DIR, int G = 1>
__device__ __forceinline__ float2* row_middle(float2* a, float2* b, const float2* __restrict__ tw, int tid) {
  if constexpr (G + 1 < PlanOf<N, false>::m) {
    row_stage<N, G, DIR>(RowSm<N>{a}, RowSm<N>{b}, tw, tid);
    __syncthreads();
    return row_middle<N, DIR, G + 1>(b, a, tw, tid);
  } else {
    return a;
  }
}

// complex (row 2p, row 2p + 1) of real rows: floats times scale, or fixed-point cells as density contrast
template <int SRC>
struct RowPairLoad {
  const void* src;
  long long rs, pair0, npairs;
  float scale;
  mutable unsigned long long mlo = 0, mhi = 0;   // 128-bit sum of the fixed-point values read
  template <int STEP, bool, int R>
  __device__ __forceinline__ void load(int p, int j0, float2 (&v)[R]) const {
    const long long row = 2 * (pair0 + p);
    const bool ok = pair0 + p < npairs;
    if constexpr (SRC == kSrcFixedPoint) {
      const unsigned long long* a = static_cast<const unsigned long long*>(src) + row * rs + j0;
#pragma unroll
      for (int r = 0; r < R; ++r) {
        v[r] = make_float2(0.f, 0.f);
        if (ok) {
          const unsigned long long va = a[r * STEP], vb = a[rs + r * STEP];
          v[r] = make_float2(fixed_to_delta(va, scale), fixed_to_delta(vb, scale));
          mlo += va;
          mhi += (mlo < va);
          mlo += vb;
          mhi += (mlo < vb);
        }
      }
    } else {
      const float* a = static_cast<const float*>(src) + row * rs + j0;
#pragma unroll
      for (int r = 0; r < R; ++r) v[r] = ok ? make_float2(a[r * STEP] * scale, a[rs + r * STEP] * scale) : make_float2(0.f, 0.f);
    }
  }
};

// half rows of the two real rows that a transformed complex row holds
template <int N>
__device__ __forceinline__ void untangle_rows(const float2* res, float2* dst, long long pair0, long long npairs, int tid) {
  using C = RowCfg<N>;
  constexpr int NH = N / 2, TOT = C::pairs * (NH + 1);
  for (int idx = tid; idx < TOT; idx += C::T) {
    const int p = idx / (NH + 1), k = idx - p * (NH + 1);
    if (pair0 + p >= npairs) break;
    const float2 zk = res[p * C::RS + rpos(k)];
    const float2 zn = res[p * C::RS + rpos(k == 0 ? 0 : N - k)];
    float2* o = dst + 2 * (pair0 + p) * C::PC + k;
    o[0] = make_float2(0.5f * (zk.x + zn.x), 0.5f * (zk.y - zn.y));
    o[C::PC] = make_float2(0.5f * (zk.y + zn.y), -0.5f * (zk.x - zn.x));
  }
}

template <int N>
struct R2cCfg {
  static constexpr int bufs = 2;
  static constexpr int smem = bufs * RowCfg<N>::buf * 8;
};

// Forward R2C of the row pairs (in place when src is dst's own rows: a CTA reads its rows whole first)
// of the fields src.p[blockIdx.y] into dst.p[blockIdx.y]
template <int N, int SRC>
__global__ void __launch_bounds__(RowCfg<N>::T, RowCfg<N>::minb(2)) k_r2c(Src3 src, long long rs, float scale,
                                                                          Ptr3 dst, long long npairs,
                                                                          const float2* __restrict__ tw,
                                                                          unsigned long long* mass_acc) {
  extern __shared__ float2 sm[];
  using C = RowCfg<N>;
  const int tid = threadIdx.x;
  const long long pair0 = (long long)blockIdx.x * C::pairs;
  const RowPairLoad<SRC> g{src.p[blockIdx.y], rs, pair0, npairs, scale};
  float2* a = sm;
  float2* b = sm + C::buf;
  row_stage<N, 0, -1>(g, RowSm<N>{a}, tw, tid);
  if (SRC == kSrcFixedPoint && mass_acc) mass_accumulate(g.mlo, g.mhi, mass_slot(mass_acc));
  __syncthreads();
  float2* cur = row_middle<N, -1>(a, b, tw, tid);
  float2* res = cur == a ? b : a;
  row_stage<N, PlanOf<N, false>::m - 1, -1>(RowSm<N>{cur}, RowSm<N>{res}, tw, tid);
  __syncthreads();
  untangle_rows<N>(res, dst.p[blockIdx.y], pair0, npairs, tid);
}

// C[k] = A[k] + i B[k] of two Hermitian half rows
template <int N>
struct HalfPairLoad {
  const float2* data;
  long long pair0, npairs;
  template <int STEP, bool, int R>
  __device__ __forceinline__ void load(int p, int j0, float2 (&v)[R]) const {
    constexpr int PC = RowCfg<N>::PC, NH = N / 2;
    const float2* row = data + 2 * (pair0 + p) * PC;
    const bool ok = pair0 + p < npairs;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int k = j0 + r * STEP, kk = k <= NH ? k : N - k;
      float2 A = make_float2(0.f, 0.f), B = make_float2(0.f, 0.f);
      if (ok) {
        A = row[kk];
        B = row[PC + kk];
      }
      if (kk == 0 || kk == NH) {
        A.y = 0.f;
        B.y = 0.f;
      }
      v[r] = k <= NH ? make_float2(A.x - B.y, A.y + B.x) : make_float2(A.x + B.y, B.x - A.y);
    }
  }
};
// (re, im) to real rows 2p, 2p + 1 of stride rs; DENSE: times scale
template <int N, bool DENSE>
struct RealPairStore {
  float* out;
  long long rs, pair0, npairs;
  float scale;
  template <int STEP, bool, int R>
  __device__ __forceinline__ void store(int p, int j0, const float2 (&v)[R]) const {
    if (pair0 + p >= npairs) return;
    float* o = out + 2 * (pair0 + p) * rs + j0;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      o[r * STEP] = DENSE ? v[r].x * scale : v[r].x;
      o[rs + r * STEP] = DENSE ? v[r].y * scale : v[r].y;
    }
  }
};
template <int N>
struct C2rCfg {
  static constexpr int bufs = make_groups(N, false).m > 2 ? 2 : 1;
  static constexpr int smem = bufs * RowCfg<N>::buf * 8;
};

// Inverse C2R of the row pairs: in place (real rows of 2 PC floats) of the fields data.p[blockIdx.y], or,
// DENSE, into out as dense rows of N floats times scale
template <int N, bool DENSE>
__global__ void __launch_bounds__(RowCfg<N>::T, RowCfg<N>::minb(C2rCfg<N>::bufs)) k_c2r(Ptr3 data, long long npairs,
                                                                                       const float2* __restrict__ tw,
                                                                                       float* out, float scale) {
  extern __shared__ float2 sm[];
  using C = RowCfg<N>;
  const int tid = threadIdx.x;
  const long long pair0 = (long long)blockIdx.x * C::pairs;
  float2* d = data.p[blockIdx.y];
  row_stage<N, 0, +1>(HalfPairLoad<N>{d, pair0, npairs}, RowSm<N>{sm}, tw, tid);
  __syncthreads();
  float2* cur = row_middle<N, +1>(sm, sm + C::buf, tw, tid);
  const RealPairStore<N, DENSE> o{DENSE ? out : reinterpret_cast<float*>(d), DENSE ? (long long)N : 2LL * C::PC, pair0,
                                  npairs, scale};
  row_stage<N, PlanOf<N, false>::m - 1, +1>(RowSm<N>{cur}, o, tw, tid);
}

// ---- 2LPT (row passes) ----------------------------------------------------------------------------
// A Hermitian half row's entry kk times the factor of MODE: k^p (p = MODE & 3, as times_k) and i (MODE & 4).
template <int N, int MODE>
__device__ __forceinline__ float2 ic_entry(float2 z, int kk) {
  z = times_k<N, MODE & 3>(z, kk);
  return (MODE & 4) ? make_float2(-z.y, z.x) : z;
}
// Rows A and B (as complex rows A + i B after the transform) of two half rows per pair slot, with factors
template <int N, int MA, int MB>
struct FieldPairLoad {
  const float2* a;   // row of slot 0
  const float2* b;
  long long stride;  // entries between slots' rows
  int slots;         // valid slots
  template <int STEP, bool, int R>
  __device__ __forceinline__ void load(int p, int j0, float2 (&v)[R]) const {
    constexpr int NH = N / 2;
    const float2* ra = a + p * stride;
    const float2* rb = b + p * stride;
    const bool ok = p < slots;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int k = j0 + r * STEP, kk = k <= NH ? k : N - k;
      float2 A = make_float2(0.f, 0.f), B = make_float2(0.f, 0.f);
      if (ok) {
        A = ic_entry<N, MA>(ra[kk], kk);
        B = ic_entry<N, MB>(rb[kk], kk);
      }
      if (kk == 0 || kk == NH) {
        A.y = 0.f;
        B.y = 0.f;
      }
      v[r] = k <= NH ? make_float2(A.x - B.y, A.y + B.x) : make_float2(A.x + B.y, B.x - A.y);
    }
  }
};

template <int N>
struct IcRowCfg {
  using C = RowCfg<N>;
  static constexpr int smem = 3 * C::buf * 8;
  static constexpr int regs = C::ept == 16 ? 128 : 96;
  static constexpr int minb = imax(1, imin(imin(imax(1, imin(2048, 65536 / regs) / C::T), 16), (224 * 1024) / (smem + 1024)));
};

// all groups but the last of the inverse transform of src; returns the buffer the last group reads
template <int N, class Src>
__device__ __forceinline__ const float2* ic_row_inverse(const Src& src, float2* a, float2* b, const float2* __restrict__ tw,
                                                        int tid) {
  __syncthreads();   // the buffers' last readers are done
  row_stage<N, 0, +1>(src, RowSm<N>{a}, tw, tid);
  __syncthreads();
  return row_middle<N, +1>(a, b, tw, tid);
}
// the last group of the rows in buf, each butterfly's values (at positions b + r NS of slot p) to f(it, p, b, v)
template <int N, class F>
__device__ __forceinline__ void ic_row_last(const float2* buf, const float2* __restrict__ tw, int tid, F&& f) {
  using Q = Group<N, false, PlanOf<N, false>::m - 1, +1>;
  using C = RowCfg<N>;
  constexpr int TOT = C::pairs * Q::NB, IT = (TOT + C::T - 1) / C::T;
#pragma unroll
  for (int it = 0; it < IT; ++it) {
    const int idx = tid + it * C::T;
    if (TOT % C::T == 0 || idx < TOT) {
      const int p = idx / Q::NB, b = idx - p * Q::NB;
      float2 v[Q::R];
      RowSm<N>{const_cast<float2*>(buf)}.template load<Q::NB, false>(p, b, v);
      Q::run(v, tw, b);
      f(it, p, b, v);
    }
  }
}

struct IcRows {
  const float2* t[6];   // spectra over k_z: 1, k_y, k_y^2 (of the x transform), k_x, k_x k_y, k_x^2
};

// The first-order fields of row pairs: Psi1 (dense rows times r_scale into psi1, component stride npart),
// the Hessians and from them the second-order source S = sum_{i<j} h_ii h_jj - h_ij^2, whose forward row
// transform goes to src_k.  The Hessians and the source stay on chip.  Two Hessians of one row make one
// complex transform, so that a thread meets both at the same site; Psi1_x and Psi1_y likewise, Psi1_z with
// the other row's.
template <int N>
__global__ void __launch_bounds__(RowCfg<N>::T, IcRowCfg<N>::minb) k_ic_z1(IcRows f, float2* src_k, float* psi1,
                                                                           long long npart, float r_scale, long long npairs,
                                                                           const float2* __restrict__ tw) {
  extern __shared__ float2 sm[];
  using C = RowCfg<N>;
  using Q = Group<N, false, PlanOf<N, false>::m - 1, +1>;
  constexpr int TOT = C::pairs * Q::NB, IT = (TOT + C::T - 1) / C::T, NS = Q::NS;
  const int tid = threadIdx.x;
  const long long pair0 = (long long)blockIdx.x * C::pairs;
  const int slots = npairs - pair0 < C::pairs ? (int)(npairs - pair0) : C::pairs;
  float2* a = sm;
  float2* b = sm + C::buf;
  float* src = reinterpret_cast<float*>(sm + 2 * C::buf);   // the source: (row 2p, row 2p + 1) of a site as one complex
#pragma unroll 1
  for (int row = 0; row < 2; ++row) {
    const long long o = (2 * pair0 + row) * C::PC, st = 2 * C::PC;
    float s[IT][Q::R], sum[IT][Q::R];
    ic_row_last<N>(ic_row_inverse<N>(FieldPairLoad<N, 0, 0>{f.t[5] + o, f.t[2] + o, st, slots}, a, b, tw, tid), tw, tid,
                   [&](int it, int, int, float2(&v)[Q::R]) {   // h00, h11
#pragma unroll
                     for (int r = 0; r < Q::R; ++r) {
                       s[it][r] = v[r].x * v[r].y;
                       sum[it][r] = v[r].x + v[r].y;
                     }
                   });
    ic_row_last<N>(ic_row_inverse<N>(FieldPairLoad<N, 2, 1>{f.t[0] + o, f.t[1] + o, st, slots}, a, b, tw, tid), tw, tid,
                   [&](int it, int, int, float2(&v)[Q::R]) {   // h22, h12
#pragma unroll
                     for (int r = 0; r < Q::R; ++r) s[it][r] += sum[it][r] * v[r].x - v[r].y * v[r].y;
                   });
    ic_row_last<N>(ic_row_inverse<N>(FieldPairLoad<N, 0, 1>{f.t[4] + o, f.t[3] + o, st, slots}, a, b, tw, tid), tw, tid,
                   [&](int it, int p, int bb, float2(&v)[Q::R]) {   // h01, h02
#pragma unroll
                     for (int r = 0; r < Q::R; ++r)
                       src[2 * (p * C::RS + rpos(bb + r * NS)) + row] = s[it][r] - v[r].x * v[r].x - v[r].y * v[r].y;
                   });
    ic_row_last<N>(ic_row_inverse<N>(FieldPairLoad<N, 4, 4>{f.t[3] + o, f.t[1] + o, st, slots}, a, b, tw, tid), tw, tid,
                   [&](int, int p, int bb, float2(&v)[Q::R]) {   // Psi1_x, Psi1_y
                     if (p >= slots) return;
                     float* q = psi1 + (2 * (pair0 + p) + row) * N + bb;
#pragma unroll
                     for (int r = 0; r < Q::R; ++r) {
                       q[r * NS] = v[r].x * r_scale;
                       q[npart + r * NS] = v[r].y * r_scale;
                     }
                   });
  }
  {
    const long long o = 2 * pair0 * C::PC;
    ic_row_last<N>(ic_row_inverse<N>(FieldPairLoad<N, 5, 5>{f.t[0] + o, f.t[0] + o + C::PC, 2 * C::PC, slots}, a, b, tw, tid),
                   tw, tid, [&](int, int p, int bb, float2(&v)[Q::R]) {   // Psi1_z of both rows
                     if (p >= slots) return;
                     float* q = psi1 + 2 * npart + 2 * (pair0 + p) * N + bb;
#pragma unroll
                     for (int r = 0; r < Q::R; ++r) {
                       q[r * NS] = v[r].x * r_scale;
                       q[N + r * NS] = v[r].y * r_scale;
                     }
                   });
  }
  __syncthreads();
  // the source's forward rows
  row_stage<N, 0, -1>(RowSm<N>{sm + 2 * C::buf}, RowSm<N>{a}, tw, tid);
  __syncthreads();
  float2* cur = row_middle<N, -1>(a, b, tw, tid);
  float2* res = cur == a ? b : a;
  row_stage<N, PlanOf<N, false>::m - 1, -1>(RowSm<N>{cur}, RowSm<N>{res}, tw, tid);
  __syncthreads();
  untangle_rows<N>(res, src_k, pair0, npairs, tid);
}

// Psi2 (component blockIdx.y, factors -i k_j) of row pairs into dense rows times r_scale, and the first
// positions s = d1 Psi1 + d2 Psi2 and velocities 0 of the same particles.
template <int N>
__global__ void __launch_bounds__(RowCfg<N>::T, RowCfg<N>::minb(C2rCfg<N>::bufs)) k_ic_z2(Ptr3 f, const float* __restrict__ psi1,
                                                                                         float* psi2, float* s, float* v0,
                                                                                         long long npart, float r_scale, float d1,
                                                                                         float d2, long long npairs,
                                                                                         const float2* __restrict__ tw) {
  extern __shared__ float2 sm[];
  using C = RowCfg<N>;
  using Q = Group<N, false, PlanOf<N, false>::m - 1, +1>;
  const int tid = threadIdx.x, comp = blockIdx.y;
  const long long pair0 = (long long)blockIdx.x * C::pairs;
  const int slots = npairs - pair0 < C::pairs ? (int)(npairs - pair0) : C::pairs;
  const float2* row = f.p[comp] + 2 * pair0 * C::PC;
  // i k_z for z, i for x and y (their k is in the spectrum); the sign of -i with the scale
  if (comp == 2) row_stage<N, 0, +1>(FieldPairLoad<N, 5, 5>{row, row + C::PC, 2 * C::PC, slots}, RowSm<N>{sm}, tw, tid);
  else row_stage<N, 0, +1>(FieldPairLoad<N, 4, 4>{row, row + C::PC, 2 * C::PC, slots}, RowSm<N>{sm}, tw, tid);
  __syncthreads();
  const float2* cur = row_middle<N, +1>(sm, sm + C::buf, tw, tid);
  ic_row_last<N>(cur, tw, tid, [&](int, int p, int bb, float2(&v)[Q::R]) {
    if (p >= slots) return;
    const long long o = comp * npart + 2 * (pair0 + p) * N + bb;
#pragma unroll
    for (int r = 0; r < Q::R; ++r) {
      const float p2[2] = {v[r].x * -r_scale, v[r].y * -r_scale};
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const long long i = o + h * N + r * Q::NS;
        psi2[i] = p2[h];
        s[i] = d1 * psi1[i] + d2 * p2[h];
        v0[i] = 0.0f;
      }
    }
  });
}

}  // namespace ct
}  // namespace cola
