// FFT pass kernels compiled for one length N each: radices, strides, tile shapes and twiddle offsets are
// compile-time constants, so a butterfly costs its arithmetic, its loads and stores with immediate
// offsets and one index computation.
//
// Every pass reads a tile of pencils from HBM once, runs the groups of the length's plan (fft_plan.h) on
// it through shared memory and writes it once; the first group loads straight from HBM and the last
// stores straight to it.  Strided passes (y, x) take tiles of 8 adjacent columns (64-byte row segments; 16
// from 144 to 320 points, 4 beyond 1536: PenCfg), lanes running over the columns first; the contiguous passes
// (z) take pairs of real rows as complex rows, lanes running along the row, so that their global accesses are
// whole 128-byte lines.
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
    run(reinterpret_cast<float2(&)[1][R]>(v), table, k);
  }
  // NV butterflies of the same index (adjacent columns)
  template <int NV>
  __device__ __forceinline__ static void run(float2 (&v)[NV][R], const float2* __restrict__ table, int k) {
    const float2* t1 = table + O1 + k;
    if constexpr (NS > 1) {
#pragma unroll
      for (int r = 1; r < R1; ++r) {
        const float2 t = tw(t1 + (r - 1) * NS);
#pragma unroll
        for (int c = 0; c < NV; ++c)
#pragma unroll
          for (int i = 0; i < R2; ++i) v[c][i + r * R2] = cmul(v[c][i + r * R2], t);
      }
    }
    if constexpr (R2 == 1) {
#pragma unroll
      for (int c = 0; c < NV; ++c) Dft<R1, DIR>::run(v[c]);
    } else {
      // stage r1 on the R2 sub-butterflies b + i N/R, then stage r2 on the R1 butterflies their
      // outputs r share
#pragma unroll
      for (int c = 0; c < NV; ++c)
#pragma unroll
        for (int i = 0; i < R2; ++i) {
          float2 t[R1];
#pragma unroll
          for (int r = 0; r < R1; ++r) t[r] = v[c][i + r * R2];
          Dft<R1, DIR>::run(t);
#pragma unroll
          for (int r = 0; r < R1; ++r) v[c][i + r * R2] = t[r];
        }
      const float2* t2 = table + O2 + k;
#pragma unroll
      for (int r = 0; r < R1; ++r)
#pragma unroll
        for (int i = 1; i < R2; ++i)
          if (NS > 1 || r > 0) {
            const float2 t = tw(t2 + (i - 1) * NS * R1 + r * NS);
#pragma unroll
            for (int c = 0; c < NV; ++c) v[c][i + r * R2] = cmul(v[c][i + r * R2], t);
          }
#pragma unroll
      for (int c = 0; c < NV; ++c) {
        float2 o[R];
#pragma unroll
        for (int r = 0; r < R1; ++r) {
          float2 u[R2];
#pragma unroll
          for (int i = 0; i < R2; ++i) u[i] = v[c][i + r * R2];
          Dft<R2, DIR>::run(u);
#pragma unroll
          for (int i = 0; i < R2; ++i) o[r + i * R1] = u[i];
        }
#pragma unroll
        for (int r = 0; r < R; ++r) v[c][r] = o[r];
      }
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
// element (j, w) at (j << lw) + w (Tile).
//
// Groups up to radix kPairR run on two adjacent columns per thread: every access moves 16 bytes and a
// twiddle serves both.  On single columns the passes waited on the load/store queue (mio_throttle 13 of 30
// warp cycles per instruction, L1 at 73%, DRAM at 52%; now 7, 81% and 62%).  ms, before -> after: 512^3 y
// 0.254 -> 0.214, Green 0.554 -> 0.505, inverse y 0.617 -> 0.580; 384^3 inverse y 0.268 -> 0.247.  A column beyond the row's valid entries may be the
// row's pad entry (rows hold an even number): it is transformed like the others and never used.
constexpr int kPairR = 10;

template <int N>
struct PenCfg {
  // 16 columns where two tiles still leave two CTAs per SM and the last, partly empty chunk of columns is
  // small beside the rest; 4 where two tiles of 8 would not fit a CTA.  us of y / Green / inverse y with 8
  // and 16: 192^3 16.6/32.3/39.8 and 16.2/28.9/33.3, 320^3 57/142/176 and 55/120/133, 360^3 78/175/207 and
  // 92/195/221, 120^3 8.1/12.4/14.9 and 8.2/12.5/13.7; 4 columns at 1024^3 1976/7846/5692 for 1854/5074/5546.
  static constexpr int lw = N > 1536 ? 2 : (N >= 144 && N <= 320 ? 4 : 3);
  static constexpr int W = 1 << lw;
  static constexpr Groups P = make_groups(N, false);
  static constexpr int T = imin(1024, round_up((N * W + 15) / 16, 32));   // 16 values per thread
  static constexpr int PC = ((N / 2 + 1) + 1) & ~1;
  static constexpr int NC = N / 2 + 1;
  static constexpr int chunks = (NC + W - 1) / W;
  static constexpr int tile = N * W;                       // complex elements
  // one work buffer that the middle groups overwrite (each thread's values in registers over a barrier);
  // two where two still leave as many CTAs per SM as the registers do
  static constexpr int regs = 64;
  static constexpr int by_regs = imax(1, imin(2048, 65536 / regs) / T);
  static constexpr bool pp = P.m > 2 && 2 * tile * 8 * by_regs <= 220 * 1024;
  static constexpr int bufs = pp ? 2 : 1;
  static constexpr int smem = bufs * tile * 8;
  static constexpr int minb = imax(1, imin(imin(by_regs, 24), (224 * 1024) / (smem + 1024)));
};

// The butterflies of a radix-R group over a tile: columns per task and task idx's columns w.. and butterfly
template <int N, int R>
struct PenTask {
  using C = PenCfg<N>;
  static constexpr int NV = R <= kPairR ? 2 : 1;
  static constexpr int TOT = ((N / R) << C::lw) / NV, IT = (TOT + C::T - 1) / C::T;
  __device__ __forceinline__ static bool live(int idx) { return TOT % C::T == 0 || idx < TOT; }
  __device__ __forceinline__ static int w(int idx) { return (idx & (C::W / NV - 1)) * NV; }
  __device__ __forceinline__ static int b(int idx) { return idx / (C::W / NV); }
};

// Rows j0 + r STEP of columns w.. of a tile in shared memory, in the transforms of the plan or (REV) the
// reversed plan.  With 64-byte rows, row j of a first group of even radix S lies at slot j ^ (j/S & 1): its
// stores, S rows apart in neighbouring threads, then meet both halves of the banks.  Every later stride is a
// multiple of S, so a butterfly's slots are two pointers plus multiples of the stride.  (768^3 inverse y 2.24
// -> 2.11 ms, y 0.903 -> 0.871; 512^3 y 0.213 -> 0.204; 1024^3 inverse y 5.55 -> 5.42.)
template <int N, bool REV>
struct Tile {
  static constexpr int R0 = Group<N, REV, 0, 1>::R;
  static constexpr int S = PenCfg<N>::W == 8 && R0 % 2 == 0 ? R0 : 0;
  float2* s;
  // pointers of the rows of even and odd r (STEP 1: j0 is a multiple of S; else STEP is)
  template <int STEP>
  __device__ __forceinline__ void places(int j0, int w, float2** even, float2** odd) const {
    constexpr int lw = PenCfg<N>::lw;
    if constexpr (S == 0) {
      *even = *odd = s + (j0 << lw) + w;
    } else if constexpr (STEP == 1) {
      const int t = j0 / S & 1;
      *even = s + ((j0 + t) << lw) + w;
      *odd = s + ((j0 - t) << lw) + w;
    } else {
      static_assert(STEP % S == 0, "strides after the first group");
      const int t = j0 / S & 1;
      *even = s + ((j0 ^ t) << lw) + w;
      *odd = s + ((j0 ^ t ^ (STEP / S & 1)) << lw) + w;
    }
  }
  template <int STEP, int NV, int R>
  __device__ __forceinline__ void load(int j0, int w, float2 (&v)[NV][R]) const {
    float2 *even, *odd;
    places<STEP>(j0, w, &even, &odd);
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const float2* q = (r & 1 ? odd : even) + r * (STEP << PenCfg<N>::lw);
      if constexpr (NV == 2) {
        const float4 t = *reinterpret_cast<const float4*>(q);
        v[0][r] = make_float2(t.x, t.y);
        v[1][r] = make_float2(t.z, t.w);
      } else {
        v[0][r] = *q;
      }
    }
  }
  template <int STEP, int NV, int R>
  __device__ __forceinline__ void store(int j0, int w, const float2 (&v)[NV][R]) const {
    float2 *even, *odd;
    places<STEP>(j0, w, &even, &odd);
#pragma unroll
    for (int r = 0; r < R; ++r) {
      float2* q = (r & 1 ? odd : even) + r * (STEP << PenCfg<N>::lw);
      if constexpr (NV == 2) *reinterpret_cast<float4*>(q) = make_float4(v[0][r].x, v[0][r].y, v[1][r].x, v[1][r].y);
      else *q = v[0][r];
    }
  }
};

// the same of a strided pencil in global memory (row stride JS); columns from `left` on read 0
template <long long JS>
struct ColG {
  float2* base;   // column 0 of the tile, row 0
  int left;       // valid columns
  template <int STEP, int NV, int R>
  __device__ __forceinline__ void load(int j0, int w, float2 (&v)[NV][R]) const {
    const float2* q = base + j0 * JS + w;
    const bool ok = w < left;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      if constexpr (NV == 2) {
        const float4 t = ok ? *reinterpret_cast<const float4*>(q + r * (STEP * JS)) : make_float4(0.f, 0.f, 0.f, 0.f);
        v[0][r] = make_float2(t.x, t.y);
        v[1][r] = make_float2(t.z, t.w);
      } else {
        v[0][r] = ok ? q[r * (STEP * JS)] : make_float2(0.f, 0.f);
      }
    }
  }
  template <int STEP, int NV, int R>
  __device__ __forceinline__ void store(int j0, int w, const float2 (&v)[NV][R]) const {
    if (w >= left) return;
    float2* q = base + j0 * JS + w;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      if constexpr (NV == 2)
        *reinterpret_cast<float4*>(q + r * (STEP * JS)) = make_float4(v[0][r].x, v[0][r].y, v[1][r].x, v[1][r].y);
      else q[r * (STEP * JS)] = v[0][r];
    }
  }
};
// where the tile of this block lies in a grid: AXIS 1 (y pencils of plane blockIdx.y) or 0 (x pencils of row)
template <int N, int AXIS>
struct PenPlace {
  using C = PenCfg<N>;
  static constexpr long long JS = AXIS == 1 ? C::PC : (long long)N * C::PC, OS = AXIS == 1 ? (long long)N * C::PC : C::PC;
  int col0, left;
  long long off;
  __device__ __forceinline__ PenPlace() {
    col0 = blockIdx.x * C::W;
    left = C::NC - col0;
    off = blockIdx.y * OS + col0;
  }
  __device__ __forceinline__ ColG<JS> of(const float2* p) const { return ColG<JS>{const_cast<float2*>(p) + off, left}; }
};

template <int N, bool REV, int G, int DIR, class Src, class Dst>
__device__ __forceinline__ void pen_stage(const Src& src, const Dst& dst, const float2* __restrict__ tw, int tid) {
  using Q = Group<N, REV, G, DIR>;
  using K = PenTask<N, Q::R>;
#pragma unroll(K::IT <= 2 ? K::IT : 1)
  for (int it = 0; it < K::IT; ++it) {
    const int idx = tid + it * PenCfg<N>::T;
    if (K::live(idx)) {
      const int w = K::w(idx), b = K::b(idx), k = Q::k_of(b);
      float2 v[K::NV][Q::R];
      src.template load<Q::NB>(b, w, v);
      Q::run(v, tw, k);
      dst.template store<Q::NS>(Q::out_row(b, k), w, v);
    }
  }
}

// a middle group that overwrites its buffer; the caller synchronises before the next group reads
template <int N, bool REV, int G, int DIR>
__device__ __forceinline__ void pen_inplace(float2* buf, const float2* __restrict__ tw, int tid) {
  using Q = Group<N, REV, G, DIR>;
  using K = PenTask<N, Q::R>;
  float2 v[K::IT][K::NV][Q::R];
#pragma unroll
  for (int it = 0; it < K::IT; ++it) {
    const int idx = tid + it * PenCfg<N>::T;
    if (K::live(idx)) Tile<N, REV>{buf}.template load<Q::NB>(K::b(idx), K::w(idx), v[it]);
  }
  __syncthreads();
#pragma unroll
  for (int it = 0; it < K::IT; ++it) {
    const int idx = tid + it * PenCfg<N>::T;
    if (K::live(idx)) {
      const int b = K::b(idx), k = Q::k_of(b);
      Q::run(v[it], tw, k);
      Tile<N, REV>{buf}.template store<Q::NS>(Q::out_row(b, k), K::w(idx), v[it]);
    }
  }
}

// groups 1 .. m-2 from a (ping-pong with b, or in place); returns the buffer that holds the result,
// synchronised
template <int N, bool REV, int DIR, bool PP, int G = 1>
__device__ __forceinline__ float2* pen_middle(float2* a, float2* b, const float2* __restrict__ tw, int tid) {
  if constexpr (G + 1 < PlanOf<N, REV>::m) {
    if constexpr (PP) {
      pen_stage<N, REV, G, DIR>(Tile<N, REV>{a}, Tile<N, REV>{b}, tw, tid);
      __syncthreads();
      return pen_middle<N, REV, DIR, PP, G + 1>(b, a, tw, tid);
    } else {
      pen_inplace<N, REV, G, DIR>(a, tw, tid);
      __syncthreads();
      return pen_middle<N, REV, DIR, PP, G + 1>(a, b, tw, tid);
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
  after_previous();
  extern __shared__ __align__(16) float2 sm[];
  using C = PenCfg<N>;
  const int tid = threadIdx.x;
  const auto g = PenPlace<N, AXIS>().of(data.p[blockIdx.z]);
  pen_stage<N, false, 0, DIR>(g, Tile<N, false>{sm}, tw, tid);
  __syncthreads();
  float2* cur = pen_middle<N, false, DIR, C::pp>(sm, sm + C::tile, tw, tid);
  pen_stage<N, false, PlanOf<N, false>::m - 1, DIR>(Tile<N, false>{cur}, g, tw, tid);
}

// The inverse x pass of the 2LPT multiplier mp times the lattice spectrum src, into dst
template <int N, long long JS>
struct ColMul {
  ColG<JS> g;
  int my, col0;
  IcMul mp;
  template <int STEP, int NV, int R>
  __device__ __forceinline__ void load(int j0, int w, float2 (&v)[NV][R]) const {
    g.template load<STEP>(j0, w, v);
#pragma unroll
    for (int c = 0; c < NV; ++c)
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const int m[3] = {signed_mode(j0 + r * STEP, N), my, col0 + w + c};
        v[c][r] = ic_multiply_mode(v[c][r], m, N, mp);
      }
  }
};
template <int N>
__global__ void __launch_bounds__(PenCfg<N>::T, PenCfg<N>::minb) k_pen_mul(const float2* src, float2* dst,
                                                                           IcMul mp, const float2* __restrict__ tw) {
  after_previous();
  extern __shared__ __align__(16) float2 sm[];
  using C = PenCfg<N>;
  const int tid = threadIdx.x;
  const PenPlace<N, 0> at;
  const ColMul<N, PenPlace<N, 0>::JS> g{at.of(src), signed_mode(blockIdx.y, N), at.col0, mp};
  pen_stage<N, false, 0, +1>(g, Tile<N, false>{sm}, tw, tid);
  __syncthreads();
  float2* cur = pen_middle<N, false, +1, C::pp>(sm, sm + C::tile, tw, tid);
  pen_stage<N, false, PlanOf<N, false>::m - 1, +1>(Tile<N, false>{cur}, at.of(dst), tw, tid);
}

// NT transforms at once from here on, in the tiles s, s + tile, ...: middle groups in place, last groups
// to d[0], d[1], ...
template <int N, bool REV, int DIR, int G, int NT, class D>
__device__ __forceinline__ void multi_finish(float2* s, const D (&d)[NT], const float2* __restrict__ tw, int tid) {
  if constexpr (G + 1 < PlanOf<N, REV>::m) {
#pragma unroll
    for (int i = 0; i < NT; ++i) pen_inplace<N, REV, G, DIR>(s + i * PenCfg<N>::tile, tw, tid);
    __syncthreads();
    multi_finish<N, REV, DIR, G + 1>(s, d, tw, tid);
  } else {
#pragma unroll
    for (int i = 0; i < NT; ++i) pen_stage<N, REV, G, DIR>(Tile<N, REV>{s + i * PenCfg<N>::tile}, d[i], tw, tid);
  }
}

// NT forward transforms of the tiles s, s + tile, .. whose first groups are done, but for the last groups
template <int N, int NT, int G = 1>
__device__ __forceinline__ void multi_forward(float2* s, const float2* __restrict__ tw, int tid) {
  if constexpr (G + 1 < PlanOf<N, false>::m) {
#pragma unroll
    for (int i = 0; i < NT; ++i) pen_inplace<N, false, G, -1>(s + i * PenCfg<N>::tile, tw, tid);
    __syncthreads();
    multi_forward<N, NT, G + 1>(s, tw, tid);
  }
}

// Configuration of the passes that hold NT tiles
template <int N, int NT>
struct MultiCfg {
  using C = PenCfg<N>;
  static constexpr int smem = NT * C::tile * 8;
  static constexpr int regs = NT == 2 ? 80 : 96;
  static constexpr int minb = imax(1, imin(imin(imax(1, imin(2048, 65536 / regs) / C::T), 16), (224 * 1024) / (smem + 1024)));
};

// Last group of a forward x transform (L) and first of the inverse (F): the same butterflies on the same
// registers
template <int N>
struct Turn {
  using L = Group<N, false, PlanOf<N, false>::m - 1, -1>;
  using F = Group<N, true, 0, +1>;
  using K = PenTask<N, L::R>;
  static_assert(L::R == F::R && L::NS == L::NB && F::NS == 1, "the inverse starts from the forward's registers");
  float2 spec[K::IT][K::NV][L::R];   // values at rows b + r NS of the task's columns
  // f(value, x row, column) of every value
  template <class Fn>
  __device__ __forceinline__ void each(int it, int idx, int col0, Fn&& f) {
#pragma unroll
    for (int c = 0; c < K::NV; ++c)
#pragma unroll
      for (int r = 0; r < L::R; ++r) f(spec[it][c][r], K::b(idx) + r * L::NS, col0 + K::w(idx) + c);
  }
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
  after_previous();
  extern __shared__ __align__(16) float2 sm[];
  using C = PenCfg<N>;
  using X = Turn<N>;
  using K = typename X::K;
  constexpr long long JS = PenPlace<N, 0>::JS;
  const int tid = threadIdx.x, y = blockIdx.y;
  const PenPlace<N, 0> at;
  pen_stage<N, false, 0, -1>(at.of(in), Tile<N, false>{sm}, twf, tid);
  __syncthreads();
  float2* cur = pen_middle<N, false, -1, true>(sm, sm + C::tile, twf, tid);
  X x;
  const int my = y < N / 2 ? y : y - N;
#pragma unroll
  for (int it = 0; it < K::IT; ++it) {
    const int idx = tid + it * C::T;
    if (K::live(idx)) {
      Tile<N, false>{cur}.template load<X::L::NB>(K::b(idx), K::w(idx), x.spec[it]);
      X::L::run(x.spec[it], twf, K::b(idx));
      if (spec_out) at.of(spec_out).template store<X::L::NS>(K::b(idx), K::w(idx), x.spec[it]);
      x.each(it, idx, at.col0, [&](float2& z, int j, int col) {
        const int mx = j < N / 2 ? j : j - N;
        const int m2 = mx * mx + (my * my + col * col);
        z = (m2 > 0 ? g_scale / (float)m2 : 0.0f) * z;
      });
    }
  }
  __syncthreads();   // the forward's buffers are free
#pragma unroll
  for (int it = 0; it < K::IT; ++it) {
    const int idx = tid + it * C::T;
    if (K::live(idx)) {
      const int b = K::b(idx), w = K::w(idx);
      float2 v[K::NV][X::L::R];
#pragma unroll
      for (int r = 0; r < X::L::R; ++r) {
        const float d = __ldg(dtab + b + r * X::L::NS);
#pragma unroll
        for (int c = 0; c < K::NV; ++c) v[c][r] = make_float2(-d * x.spec[it][c][r].y, d * x.spec[it][c][r].x);   // i D H
      }
      X::F::run(v, twr, 0);
      Tile<N, true>{sm}.template store<1>(b * X::L::R, w, v);
      X::F::run(x.spec[it], twr, 0);
      Tile<N, true>{sm + C::tile}.template store<1>(b * X::L::R, w, x.spec[it]);
    }
  }
  __syncthreads();
  const ColG<JS> d[2] = {at.of(out_f), at.of(out_h)};
  multi_finish<N, true, +1, 1>(sm, d, twr, tid);
}

// Inverse y pass of H into the y and z components: i D(k_y) H to out_y and i D(k_z) H to out_z (which
// may be h: a tile is read whole before it is written)
template <int N>
__global__ void __launch_bounds__(PenCfg<N>::T, MultiCfg<N, 2>::minb) k_pen_yz(const float2* h, float2* out_y, float2* out_z,
                                                                               const float* __restrict__ dtab,
                                                                               const float2* __restrict__ tw) {
  after_previous();
  extern __shared__ __align__(16) float2 sm[];
  using C = PenCfg<N>;
  using Q = Group<N, false, 0, +1>;
  using K = PenTask<N, Q::R>;
  const int tid = threadIdx.x;
  const PenPlace<N, 1> at;
#pragma unroll(K::IT <= 2 ? K::IT : 1)
  for (int it = 0; it < K::IT; ++it) {
    const int idx = tid + it * C::T;
    if (K::live(idx)) {
      const int w = K::w(idx), b = K::b(idx);
      float2 z[K::NV][Q::R], v[K::NV][Q::R];
      at.of(h).template load<Q::NB>(b, w, z);
#pragma unroll
      for (int r = 0; r < Q::R; ++r) {
        const float d = __ldg(dtab + b + r * Q::NB);
#pragma unroll
        for (int c = 0; c < K::NV; ++c) v[c][r] = make_float2(-d * z[c][r].y, d * z[c][r].x);
      }
      Q::run(v, tw, 0);
      Tile<N, false>{sm}.template store<1>(b * Q::R, w, v);
#pragma unroll
      for (int c = 0; c < K::NV; ++c) {
        const float d = w + c < at.left ? __ldg(dtab + at.col0 + w + c) : 0.0f;
#pragma unroll
        for (int r = 0; r < Q::R; ++r) z[c][r] = make_float2(-d * z[c][r].y, d * z[c][r].x);
      }
      Q::run(z, tw, 0);
      Tile<N, false>{sm + C::tile}.template store<1>(b * Q::R, w, z);
    }
  }
  __syncthreads();
  const ColG<PenPlace<N, 1>::JS> d[2] = {at.of(out_y), at.of(out_z)};
  multi_finish<N, false, +1, 1>(sm, d, tw, tid);
}

// ---- 2LPT (x and y passes) ----------------------------------------------------------------------
// The 2LPT fields are delta_L(k) / k^2 times products of at most two wave numbers.  A wave number of an
// axis is constant along the other axes' pencils, so one forward x pass makes the inverse x transforms of
// delta/k^2 times 1, k_x and k_x^2, and each y pass those times 1, k_y and k_y^2 as far as they are
// needed; k_z waits for the row pass.  3 x and 6 y transforms then serve the nine first-order fields,
// where a transform of its own for each takes nine and nine (and a multiply each).  The factor of a single
// derivative is 0 on its Nyquist plane, a square keeps it; factors i are left to the row pass.
// With the row passes below (Hessians and source on chip, first positions written with Psi2) a call is 12
// launches and moves 52 field-sized reads and writes where 45 launches moved 120: 256^3 lattice 1706 -> 833
// us (0.51 ms for the 52 at the copy rate), 32^3 271 -> 82 us.

// factor k^p, p = 0, 1, 2, k = 2 pi m / n of storage index j
template <int N>
__device__ __forceinline__ float k_power(int p, int j) {
  constexpr float kf = 6.283185307179586f / N;
  const float k = (j < N / 2 ? j : j - N) * kf;
  return p == 0 ? 1.0f : (p == 1 ? (2 * j == N ? 0.0f : k) : k * k);
}
// z times k^p of storage index j
template <int N, int PW>
__device__ __forceinline__ float2 times_k(float2 z, int j) {
  if constexpr (PW == 0) return z;
  else return k_power<N>(PW, j) * z;
}
// first group of the inverse transforms of z times 1, k, .., k^(NT-1) into the tiles s, s + tile, ..
template <int N, bool REV, int NT, int PW = 0, int NV, int R>
__device__ __forceinline__ void powers_stage(const float2 (&z)[NV][R], int b, int w, float2* s, const float2* __restrict__ tw) {
  if constexpr (PW < NT) {
    using Q = Group<N, REV, 0, +1>;
    static_assert(Q::R == R, "a first group's butterfly");
    float2 v[NV][R];
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
      for (int c = 0; c < NV; ++c) v[c][r] = times_k<N, PW>(z[c][r], b + r * Q::NB);
    Q::run(v, tw, 0);
    Tile<N, REV>{s + PW * PenCfg<N>::tile}.template store<1>(b * R, w, v);
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
  after_previous();
  extern __shared__ __align__(16) float2 sm[];
  using C = PenCfg<N>;
  using X = Turn<N>;
  using K = typename X::K;
  constexpr float kf = 6.283185307179586f / N;
  const int tid = threadIdx.x, y = blockIdx.y;
  const PenPlace<N, 0> at;
  pen_stage<N, false, 0, -1>(at.of(in), Tile<N, false>{sm}, twf, tid);
  __syncthreads();
  float2* cur = pen_middle<N, false, -1, true>(sm, sm + C::tile, twf, tid);
  X x;
  const int my = y < N / 2 ? y : y - N;
#pragma unroll
  for (int it = 0; it < K::IT; ++it) {
    const int idx = tid + it * C::T;
    if (K::live(idx)) {
      Tile<N, false>{cur}.template load<X::L::NB>(K::b(idx), K::w(idx), x.spec[it]);
      X::L::run(x.spec[it], twf, K::b(idx));
      x.each(it, idx, at.col0, [&](float2& z, int j, int col) {
        const int mx = j < N / 2 ? j : j - N;
        const int m2 = mx * mx + (my * my + col * col);
        float g = m2 > 0 ? scale / ((float)m2 * kf * kf) : 0.0f;
        if (AMP && col < C::NC) g *= __ldg(amp_m2 + m2);
        z = g * z;
      });
    }
  }
  __syncthreads();   // the forward's buffers are free
#pragma unroll
  for (int it = 0; it < K::IT; ++it) {
    const int idx = tid + it * C::T;
    if (K::live(idx)) powers_stage<N, true, NT>(x.spec[it], K::b(idx), K::w(idx), sm, twr);
  }
  __syncthreads();
  ColG<PenPlace<N, 0>::JS> d[NT];
#pragma unroll
  for (int i = 0; i < NT; ++i) d[i] = at.of(out.p[i]);
  multi_finish<N, true, +1, 1>(sm, d, twr, tid);
}

struct Pow3 {
  int p[3];   // powers 0, 1, 2
};
// column store times k_z^p
template <int N, long long JS>
struct ColPow {
  ColG<JS> g;
  int p, col0;
  template <int STEP, int NV, int R>
  __device__ __forceinline__ void store(int j0, int w, const float2 (&v)[NV][R]) const {
    float2 u[NV][R];
#pragma unroll
    for (int c = 0; c < NV; ++c) {
      const float f = k_power<N>(p, col0 + w + c);   // k_z <= N/2: the Nyquist entry's square is the same
#pragma unroll
      for (int r = 0; r < R; ++r) u[c][r] = f * v[c][r];
    }
    g.template store<STEP>(j0, w, u);
  }
};

// Inverse y transforms of in times 1, k_y, .. (NT of them), times k_z^zp.p[i], into out.p[0..NT-1];
// out.p[0] may be in.
template <int N, int NT>
__global__ void __launch_bounds__(PenCfg<N>::T, MultiCfg<N, NT>::minb) k_ic_y(const float2* in, Ptr3 out, Pow3 zp,
                                                                              const float2* __restrict__ tw) {
  after_previous();
  extern __shared__ __align__(16) float2 sm[];
  using C = PenCfg<N>;
  using Q = Group<N, false, 0, +1>;
  using K = PenTask<N, Q::R>;
  constexpr long long JS = PenPlace<N, 1>::JS;
  const int tid = threadIdx.x;
  const PenPlace<N, 1> at;
#pragma unroll(K::IT <= 2 ? K::IT : 1)
  for (int it = 0; it < K::IT; ++it) {
    const int idx = tid + it * C::T;
    if (K::live(idx)) {
      float2 z[K::NV][Q::R];
      at.of(in).template load<Q::NB>(K::b(idx), K::w(idx), z);
      powers_stage<N, false, NT>(z, K::b(idx), K::w(idx), sm, tw);
    }
  }
  __syncthreads();
  ColPow<N, JS> d[NT];
#pragma unroll
  for (int i = 0; i < NT; ++i) d[i] = ColPow<N, JS>{at.of(out.p[i]), zp.p[i], at.col0};
  multi_finish<N, false, +1, 1>(sm, d, tw, tid);
}

// ---- transposed gradients (the adjoint's x passes) ------------------------------------------------
// inverse x transform of the values of x, from the tile s, to d
template <int N, class D>
__device__ __forceinline__ void turn_back(Turn<N>& x, float2* s, const D& d, const float2* __restrict__ twr, int tid) {
  using X = Turn<N>;
  using K = typename X::K;
  __syncthreads();   // the forward's tiles are free
#pragma unroll
  for (int it = 0; it < K::IT; ++it) {
    const int idx = tid + it * PenCfg<N>::T;
    if (K::live(idx)) {
      X::F::run(x.spec[it], twr, 0);
      Tile<N, true>{s}.template store<1>(K::b(idx) * X::L::R, K::w(idx), x.spec[it]);
    }
  }
  __syncthreads();
  const D ds[1] = {d};
  multi_finish<N, true, +1, 1>(s, ds, twr, tid);
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
  after_previous();
  extern __shared__ __align__(16) float2 sm[];
  using C = PenCfg<N>;
  using A = Group<N, false, 0, -1>;
  using KA = PenTask<N, A::R>;
  using X = Turn<N>;
  using K = typename X::K;
  const int tid = threadIdx.x, y = blockIdx.y;
  const PenPlace<N, 0> at;
  const float dy = __ldg(dtab + y);
#pragma unroll(KA::IT <= 2 ? KA::IT : 1)
  for (int it = 0; it < KA::IT; ++it) {
    const int idx = tid + it * C::T;
    if (KA::live(idx)) {
      const int w = KA::w(idx), b = KA::b(idx);
      float2 v[KA::NV][A::R], u[KA::NV][A::R];
      at.of(l0).template load<A::NB>(b, w, v);
      A::run(v, twf, 0);
      Tile<N, false>{sm}.template store<1>(b * A::R, w, v);
      at.of(l1).template load<A::NB>(b, w, v);
      at.of(l2).template load<A::NB>(b, w, u);
#pragma unroll
      for (int c = 0; c < KA::NV; ++c) {
        const float dz = w + c < at.left ? __ldg(dtab + at.col0 + w + c) : 0.0f;
#pragma unroll
        for (int r = 0; r < A::R; ++r) u[c][r] = dy * v[c][r] + dz * u[c][r];
      }
      A::run(u, twf, 0);
      Tile<N, false>{sm + C::tile}.template store<1>(b * A::R, w, u);
    }
  }
  __syncthreads();
  multi_forward<N, 2>(sm, twf, tid);
  X x;
  const int my = y < N / 2 ? y : y - N;
#pragma unroll
  for (int it = 0; it < K::IT; ++it) {
    const int idx = tid + it * C::T;
    if (K::live(idx)) {
      const int b = K::b(idx);
      float2 u[K::NV][X::L::R];
      Tile<N, false>{sm}.template load<X::L::NB>(b, K::w(idx), x.spec[it]);
      X::L::run(x.spec[it], twf, b);
      Tile<N, false>{sm + C::tile}.template load<X::L::NB>(b, K::w(idx), u);
      X::L::run(u, twf, b);
#pragma unroll
      for (int r = 0; r < X::L::R; ++r) {
        const float dx = __ldg(dtab + b + r * X::L::NS);
#pragma unroll
        for (int c = 0; c < K::NV; ++c) x.spec[it][c][r] = dx * x.spec[it][c][r] + u[c][r];
      }
      x.each(it, idx, at.col0, [&](float2& z, int j, int col) {
        const int mx = j < N / 2 ? j : j - N, m2 = mx * mx + (my * my + col * col);
        const float g = m2 > 0 ? g_scale / (float)m2 : 0.0f;
        z = make_float2(g * z.y, -g * z.x);
      });
    }
  }
  turn_back<N>(x, sm, at.of(out), twr, tid);
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
  after_previous();
  extern __shared__ __align__(16) float2 sm[];
  using C = PenCfg<N>;
  using A = Group<N, false, 0, -1>;
  using KA = PenTask<N, A::R>;
  using X = Turn<N>;
  using K = typename X::K;
  constexpr float kf = 6.283185307179586f / N;
  const int tid = threadIdx.x, y = blockIdx.y;
  const PenPlace<N, 0> at;
  const int my = y < N / 2 ? y : y - N;
  const float ky2 = k_power<N>(2, y), oy = k_power<N>(1, y);
#pragma unroll 1
  for (int it = 0; it < KA::IT; ++it) {
    const int idx = tid + it * C::T;
    if (KA::live(idx)) {
      const int w = KA::w(idx), b = KA::b(idx);
      float2 v[KA::NV][A::R], u[KA::NV][A::R];
      // v += f(column) u, u = rows of p; IMAG: times -i
      auto add = [&](const float2* p, auto&& f, bool imag) {
        at.of(p).template load<A::NB>(b, w, u);
#pragma unroll
        for (int c = 0; c < KA::NV; ++c) {
          const float g = f(at.col0 + w + c);
#pragma unroll
          for (int r = 0; r < A::R; ++r) {
            const float2 z = g * u[c][r];
            v[c][r] = v[c][r] + (imag ? make_float2(z.y, -z.x) : z);
          }
        }
      };
      auto put = [&](int q) {
        A::run(v, twf, 0);
        Tile<N, false>{sm + q * C::tile}.template store<1>(b * A::R, w, v);
      };
      auto clear = [&]() {
#pragma unroll
        for (int c = 0; c < KA::NV; ++c)
#pragma unroll
          for (int r = 0; r < A::R; ++r) v[c][r] = make_float2(0.f, 0.f);
      };
      clear();
      add(in.h[1], [&](int) { return ky2; }, false);
      add(in.h[2], [&](int col) { return k_power<N>(2, col); }, false);
      add(in.h[5], [&](int col) { return oy * k_power<N>(1, col); }, false);
      add(in.p[1], [&](int) { return r_scale * oy; }, true);
      add(in.p[2], [&](int col) { return r_scale * k_power<N>(1, col); }, true);
      put(0);
      clear();
      add(in.h[3], [&](int) { return oy; }, false);
      add(in.h[4], [&](int col) { return k_power<N>(1, col); }, false);
      add(in.p[0], [&](int) { return r_scale; }, true);
      put(1);
      at.of(in.h[0]).template load<A::NB>(b, w, v);
      put(2);
    }
  }
  __syncthreads();
  multi_forward<N, 3>(sm, twf, tid);
  X x;
#pragma unroll
  for (int it = 0; it < K::IT; ++it) {
    const int idx = tid + it * C::T;
    if (K::live(idx)) {
      const int b = K::b(idx);
      Tile<N, false>{sm}.template load<X::L::NB>(b, K::w(idx), x.spec[it]);
      X::L::run(x.spec[it], twf, b);
#pragma unroll
      for (int q = 1; q < 3; ++q) {
        float2 u[K::NV][X::L::R];
        Tile<N, false>{sm + q * C::tile}.template load<X::L::NB>(b, K::w(idx), u);
        X::L::run(u, twf, b);
#pragma unroll
        for (int r = 0; r < X::L::R; ++r) {
          const float f = k_power<N>(q, b + r * X::L::NS);
#pragma unroll
          for (int c = 0; c < K::NV; ++c) x.spec[it][c][r] = x.spec[it][c][r] + f * u[c][r];
        }
      }
      x.each(it, idx, at.col0, [&](float2& z, int j, int col) {
        const int mx = j < N / 2 ? j : j - N, m2 = mx * mx + (my * my + col * col);
        const float g = m2 > 0 && col < C::NC ? __ldg(amp_m2 + m2) / ((float)m2 * kf * kf) : 0.0f;
        z = g * z;
      });
    }
  }
  turn_back<N>(x, sm, at.of(out), twr, tid);
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
  after_previous();
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
  after_previous();
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
  after_previous();
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
__global__ void __launch_bounds__(RowCfg<N>::T, RowCfg<N>::minb(C2rCfg<N>::bufs)) k_ic_z2(Ptr3 f, const float* psi1,
                                                                                         float* psi2, float* s, float* v0,
                                                                                         long long npart, float r_scale, float d1,
                                                                                         float d2, long long npairs,
                                                                                         const float2* __restrict__ tw) {
  after_previous();
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
    for (int h = 0; h < 2; ++h) {
      float p1[Q::R];   // every load of a row before its stores, which may alias as far as the compiler knows
#pragma unroll
      for (int r = 0; r < Q::R; ++r) p1[r] = psi1[o + h * N + r * Q::NS];
#pragma unroll
      for (int r = 0; r < Q::R; ++r) {
        const long long i = o + h * N + r * Q::NS;
        const float p2 = (h ? v[r].y : v[r].x) * -r_scale;
        psi2[i] = p2;
        s[i] = d1 * p1[r] + d2 * p2;
        v0[i] = 0.0f;
      }
    }
  });
}

}  // namespace ct
}  // namespace cola
