// Host side of the FFT passes: plans (factorisation, twiddle tables) and the choice between the kernels
// compiled for a length (fft_ct.cu) and the run-time plans (fft_generic.cu).
#include "fft_core.cuh"
#include "fft_ops.h"

#include <mutex>
#include <set>
#include <utility>

namespace cola {
using namespace fftk;
namespace {

struct TileShape {
  int lw;
  int threads;
  size_t smem;
};

constexpr int kTileElems = 6144;    // complex elements per tile of a run-time plan (two buffers: about 100 KB)

TileShape tile_shape(int n, int wmax) {
  int lw = 0;
  while ((2 << lw) <= wmax && n * (2 << lw) <= kTileElems) ++lw;
  TileShape t;
  t.lw = lw;
  int th = ((n << lw) + kEpt - 1) / kEpt;
  th = ((th + 31) / 32) * 32;
  t.threads = th < 32 ? 32 : th;
  t.smem = 2 * (size_t)(n + n / 16 + 1) * (1u << lw) * sizeof(float2);
  return t;
}

int largest_pow2_le(int v) {
  int p = 1;
  while (p * 2 <= v) p *= 2;
  return p;
}

int check_launch(const char* what) {
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) {
    std::fprintf(stderr, "cola: launch of %s failed: %s\n", what, cudaGetErrorString(e));
    return COLA_ERR_CUDA;
  }
  return COLA_OK;
}

template <int PART>
const FftOps* find_ops(int n) {
  if constexpr (PART < COLA_CT_PARTS) {
    const FftOps* o = ct::ops_in_part<PART>(n);
    return o ? o : find_ops<PART + 1>(n);
  } else {
    return nullptr;
  }
}

}  // namespace

bool fft_plan_set(FftPlan* plan, int n, const float2* table) {
  const Radices f = factor_radices(n);
  if (!f.ok) return false;
  plan->dev.n = n;
  plan->dev.nstages = f.m;
  for (int i = 0; i < kMaxStages; ++i) plan->dev.radix[i] = i < f.m ? f.r[i] : 1;
  plan->dev.tw = table;
  plan->tab = FftTables{table + n, table + 2 * n};
  plan->ops = find_ops<0>(n);
  return true;
}

int fft_plan_init(FftPlan* plan, int n) {
  if (!factor_radices(n).ok) return COLA_ERR_INVALID;
  const size_t total = fft_table_entries(n);
  std::vector<float2> h(total, make_float2(0.f, 0.f));
  for (int t = 0; t < n; ++t) {
    const double ang = -2.0 * M_PI * (double)t / (double)n;
    h[t] = make_float2((float)std::cos(ang), (float)std::sin(ang));
  }
  for (int rev = 0; rev < 2; ++rev) {
    const Groups g = make_groups(n, rev != 0);
    if (!g.ok) continue;
    for (int e = 0; e + 1 < n; ++e) h[(size_t)(1 + rev) * n + e] = h[stage_twiddle(g, e)];
  }
  if (cudaMalloc(&plan->tw, total * sizeof(float2)) != cudaSuccess) return COLA_ERR_OOM;
  if (cudaMemcpy(plan->tw, h.data(), total * sizeof(float2), cudaMemcpyHostToDevice) != cudaSuccess)
    return COLA_ERR_CUDA;
  fft_plan_set(plan, n, plan->tw);
  once_on_device(reinterpret_cast<const void*>(&generic_set_smem_limits), [](const void*) { generic_set_smem_limits(); });
  return COLA_OK;
}

void once_on_device(const void* key, void (*set)(const void* key)) {
  static std::mutex mu;
  static std::set<std::pair<int, const void*>> done;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) dev = -1;
  std::lock_guard<std::mutex> lock(mu);   // held over set
  if (done.insert({dev, key}).second) set(key);
}

void fft_set_smem_limits() { generic_set_smem_limits(); }

void fft_plan_free(FftPlan* plan) {
  if (plan->tw) cudaFree(plan->tw);
  plan->tw = nullptr;
}

int launch_r2c_rows(const FftPlan& p, const Grid3& g, RowSource kind, const void* const* src, int fields,
                    long long src_row_stride, float scale, float2* const* dst, cudaStream_t st,
                    unsigned long long* mass_acc) {
  if (p.ops) {
    p.ops->r2c(kind, src, fields, src_row_stride, scale, dst, p.tab, mass_acc, st);
    return check_launch("r2c");
  }
  const long long nrows = (long long)g.rows();
  const TileShape t = tile_shape(g.n, 1 << 20);
  const unsigned blocks = (unsigned)((nrows + (2LL << t.lw) - 1) / (2LL << t.lw));
  for (int i = 0; i < fields; ++i)
    generic_r2c_launch(p.dev, t.lw, blocks, t.threads, t.smem, kind, src[i], src_row_stride, scale, dst[i], g.pc, nrows,
                       kind == kSrcFixedPoint ? mass_acc : nullptr, st);
  return check_launch("r2c_rows");
}

int launch_c2r_rows(const FftPlan& p, const Grid3& g, float2* const* data, int fields, cudaStream_t st) {
  if (p.ops) {
    p.ops->c2r(data, fields, p.tab, st);
    return check_launch("c2r");
  }
  const long long nrows = (long long)g.rows();
  const TileShape t = tile_shape(g.n, 1 << 20);
  const unsigned blocks = (unsigned)((nrows + (2LL << t.lw) - 1) / (2LL << t.lw));
  for (int i = 0; i < fields; ++i)
    generic_c2r_launch(p.dev, t.lw, blocks, t.threads, t.smem, data[i], g.pc, nrows, st);
  return check_launch("c2r_rows");
}

bool ic_compiled(const FftPlan& p) { return p.ops && p.ops->ic_x; }
bool x_mul_compiled(const FftPlan& p) { return p.ops && p.ops->x_mul; }

int launch_pencils_x_mul(const FftPlan& p, const Grid3&, const float2* src, const IcMul& mul, float2* dst,
                         cudaStream_t st) {
  if (!x_mul_compiled(p)) return COLA_ERR_INVALID;
  p.ops->x_mul(src, mul, dst, p.tab, st);
  return check_launch("pencils_x_mul");
}

int launch_c2r_rows_dense(const FftPlan& p, const Grid3&, const float2* data, float scale, float* out,
                          cudaStream_t st) {
  if (!p.ops) return COLA_ERR_INVALID;
  p.ops->c2r_dense(data, scale, out, p.tab, st);
  return check_launch("c2r_dense");
}


int launch_ic_x(const FftPlan& p, const float2* in, float2* const* out, int fields, float scale, const float* amp_m2,
                cudaStream_t st) {
  p.ops->ic_x(in, out, fields, scale, amp_m2, p.tab, st);
  return check_launch("ic_x");
}
int launch_ic_y(const FftPlan& p, const float2* in, float2* const* out, int fields, const int* zp, cudaStream_t st) {
  p.ops->ic_y(in, out, fields, zp, p.tab, st);
  return check_launch("ic_y");
}
int launch_ic_z1(const FftPlan& p, float2* const t[6], float2* src_k, float* psi1, float r_scale, cudaStream_t st) {
  p.ops->ic_z1(t, src_k, psi1, r_scale, p.tab, st);
  return check_launch("ic_z1");
}
int launch_ic_z2(const FftPlan& p, float2* const f[3], const float* psi1, float* psi2, float* s, float* v,
                 float r_scale, float d1, float d2, cudaStream_t st) {
  p.ops->ic_z2(f, psi1, psi2, s, v, r_scale, d1, d2, p.tab, st);
  return check_launch("ic_z2");
}

int launch_lpt_adj(const FftPlan& p, const float2* const h[6], const float2* const l[3], float2* out, float r_scale,
                   const float* amp_m2, cudaStream_t st) {
  p.ops->lpt_adj(h, l, out, r_scale, amp_m2, p.tab, st);
  return check_launch("lpt_adj");
}
int launch_grad_adj(const FftPlan& p, float2* const l[3], float2* out, const float* dtab, float g_scale,
                    cudaStream_t st) {
  p.ops->grad_adj(l, out, dtab, g_scale, p.tab, st);
  return check_launch("grad_adj");
}

int launch_pencils(const FftPlan& p, const Grid3& g, int axis, int dir, float2* const* data, int fields,
                   cudaStream_t st) {
  if (p.ops) {
    p.ops->pencils(axis, dir, data, fields, p.tab, st);
    return check_launch("pencils");
  }
  const long long plane = (long long)g.n * g.pc;
  const long long jstride = axis == 1 ? g.pc : plane;
  const long long ostride = axis == 1 ? plane : g.pc;
  const TileShape t = tile_shape(g.n, largest_pow2_le(g.nc));
  dim3 grid((g.nc + (1 << t.lw) - 1) >> t.lw, g.n);
  for (int i = 0; i < fields; ++i)
    generic_pencils_launch(p.dev, t.lw, grid, t.threads, t.smem, dir, data[i], jstride, ostride, g.nc, st);
  return check_launch("pencils_generic");
}

int launch_green_x(const FftPlan& p, const Grid3& g, float2* const out[3], const float* dtab, float scale,
                   cudaStream_t st, float2* spec_out, bool* spec_saved) {
  if (spec_saved) *spec_saved = false;
  const double kf = 2.0 * M_PI / g.n;
  const double n3 = (double)g.n * g.n * g.n;
  const float g_scale = (float)((double)scale / (kf * kf * n3));
  if (p.ops) {
    p.ops->green(out[2], out[0], out[2], dtab, g_scale, p.tab, spec_out, st);
    if (spec_saved) *spec_saved = spec_out != nullptr;
    return check_launch("green");
  }
  const TileShape t = tile_shape(g.n, largest_pow2_le(g.nc));
  dim3 grid((g.nc + (1 << t.lw) - 1) >> t.lw, g.n);
  generic_green_launch(p.dev, t.lw, grid, t.threads, t.smem, out[2], out, g.pc, g.nc, dtab, g_scale, st);
  return check_launch("green_x");
}

int launch_green_y(const FftPlan& p, const Grid3& g, float2* const out[3], const float* dtab, cudaStream_t st) {
  if (!p.ops) return launch_pencils(p, g, 1, +1, out, 3, st);
  p.ops->pencils(1, +1, out, 1, p.tab, st);
  p.ops->pencils_yz(out[2], out[1], out[2], dtab, p.tab, st);
  return check_launch("green_y");
}

}  // namespace cola
