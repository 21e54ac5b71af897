// Friends-of-friends halo finding (§2.3: run on the fly, 19% of the paper's time; §3.2: linking
// length 0.2 times the mean particle separation) on the fixed-point coordinates of the deposit.
//
// Two particles are friends when their periodic distance is at most l; groups are the connected
// components.  Distances are exact integers: G = (q R + rint(s 2^20)) mod N 2^20 per axis (an unsigned
// 32-bit number: N <= 4096), l = rint(b (N/N_p) 2^20), and the test d^2 <= l^2 runs in integers, so no
// rounding decides a link and the result is bit-identical to any exact implementation.
//   1. G per particle and a cell of side > l, about kCellsPerParticle cells per particle; counting sort
//      into (G, id) records by cell;
//   2. every record, in sorted order, meets the records behind it in its own cell and in the 13 forward
//      neighbour cells (five ranges of the sorted list: cells are contiguous along z) and joins the trees
//      of friends (lock-free union-find over sorted positions: a root is hooked, by CAS, to the larger).
//      Twice: first each record takes one friend as its parent, without atomics, which makes a few trees of
//      every group, whose root each record then carries; then all friends, where a record with the same
//      root needs no distance;
//   3. path compression, members and smallest particle id per root; label = that id;
//   4. groups of >= n_min members compacted in increasing label order by a scan; centre of mass from
//      exact 64-bit sums of minimum-image offsets to the label's particle.
#include "cola_internal.h"

#include <cstdio>

namespace cola {
namespace {

constexpr int kFlagIterations = 4;   // union-find did not converge (never expected; reported)
// Kernel time of a call at 128^3/256^3: 649 us with 8 cells per particle; 741 with 27, 971 with 64 (clearing and
// scanning them).
constexpr double kCellsPerParticle = 8.0;

int check_launch(const char* what) {
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) {
    std::fprintf(stderr, "cola: launch of %s failed: %s\n", what, cudaGetErrorString(e));
    return COLA_ERR_CUDA;
  }
  return COLA_OK;
}

unsigned grid_for(long long work, int threads) {
  long long b = (work + threads - 1) / threads;
  const long long cap = 152LL * 16 * 4;
  if (b > cap) b = cap;
  return (unsigned)(b < 1 ? 1 : b);
}

// minimum image of a difference in (-modulus, modulus)
__device__ __forceinline__ long long wrap(long long d, long long modulus) {
  const long long h = modulus / 2;
  if (d > h) d -= modulus;
  else if (d < -h) d += modulus;
  return d;
}

// root of x; path splitting (each visited node is pointed at its grandparent).  Parents are never before
// their children, so the walk ends within n hops.
__device__ __forceinline__ int find_root(int* parent, int x) {
  volatile int* p = parent;
  int cur = x, nxt = p[cur];
  while (nxt != cur) {
    const int nn = p[nxt];
    if (nn != nxt) p[cur] = nn;
    cur = nxt;
    nxt = nn;
  }
  return cur;
}

// joins the trees of a and b; returns the root they share afterwards (as far as this thread knows)
__device__ __forceinline__ int unite(int* parent, int a, int b, int* flags) {
  for (int it = 0; it < (1 << 22); ++it) {
    a = find_root(parent, a);
    b = find_root(parent, b);
    if (a == b) return a;
    if (a > b) {
      const int t = a;
      a = b;
      b = t;
    }
    if (atomicCAS(parent + a, a, b) == a) return b;   // hook the smaller root under the larger
  }
  atomicOr(flags, kFlagIterations);
  return b;
}

// cell of a coordinate: floor(g inv / 2^64), inv = floor(2^64 ncs / modulus).  The cells are at least
// modulus / ncs wide but for the last, which rounding may narrow by less than one unit; ncs is chosen
// for l + 2, so points within l of each other are in the same or adjacent cells, around the edge too.
__device__ __forceinline__ int cell_of(unsigned g, unsigned long long inv) { return (int)__umul64hi(g, inv); }

__global__ void __launch_bounds__(256) k_fof_prepare(ParticleGeom pg, const float* s, FofGeom f, unsigned* g0,
                                                     unsigned* g1, unsigned* g2, int* key, unsigned* counts) {
  after_previous();
  const long long n = pg.npart;
  const long long modulus = f.modulus;
  const int np = pg.np, qx = blockIdx.y, qy = blockIdx.x * blockDim.y + threadIdx.y;
  if (qy >= np) return;
  for (int qz = threadIdx.x; qz < np; qz += blockDim.x) {
    const long long id = ((long long)qx * np + qy) * np + qz;
    const unsigned a = (unsigned)fixed_coord(qx, s[id], pg.r_fixed, modulus);
    const unsigned b = (unsigned)fixed_coord(qy, s[n + id], pg.r_fixed, modulus);
    const unsigned c = (unsigned)fixed_coord(qz, s[2 * n + id], pg.r_fixed, modulus);
    g0[id] = a;
    g1[id] = b;
    g2[id] = c;
    const int k = (cell_of(a, f.inv) * f.ncs + cell_of(b, f.inv)) * f.ncs + cell_of(c, f.inv);
    key[id] = k;
    atomicAdd(counts + k, 1u);
  }
}

// records by cell; a cell's count runs down to zero
__global__ void k_fof_scatter(int n, const int* key, const unsigned* off, unsigned* counts,
                              const unsigned* g0, const unsigned* g1,
                              const unsigned* g2, uint4* rec, int* ids, int* min_id) {
  after_previous();
  for (long long id = blockIdx.x * (long long)blockDim.x + threadIdx.x; id < n; id += (long long)gridDim.x * blockDim.x) {
    const int k = key[id];
    const unsigned t = off[k] + atomicSub(counts + k, 1u) - 1u;
    rec[t] = make_uint4(g0[id], g1[id], g2[id], t);
    ids[t] = (int)id;
    min_id[t] = (int)id;
  }
}

// Whether records me and o, the latter shifted by (sx, sy, sz) modulo 2^32, are friends.
// ONE: a single cell (l over a third of the box), minimum images by comparison.
template <bool ONE>
__device__ __forceinline__ bool friends(const uint4& me, const uint4& o, unsigned sx, unsigned sy, unsigned sz, int ell,
                                        unsigned long long ell2, long long modulus) {
  int d0, d1, d2;
  if (ONE) {
    const long long w0 = wrap((long long)o.x - me.x, modulus), w1 = wrap((long long)o.y - me.y, modulus),
                    w2 = wrap((long long)o.z - me.z, modulus);
    if (w0 > ell || w0 < -ell || w1 > ell || w1 < -ell || w2 > ell || w2 < -ell) return false;
    d0 = (int)w0;
    d1 = (int)w1;
    d2 = (int)w2;
  } else {
    d0 = (int)(o.x + sx - me.x);
    d1 = (int)(o.y + sy - me.y);
    d2 = (int)(o.z + sz - me.z);
    if (d0 > ell || d0 < -ell || d1 > ell || d1 < -ell || d2 > ell || d2 < -ell) return false;
  }
  return (unsigned long long)((long long)d0 * d0) + (unsigned long long)((long long)d1 * d1) +
             (unsigned long long)((long long)d2 * d2) <=
         ell2;
}

// Calls meet(lo, hi, sx, sy, sz) for the ranges of records behind t in its own and its forward neighbour
// cells, the farthest columns first; stops when it returns true.
template <bool ONE, class F>
__device__ __forceinline__ void forward_ranges(int t, int n, const uint4& me, const unsigned* off,
                                               const FofGeom& f, F&& meet) {
  if (ONE) {
    meet((unsigned)t + 1u, (unsigned)n, 0u, 0u, 0u);
    return;
  }
  const int ncs = f.ncs;
  const unsigned mod = (unsigned)f.modulus;   // shifts are modulo 2^32
  const int cx = cell_of(me.x, f.inv), cy = cell_of(me.y, f.inv), cz = cell_of(me.z, f.inv);
  const int xp = cx + 1 < ncs ? cx + 1 : 0, yp = cy + 1 < ncs ? cy + 1 : 0, ym = cy > 0 ? cy - 1 : ncs - 1;
  const unsigned sx = cx + 1 < ncs ? 0u : mod, syp = cy + 1 < ncs ? 0u : mod, sym = cy > 0 ? 0u : 0u - mod;
  const int a = cz > 0 ? cz - 1 : 0, b = cz + 1 < ncs ? cz + 1 : ncs - 1;
#pragma unroll 1
  for (int c = 0; c < 4; ++c) {   // cells cz - 1 .. cz + 1 of a column, in up to two ranges
    const int x = c < 3 ? xp : cx, y = c == 1 ? cy : (c == 2 ? ym : yp);
    const unsigned dx = c < 3 ? sx : 0u, dy = c == 1 ? 0u : (c == 2 ? sym : syp);
    const unsigned* o = off + ((long long)x * ncs + y) * ncs;
    if (meet(o[a], o[b + 1], dx, dy, 0u)) return;
    if (cz == 0 && meet(o[ncs - 1], o[ncs], dx, dy, 0u - mod)) return;
    if (cz + 1 == ncs && meet(o[0], o[1], dx, dy, mod)) return;
  }
  const unsigned* own = off + ((long long)cx * ncs + cy) * ncs;
  if (cz + 1 == ncs && meet(own[0], own[1], 0u, 0u, mod)) return;
  meet((unsigned)t + 1u, own[b + 1], 0u, 0u, 0u);
}

// First pass: the record's parent is one friend behind it (itself if it has none), from the last of the
// farthest column, so that paths are short; only this thread writes it.  Element counts come near 2^31, so
// here and below the index of a walk, and its step of a whole grid above all, has 64 bits.
template <bool ONE>
__global__ void __launch_bounds__(256) k_fof_first(int n, const uint4* rec, const unsigned* off,
                                                   FofGeom f, int* parent) {
  after_previous();
  const int ell = (int)f.ell;
  const unsigned long long ell2 = (unsigned long long)f.ell * (unsigned long long)f.ell;
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int t = (int)i;
  const uint4 me = *(rec + t);
  int p = t;
  forward_ranges<ONE>(t, n, me, off, f, [&](unsigned lo, unsigned hi, unsigned sx, unsigned sy, unsigned sz) {
    for (unsigned u = hi; u > lo && (int)u > t + 1; --u)   // a parent comes after its child
      if (friends<ONE>(me, *(rec + u - 1), sx, sy, sz, ell, ell2, f.modulus)) {
        p = (int)u - 1;
        return true;
      }
    return false;
  });
  parent[t] = p;
}

// Second pass: joins record t with its friends behind it of another tree than its own after the first
// (rec.w).  What bounds the passes: the latency of the neighbours' records and of the union-find's
// parents, which come from L2.  Sorted order keeps the records near and a warp's lanes in the same cells;
// in a dense halo, where a record has hundreds of friends, they are passed over by the root that comes
// with their coordinates.  (In lattice order, 27 cells of side l looked up one by one, 134 M of them, and
// two root searches for every friend, 128^3/256^3 at b = 0.2 took 1225 us for the links and 1240 us for
// scanning the cells; in sorted order with one pass 1000 and 40; now 280 to 340 for both passes.)
template <bool ONE>
__global__ void __launch_bounds__(256) k_fof_link(int n, const uint4* rec, const unsigned* off,
                                                  FofGeom f, int* parent, int* flags) {
  after_previous();
  const int ell = (int)f.ell;
  const unsigned long long ell2 = (unsigned long long)f.ell * (unsigned long long)f.ell;
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int t = (int)i;
  const uint4 me = *(rec + t);
  int root = (int)me.w;
  forward_ranges<ONE>(t, n, me, off, f, [&](unsigned lo, unsigned hi, unsigned sx, unsigned sy, unsigned sz) {
    for (unsigned u = lo; u < hi; ++u) {
      const uint4 o = *(rec + u);
      if (o.w != me.w && friends<ONE>(me, o, sx, sy, sz, ell, ell2, f.modulus))
        root = unite(parent, root, (int)o.w, flags);
    }
    return false;
  });
}

// each record takes its tree's root after the first pass
__global__ void k_fof_carry(int n, uint4* rec, int* parent) {
  after_previous();
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n; t += (long long)gridDim.x * blockDim.x)
    rec[t].w = (unsigned)find_root(parent, (int)t);
}

// root of every record, members and smallest id per root (one atomic per run of lanes with one root)
__global__ void k_fof_roots(int n, const int* ids, int* parent, int* root, unsigned* cnt, int* min_id) {
  after_previous();
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n; t += (long long)gridDim.x * blockDim.x) {
    const int r = find_root(parent, (int)t);
    root[t] = r;
    const unsigned grp = __match_any_sync(__activemask(), r);
    const int least = __reduce_min_sync(grp, ids[t]);
    if ((int)(threadIdx.x & 31) == __ffs(grp) - 1) {
      atomicAdd(cnt + r, (unsigned)__popc(grp));
      atomicMin(min_id + r, least);
    }
  }
}

__global__ void k_fof_label(int n, const int* ids, const int* root,
                            const unsigned* cnt, const int* min_id, int n_min, int* label,
                            int* size, unsigned* halo_flag) {
  after_previous();
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n; t += (long long)gridDim.x * blockDim.x) {
    const int id = ids[t], r = root[t], l = min_id[r];
    const unsigned c = cnt[r];
    label[id] = l;
    size[id] = (int)c;
    halo_flag[id] = (l == id && c >= (unsigned)n_min) ? 1u : 0u;
  }
}

__global__ void k_fof_halo_sums(int n, const uint4* rec, const int* root,
                                const unsigned* cnt, const int* min_id, int n_min,
                                const unsigned* hoff, const unsigned* g0,
                                const unsigned* g1, const unsigned* g2, long long modulus,
                                int capacity, unsigned long long* sums) {
  after_previous();
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n; t += (long long)gridDim.x * blockDim.x) {
    const int r = root[t];
    if (cnt[r] < (unsigned)n_min) continue;
    const int l = min_id[r];
    const unsigned h = hoff[l];
    if (h >= (unsigned)capacity) continue;
    const uint4 me = rec[t];
    long long d[3] = {wrap((long long)me.x - g0[l], modulus), wrap((long long)me.y - g1[l], modulus),
                      wrap((long long)me.z - g2[l], modulus)};
    // a whole warp inside one halo, usual in large ones, adds once
    const unsigned active = __activemask();
    int same = 0;
    __match_all_sync(active, r, &same);
    if (active == 0xffffffffu && same) {
#pragma unroll
      for (int a = 0; a < 3; ++a)
        for (int o = 16; o > 0; o >>= 1) d[a] += __shfl_down_sync(0xffffffffu, d[a], o);
      if (threadIdx.x & 31) continue;
    }
#pragma unroll
    for (int a = 0; a < 3; ++a) atomicAdd(sums + (long long)a * capacity + h, (unsigned long long)d[a]);
  }
}

__global__ void k_fof_halo_finish(int n, const unsigned* halo_flag, const int* size,
                                  const unsigned* hoff, const unsigned* g0,
                                  const unsigned* g1, const unsigned* g2, long long modulus,
                                  int capacity, const unsigned long long* sums, int* halo_label,
                                  int* halo_size, double* halo_pos, int* nhalo) {
  after_previous();
  for (long long id = blockIdx.x * (long long)blockDim.x + threadIdx.x; id < n; id += (long long)gridDim.x * blockDim.x) {
    if (id == 0) *nhalo = (int)hoff[n];
    if (!halo_flag[id]) continue;
    const unsigned h = hoff[id];
    if (h >= (unsigned)capacity) continue;
    const unsigned c = (unsigned)size[id];
    if (halo_label) halo_label[h] = (int)id;
    if (halo_size) halo_size[h] = (int)c;
    if (halo_pos) {
      const unsigned g[3] = {g0[id], g1[id], g2[id]};
      const double mod = (double)modulus;
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        const double com = (double)g[a] + (double)(long long)sums[a * (long long)capacity + h] / (double)c;
        double m = fmod(com, mod);
        if (m < 0.0) m += mod;
        halo_pos[a * (long long)capacity + h] = m / (double)(1LL << kFracBits);
      }
    }
  }
}

}  // namespace

bool fof_geometry(int nmesh, int np, double b, FofGeom* f) {
  const long long modulus = (long long)nmesh << kFracBits;
  const double ell = rint(b * ((double)nmesh / np) * (double)(1LL << kFracBits));
  if (!(ell >= 1.0) || ell > (double)(1LL << 30)) return false;   // d^2 sums stay below 2^62
  f->modulus = modulus;
  f->ell = (long long)ell;
  // Cells of side > l, about kCellsPerParticle per particle and at most 512^3: smaller cells hold fewer
  // strangers to test, larger ones cost less to clear, scan and look up.
  long long ncs = modulus / (f->ell + 2);
  const double want = cbrt(kCellsPerParticle * np * (double)np * np);
  if (ncs > (long long)want) ncs = (long long)want;
  if (ncs > 512) ncs = 512;
  if (ncs < 3) ncs = 1;   // every neighbour cell is a different one from three cells on
  f->ncs = (int)ncs;
  f->ncells = (long long)ncs * ncs * ncs;
  f->inv = (unsigned long long)(((unsigned __int128)ncs << 64) / (unsigned __int128)modulus);
  return true;
}

int launch_fof(const ParticleGeom& pg, const FofGeom& f, const float* s, const FofBuffers& fb, int n_min, int* label,
               int* size, int* halo_label, int* halo_size, double* halo_pos, int capacity, int* nhalo, int* flags,
               cudaStream_t st) {
  const int n = (int)pg.npart;   // below 2^31
  int e;
  if (cudaMemsetAsync(fb.counts, 0, f.ncells * sizeof(unsigned), st) != cudaSuccess ||
      cudaMemsetAsync(fb.cnt, 0, (size_t)n * sizeof(unsigned), st) != cudaSuccess)
    return COLA_ERR_CUDA;
  const unsigned gp = grid_for(n, 256);
  const RowBlocks rb = row_blocks(pg.np);
  launch_after(k_fof_prepare, rb.grid, rb.block, 0, st, pg, s, f, fb.g[0], fb.g[1], fb.g[2], fb.key, fb.counts);
  if ((e = check_launch("fof_prepare")) != COLA_OK) return e;
  if ((e = launch_excl_scan(fb.counts, (int)f.ncells, fb.seg, fb.off, st)) != COLA_OK) return e;
  launch_after(k_fof_scatter, gp, 256, 0, st, n, fb.key, fb.off, fb.counts, fb.g[0], fb.g[1], fb.g[2], fb.rec, fb.ids, fb.min_id);
  const unsigned gl = (unsigned)((n + 255LL) / 256);   // one record per thread: their work differs most
  if (f.ncs == 1) launch_after(k_fof_first<true>, gl, 256, 0, st, n, fb.rec, fb.off, f, fb.parent);
  else launch_after(k_fof_first<false>, gl, 256, 0, st, n, fb.rec, fb.off, f, fb.parent);
  launch_after(k_fof_carry, gp, 256, 0, st, n, fb.rec, fb.parent);
  if (f.ncs == 1) launch_after(k_fof_link<true>, gl, 256, 0, st, n, fb.rec, fb.off, f, fb.parent, flags);
  else launch_after(k_fof_link<false>, gl, 256, 0, st, n, fb.rec, fb.off, f, fb.parent, flags);
  launch_after(k_fof_roots, gp, 256, 0, st, n, fb.ids, fb.parent, fb.key, fb.cnt, fb.min_id);   // key: the roots from here on
  launch_after(k_fof_label, gp, 256, 0, st, n, fb.ids, fb.key, fb.cnt, fb.min_id, n_min, label, size, fb.flag);
  if ((e = check_launch("fof_link")) != COLA_OK) return e;
  if ((e = launch_excl_scan(fb.flag, n, fb.seg, fb.hoff, st)) != COLA_OK) return e;
  const int cap = capacity > 0 ? capacity : 0;
  if (cap > 0 && halo_pos) {
    if (cudaMemsetAsync(fb.sums, 0, 3ULL * cap * sizeof(unsigned long long), st) != cudaSuccess) return COLA_ERR_CUDA;
    launch_after(k_fof_halo_sums, gp, 256, 0, st, n, fb.rec, fb.key, fb.cnt, fb.min_id, n_min, fb.hoff, fb.g[0], fb.g[1], fb.g[2], f.modulus, cap, fb.sums);
  }
  launch_after(k_fof_halo_finish, gp, 256, 0, st, n, fb.flag, size, fb.hoff, fb.g[0], fb.g[1], fb.g[2], f.modulus, cap, fb.sums, halo_label, halo_size, cap > 0 ? halo_pos : nullptr, nhalo);
  return check_launch("fof_halos");
}

}  // namespace cola
