// Spatial binning of particles by mesh column tiles, and the tile-wise CIC deposit and gather.
//
// The particle arrays stay in Lagrangian order (particle id = lattice index).  At late times the
// particles of one lattice plane are spread over tens of mesh planes (§2.3 mesh; displacements of
// ~8 cells rms at a = 1 for the 0.78 Mpc/h cells of the 1536^3 mesh), so visiting them in lattice
// order touches far more mesh than the L2 holds.  Each step therefore
//   1. counts particles per tile of T x T x TZ mesh cells (T = 8 across, TZ = 64 along z) from the
//      fixed-point base cell (the same integer cell as the deposit), with warp-aggregated atomics;
//   2. scans the counts into offsets;
//   3. scatters packed lattice coordinates into their tile's list.  A particle whose base cell
//      lies on an upper face of its tile also goes, as a "spill" entry, to the neighbouring tiles
//      its cloud reaches (at most seven);
//   4. deposits tile by tile: one CTA sums the 8 fixed-point weights of its primary and spill
//      particles that fall inside the tile in shared memory (64-bit integers, exact) and writes
//      the whole tile once with plain stores: no clearing pass and no global atomics on the mesh;
//   5. gathers the force and applies the kick and drift tile by tile (primary entries only): the
//      CTA first copies the tile's force values with a one-cell halo ((T+1)^2 (TZ+1) x 3 floats in
//      padded rows, 66 KB) into shared memory with coalesced loads, then interpolates from shared memory.  The
//      tile index runs fastest along z, so neighbouring tiles (which share halos) run together.
// The order of particles inside a tile's list depends on atomic timing, but neither result does:
// integer sums are order independent and every particle's gather is computed on its own.
#include "cola_internal.h"

#include <cstdio>

namespace cola {
namespace {

constexpr int kThreads = 256;
// Tiles of T x T x TZ mesh cells.  The last tile of an axis is cut off where the mesh side is no multiple
// of the tile's, so that every mesh has tiles of the same shape (a 360^3 mesh with tiles of the largest
// power of two dividing its side, 8 x 8 x 8, took 399 us for the deposit and 161 us for the binning of
// 180^3 particles).  TZ = 64: a tile's particles come in runs of neighbours along the lattice's z, and a
// longer tile makes longer runs, so that a warp's 18 particle accesses touch fewer lines and its lanes
// fewer rows of the staged forces (TZ = 32: gather 616 against 531 us at 256^3/384^3, 5465 against
// 4730 us at 512^3/768^3, 762 against 630 us at 256^3/512^3).
constexpr int kLt = 3, kT = 1 << kLt, kLz = 6, kTz = 1 << kLz;
constexpr int kDepositThreads = 512, kGatherThreads = 512;
// Deposit accumulator columns of TZ + 1 cells: without the pad every column of a tile started on the
// same shared-memory bank, and a warp's lanes from two columns with equal z conflicted (24.4 against
// 26.7 ms at 1024^3/1536^3).
constexpr int kCol = kTz + 1;
constexpr int kAccWords = kT * kT * kCol;

int check_launch(const char* what) {
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) {
    std::fprintf(stderr, "cola: launch of %s failed: %s\n", what, cudaGetErrorString(e));
    return COLA_ERR_CUDA;
  }
  return COLA_OK;
}

// Bin entries hold the lattice coordinates packed as qx << 20 | qy << 10 | qz (np <= 1024).
__device__ __forceinline__ unsigned pack_q(int qx, int qy, int qz) {
  return ((unsigned)qx << 20) | ((unsigned)qy << 10) | (unsigned)qz;
}
__device__ __forceinline__ void unpack_q(unsigned e, int np, int* q, long long* id) {
  q[0] = (int)(e >> 20);
  q[1] = (int)((e >> 10) & 1023u);
  q[2] = (int)(e & 1023u);
  *id = ((long long)q[0] * np + q[1]) * np + q[2];
}

// warp-aggregated increment of counter[key] for the lanes whose key >= 0; returns the lane's slot
// (old value + rank among equal keys).
__device__ __forceinline__ unsigned agg_inc(unsigned* counter, int key) {
  const unsigned active = __activemask();
  const unsigned grp = __match_any_sync(active, key);
  const int lane = threadIdx.x & 31;
  const int leader = __ffs(grp) - 1;
  unsigned base = 0;
  if (key >= 0 && lane == leader) base = atomicAdd(counter + key, (unsigned)__popc(grp));
  base = __shfl_sync(grp, base, leader);
  return base + __popc(grp & ((1u << lane) - 1u));
}

// A particle's tile: its coordinates and which upper faces of the tile its base cell lies on (1: x,
// 2: y, 4: z), packed as flags << 25 | bx << 16 | by << 7 | bz (nt <= 512, nz <= 128).  Tile index
// (bx nt + by) nz + bz runs fastest along z.  With a single tile along an axis the cloud wraps inside
// the tile itself: no upper face there.
__device__ __forceinline__ unsigned tile_code(const BinGeom& b, int n, int cx, int cy, int cz) {
  const unsigned sx = b.nt > 1 && ((cx & (kT - 1)) == kT - 1 || cx == n - 1);
  const unsigned sy = b.nt > 1 && ((cy & (kT - 1)) == kT - 1 || cy == n - 1);
  const unsigned sz = b.nz > 1 && ((cz & (kTz - 1)) == kTz - 1 || cz == n - 1);
  return (sx << 25) | (sy << 26) | (sz << 27) | ((unsigned)(cx >> kLt) << 16) | ((unsigned)(cy >> kLt) << 7) |
         (unsigned)(cz >> kLz);
}
__device__ __forceinline__ unsigned code_flags(unsigned code) { return code >> 25; }
__device__ __forceinline__ int code_key(const BinGeom& b, unsigned code) {
  return (int)((((code >> 16) & 511u) * b.nt + ((code >> 7) & 511u)) * b.nz + (code & 127u));
}
// Calls f(key) for every other tile the cloud of a particle with upper faces reaches (at most seven):
// the non-empty subsets of its faces.  One face, the usual case, costs one turn.
template <class F>
__device__ __forceinline__ void for_spill_keys(const BinGeom& b, unsigned code, F&& f) {
  const unsigned flags = code_flags(code);
  const int bx = (code >> 16) & 511u, by = (code >> 7) & 511u, bz = code & 127u;
  const int key = (bx * b.nt + by) * b.nz + bz;
  const int col = b.nt * b.nz;
  const int dx = bx + 1 == b.nt ? -bx * col : col;
  const int dy = by + 1 == b.nt ? -by * b.nz : b.nz;
  const int dz = bz + 1 == b.nz ? -bz : 1;
  for (unsigned sub = flags; sub; sub = (sub - 1u) & flags)
    f(key + (sub & 1u ? dx : 0) + (sub & 2u ? dy : 0) + (sub & 4u ? dz : 0));
}

// Lattice row r of a walk over all rows (qx, qy), as a block's threads of one threadIdx.y take them: the
// planes in a scattered order (mul is coprime to np, a step of about 0.38 np), the rows of a plane in
// order.  Rows in flight together then belong to planes far apart and meet on fewer tile counters, while
// neighbouring rows still get neighbouring places in a tile's list, which the gather's accesses profit
// from.  32-bit divisions: 64-bit ones were about a third of both passes' instructions.
struct RowWalk {
  unsigned np, mul;
  __device__ __forceinline__ void at(unsigned r, int* qx, int* qy, long long* row) const {
    const unsigned p = r / np, y = r - p * np, x = (p * mul) % np;
    *qx = (int)x;
    *qy = (int)y;
    *row = ((long long)x * np + y) * np;
  }
};

// Count pass: per-tile primary and spill counts; every particle's rank within its primary tile (the
// aggregated atomic's return) is recorded with its tile code, so that the scatter pass needs neither the
// positions nor atomics for the primary entries: rec[id] = rank << 32 | code.
// Bound by instruction issue and by the atomics' return trips.
template <bool F32>
__global__ void __launch_bounds__(kThreads) k_bin_count(ParticleGeom pg, BinGeom b, FixedGeo fg, RowWalk walk,
                                                        const float* s, unsigned* cnt_p, unsigned* cnt_s,
                                                        unsigned long long* rec) {
  after_previous();
  const long long n = pg.npart;
  const int np = pg.np;
  const unsigned nrows = (unsigned)np * np, step = gridDim.x * blockDim.y;
  unsigned r = blockIdx.x * blockDim.y + threadIdx.y;
  int qz = threadIdx.x, qx = 0, qy = 0;
  long long row = 0;
  float p[3] = {0.f, 0.f, 0.f};
  auto load = [&](long long first, int z, float (&v)[3]) {
#pragma unroll
    for (int a = 0; a < 3; ++a) v[a] = z < np ? *(s + a * n + first + z) : 0.f;
  };
  if (r < nrows) {
    walk.at(r, &qx, &qy, &row);
    load(row, qz, p);
  }
  while (r < nrows) {
    // the next positions are loaded before this chunk's atomics, so the two latencies overlap; whole
    // warps walk the row together so that the warp-aggregated atomics see full warps
    unsigned rn = r;
    int zn = qz + (int)blockDim.x, qxn = qx, qyn = qy;
    long long rown = row;
    if (zn - (int)threadIdx.x >= np) {
      rn += step;
      zn = threadIdx.x;
      if (rn < nrows) walk.at(rn, &qxn, &qyn, &rown);
    }
    float pn[3] = {0.f, 0.f, 0.f};
    if (rn < nrows) load(rown, zn, pn);
    int key = -1;
    unsigned code = 0;
    if (qz < np) {
      int cx, cy, cz, f;
      cell_frac<F32>(qx, p[0], fg, &cx, &f);
      cell_frac<F32>(qy, p[1], fg, &cy, &f);
      cell_frac<F32>(qz, p[2], fg, &cz, &f);
      code = tile_code(b, pg.n, cx, cy, cz);
      key = code_key(b, code);
    }
    // primary keys are shared by runs of lanes: one aggregated atomic per run
    const unsigned rank = agg_inc(cnt_p, key);
    if (qz < np) rec[row + qz] = ((unsigned long long)rank << 32) | code;
    // spill keys are sparse: one atomic per entry (its result unused)
    for_spill_keys(b, code, [&](int k) { atomicAdd(cnt_s + k, 1u); });
    r = rn;
    qz = zn;
    qx = qxn;
    qy = qyn;
    row = rown;
#pragma unroll
    for (int a = 0; a < 3; ++a) p[a] = pn[a];
  }
}

// Scatter pass from the records: primary entries straight to offset + rank, spill entries through
// the spill cursors.  Bound by the latency of the records and of the offset lookups.
__global__ void __launch_bounds__(kThreads) k_bin_scatter(ParticleGeom pg, BinGeom b, RowWalk walk,
                                                          const unsigned long long* rec,
                                                          const unsigned* off_p, unsigned* cur_s,
                                                          unsigned* ent_p, unsigned* ent_s) {
  after_previous();
  const int np = pg.np;
  const unsigned nrows = (unsigned)np * np, step = gridDim.x * blockDim.y;
  constexpr int U = 2;   // records in flight per thread: their loads, then their offset lookups
  for (unsigned w = blockIdx.x * blockDim.y + threadIdx.y; w < nrows; w += step) {
    int qx, qy;
    long long row;
    walk.at(w, &qx, &qy, &row);
    for (int q0 = threadIdx.x; q0 < np; q0 += U * blockDim.x) {
      unsigned long long r[U];
      unsigned base[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int qz = q0 + u * (int)blockDim.x;
        r[u] = qz < np ? __ldcs(rec + row + qz) : 0ULL;
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int qz = q0 + u * (int)blockDim.x;
        base[u] = qz < np ? *(off_p + code_key(b, (unsigned)r[u])) : 0u;
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int qz = q0 + u * (int)blockDim.x;
        if (qz >= np) continue;
        const unsigned packed = pack_q(qx, qy, qz);
        ent_p[base[u] + (unsigned)(r[u] >> 32)] = packed;
        for_spill_keys(b, (unsigned)r[u], [&](int k) { ent_s[atomicAdd(cur_s + k, 1u)] = packed; });
      }
    }
  }
}

// Exclusive scan of one or two count arrays (the tiles' primary and spill counts) into offsets (length
// m+1) and, of the second, scatter cursors, in three coalesced phases: per-segment sums, a scan of the
// segment sums, per-segment scans.  Counts and offsets are read and written 16 bytes at a time where the
// arrays allow (they start on 256-byte boundaries).
constexpr int kScanThreads = 512;
constexpr int kScanSeg = kScanThreads * 8;   // counts per segment

__device__ __forceinline__ unsigned block_excl_scan(unsigned v, unsigned* total) {
  __shared__ unsigned wsum[kScanThreads / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  unsigned incl = v;
  for (int d = 1; d < 32; d <<= 1) {
    const unsigned o = __shfl_up_sync(0xffffffffu, incl, d);
    if (lane >= d) incl += o;
  }
  if (lane == 31) wsum[warp] = incl;
  __syncthreads();
  if (warp == 0) {
    unsigned w = lane < kScanThreads / 32 ? wsum[lane] : 0;
    for (int d = 1; d < 32; d <<= 1) {
      const unsigned o = __shfl_up_sync(0xffffffffu, w, d);
      if (lane >= d) w += o;
    }
    if (lane < kScanThreads / 32) wsum[lane] = w;
  }
  __syncthreads();
  const unsigned before = warp ? wsum[warp - 1] : 0;
  *total = wsum[kScanThreads / 32 - 1];
  __syncthreads();
  return before + incl - v;
}

// counts base + 8 tid .. + 7 (0 beyond m)
__device__ __forceinline__ void load8(const unsigned* cnt, int i0, int m, unsigned (&c)[8]) {
  if (i0 + 8 <= m) {
    const uint4 a = *reinterpret_cast<const uint4*>(cnt + i0), b = *reinterpret_cast<const uint4*>(cnt + i0 + 4);
    c[0] = a.x, c[1] = a.y, c[2] = a.z, c[3] = a.w, c[4] = b.x, c[5] = b.y, c[6] = b.z, c[7] = b.w;
  } else {
#pragma unroll
    for (int k = 0; k < 8; ++k) c[k] = i0 + k < m ? cnt[i0 + k] : 0u;
  }
}
// offsets of the counts c at base.. from run on, to off (and cur), and off[m] after the last
__device__ __forceinline__ void store8(unsigned run, const unsigned (&c)[8], int i0, int m, unsigned* off, unsigned* cur) {
  unsigned o[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    o[k] = run;
    run += c[k];
    if (i0 + k == m - 1) off[m] = run;
  }
  if (i0 + 8 <= m) {
    const uint4 a = make_uint4(o[0], o[1], o[2], o[3]), b = make_uint4(o[4], o[5], o[6], o[7]);
    *reinterpret_cast<uint4*>(off + i0) = a;
    *reinterpret_cast<uint4*>(off + i0 + 4) = b;
    if (cur) {
      *reinterpret_cast<uint4*>(cur + i0) = a;
      *reinterpret_cast<uint4*>(cur + i0 + 4) = b;
    }
  } else {
#pragma unroll
    for (int k = 0; k < 8; ++k)
      if (i0 + k < m) {
        off[i0 + k] = o[k];
        if (cur) cur[i0 + k] = o[k];
      }
  }
}

__global__ void __launch_bounds__(kScanThreads) k_scan_sums(const unsigned* cnt_p,
                                                           const unsigned* cnt_s, int m,
                                                           unsigned* seg_sums) {
  after_previous();
  const int list = blockIdx.y;
  unsigned c[8], v = 0;
  load8(list ? cnt_s : cnt_p, blockIdx.x * kScanSeg + threadIdx.x * 8, m, c);
#pragma unroll
  for (int k = 0; k < 8; ++k) v += c[k];
  unsigned tot;
  block_excl_scan(v, &tot);
  if (threadIdx.x == 0) seg_sums[list * gridDim.x + blockIdx.x] = tot;
}

__global__ void __launch_bounds__(kScanThreads) k_scan_segs(unsigned* seg_sums, int nseg) {
  after_previous();
  const int list = blockIdx.x;
  unsigned* ss = seg_sums + list * nseg;
  unsigned carry = 0;
  for (int b = 0; b < nseg; b += kScanThreads) {
    const unsigned v = b + (int)threadIdx.x < nseg ? ss[b + threadIdx.x] : 0;
    unsigned tot;
    const unsigned ex = block_excl_scan(v, &tot);
    if (b + (int)threadIdx.x < nseg) ss[b + threadIdx.x] = carry + ex;
    carry += tot;
  }
}

__global__ void __launch_bounds__(kScanThreads) k_scan_apply(const unsigned* cnt_p,
                                                            const unsigned* cnt_s, int m,
                                                            const unsigned* seg_sums, unsigned* off_p,
                                                            unsigned* off_s, unsigned* cur_s) {
  after_previous();
  const int list = blockIdx.y, i0 = blockIdx.x * kScanSeg + threadIdx.x * 8;
  // each thread scans 8 consecutive counts; the thread totals are scanned across the block
  unsigned c[8], v = 0, tot;
  load8(list ? cnt_s : cnt_p, i0, m, c);
#pragma unroll
  for (int k = 0; k < 8; ++k) v += c[k];
  const unsigned run = seg_sums[list * gridDim.x + blockIdx.x] + block_excl_scan(v, &tot);
  store8(run, c, i0, m, list ? off_s : off_p, list ? cur_s : nullptr);
}

// The scan in one launch for few segments: every block sums the counts before its segment itself (at
// most kScanOneSegs segments of 4096 counts) instead of two launches that do it once.
constexpr int kScanOneSegs = 16;
__global__ void __launch_bounds__(kScanThreads) k_scan_one(const unsigned* cnt_p,
                                                          const unsigned* cnt_s, int m, unsigned* off_p,
                                                          unsigned* off_s, unsigned* cur_s) {
  after_previous();
  const int list = blockIdx.y;
  const unsigned* cnt = list ? cnt_s : cnt_p;
  unsigned* off = list ? off_s : off_p;
  const int base = blockIdx.x * kScanSeg;
  unsigned v = 0, before, tot;
  for (int i = threadIdx.x; i < base; i += kScanThreads) v += cnt[i];
  block_excl_scan(v, &before);
  unsigned c[8];
  load8(cnt, base + threadIdx.x * 8, m, c);
  v = 0;
#pragma unroll
  for (int k = 0; k < 8; ++k) v += c[k];
  const unsigned run = before + block_excl_scan(v, &tot);
  store8(run, c, base + threadIdx.x * 8, m, off, list ? cur_s : nullptr);
}

// Tile-wise deposit.  The tile's primary and spill entries form one index range, so a CTA's threads run
// out of work together.  A cell's sum of weights (each at most 2^42) is kept as two 32-bit words, the low
// 21 bits of every weight and the rest, added by shared atomics whose result nobody reads: up to
// kDepositBatch contributions fit each word, after which the words are folded into 64-bit totals.  A
// particle adds to a cell once, so a batch of that many entries cannot overflow.
// Bound by the shared atomics.  The two-word sum with a carry (an atomic whose old value decides a second
// one) executed 510 instructions per 32 entries at 73% of the issue slots, with the atomics' return trips
// exposed.
constexpr unsigned kDepositBatch = 2047;
constexpr int kLoBits = 21;

// shared add of v at byte address a + OFF if p (a reduction: nothing comes back)
template <int OFF>
__device__ __forceinline__ void red_shared(unsigned a, unsigned v, bool p) {
  asm volatile("{\n .reg .pred q;\n setp.ne.u32 q, %2, 0;\n @q red.shared.add.u32 [%0 + %3], %1;\n}\n" ::"r"(a), "r"(v),
               "r"((unsigned)p), "n"(OFF)
               : "memory");
}

// adds the 8 weights of one entry that fall inside the tile (acc: shared address of the low words)
template <bool F32>
__device__ __forceinline__ void deposit_entry(const ParticleGeom& pg, const FixedGeo& fg, const float* s,
                                              unsigned e, int x0, int y0, int z0, unsigned acc) {
  const int nm = pg.n;
  const long long n = pg.npart;
  int q[3];
  long long id;
  unpack_q(e, pg.np, q, &id);
  int c[3], f[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) cell_frac<F32>(q[a], *(s + a * n + id), fg, &c[a], &f[a]);
  const int lx[2] = {c[0] - x0, (c[0] + 1 == nm ? 0 : c[0] + 1) - x0};
  const int ly[2] = {c[1] - y0, (c[1] + 1 == nm ? 0 : c[1] + 1) - y0};
  const int lz[2] = {c[2] - z0, (c[2] + 1 == nm ? 0 : c[2] + 1) - z0};
  const bool okz[2] = {(unsigned)lz[0] < (unsigned)kTz, (unsigned)lz[1] < (unsigned)kTz};
  const unsigned wz[2] = {(unsigned)(kWeightOne - f[2]), (unsigned)f[2]};
#pragma unroll
  for (int dx = 0; dx < 2; ++dx) {
    const unsigned wx = dx ? f[0] : kWeightOne - f[0];
    const bool okx = (unsigned)lx[dx] < (unsigned)kT;
#pragma unroll
    for (int dy = 0; dy < 2; ++dy) {
      const unsigned wxy = wx * (dy ? f[1] : kWeightOne - f[1]);   // <= 2^28
      const bool okxy = okx && (unsigned)ly[dy] < (unsigned)kT;
      const unsigned col = acc + 4u * (unsigned)((lx[dx] * kT + ly[dy]) * kCol);
#pragma unroll
      for (int dz = 0; dz < 2; ++dz) {
        const unsigned long long w = (unsigned long long)wxy * wz[dz];   // <= 2^42
        const unsigned a = col + 4u * (unsigned)lz[dz];
        const bool ok = okxy && okz[dz];
        red_shared<0>(a, (unsigned)w & ((1u << kLoBits) - 1u), ok);
        red_shared<4 * kAccWords>(a, (unsigned)(w >> kLoBits), ok);
      }
    }
  }
}

template <bool F32>
__global__ void __launch_bounds__(kDepositThreads, 4) k_deposit_tiles(ParticleGeom pg, BinGeom b, FixedGeo fg,
                                                               const float* s,
                                                               const unsigned* off_p,
                                                               const unsigned* ent_p,
                                                               const unsigned* off_s,
                                                               const unsigned* ent_s,
                                                               unsigned long long* rho, float* delta_out, float scale,
                                                               unsigned long long* tile_mass) {
  after_previous();
  __shared__ unsigned words[2 * kAccWords];
  unsigned* const lo = words;
  unsigned* const hi = words + kAccWords;
  const unsigned acc = (unsigned)__cvta_generic_to_shared(words);
  const int nm = pg.n;
  const int tile = blockIdx.x;
  const unsigned p0 = off_p[tile], np_t = off_p[tile + 1] - p0;
  const unsigned s0 = off_s[tile], total = np_t + (off_s[tile + 1] - s0);
  const int bz = tile % b.nz, bxy = tile / b.nz;
  const int bx = bxy / b.nt, by = bxy - bx * b.nt;
  const int x0 = bx << kLt, y0 = by << kLt, z0 = bz << kLz;
  for (int i = threadIdx.x; i < kAccWords; i += kDepositThreads) lo[i] = hi[i] = 0u;
  __syncthreads();
  constexpr int kCells = kT * kT * kTz / kDepositThreads;   // cells per thread, a column segment of one z each
  unsigned long long sum[kCells];
  bool folded = false;
  for (unsigned k0 = 0; k0 < total; k0 += kDepositBatch) {
    const unsigned k1 = total - k0 < kDepositBatch ? total : k0 + kDepositBatch;
    for (unsigned k = k0 + threadIdx.x; k < k1; k += kDepositThreads)
      deposit_entry<F32>(pg, fg, s, k < np_t ? ent_p[p0 + k] : ent_s[s0 + (k - np_t)], x0, y0, z0, acc);
    __syncthreads();
    if (k1 < total) {   // more to come: fold the words (a thread folds its own cells only)
#pragma unroll
      for (int i = 0; i < kCells; ++i) {
        const int j = threadIdx.x + i * kDepositThreads, a = (j >> kLz) * kCol + (j & (kTz - 1));
        const unsigned long long v = lo[a] + ((unsigned long long)hi[a] << kLoBits);
        sum[i] = folded ? sum[i] + v : v;
        lo[a] = hi[a] = 0u;
      }
      folded = true;
      __syncthreads();
    }
  }
  // the tile owns its cells: plain, coalesced stores of column segments; with delta_out the density
  // contrast, and the exact 128-bit total for the overflow check
  unsigned long long tlo = 0ULL, thi = 0ULL;
#pragma unroll
  for (int i = 0; i < kCells; ++i) {
    const int j = threadIdx.x + i * kDepositThreads, col = j >> kLz, z = j & (kTz - 1), a = col * kCol + z;
    const int gx = x0 + (col >> kLt), gy = y0 + (col & (kT - 1)), gz = z0 + z;
    if (gx < nm && gy < nm && gz < nm) {
      unsigned long long v = lo[a] + ((unsigned long long)hi[a] << kLoBits);
      if (folded) v += sum[i];
      const long long cell = ((long long)gx * nm + gy) * nm + gz;
      if (!delta_out) {
        rho[cell] = v;
      } else {
        tlo += v;
        thi += (tlo < v);
        delta_out[cell] = fixed_to_delta(v, scale);
      }
    }
  }
  if (!delta_out) return;
  // the CTA's total (warp shuffles, then the warps' partials in shared memory) and one slot update
  for (int off = 16; off > 0; off >>= 1) {
    const unsigned long long olo = __shfl_down_sync(0xffffffffu, tlo, off);
    const unsigned long long ohi = __shfl_down_sync(0xffffffffu, thi, off);
    tlo += olo;
    thi += ohi + (tlo < olo);
  }
  __shared__ unsigned long long wpart[2 * (kDepositThreads / 32)];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (lane == 0) {
    wpart[2 * warp] = tlo;
    wpart[2 * warp + 1] = thi;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    tlo = thi = 0ULL;
    for (int w = 0; w < kDepositThreads / 32; ++w) {
      tlo += wpart[2 * w];
      thi += wpart[2 * w + 1] + (tlo < wpart[2 * w]);
    }
    tile_mass[2 * blockIdx.x] = tlo;   // one pair per tile, no atomics; launch_mass_check sums them
    tile_mass[2 * blockIdx.x + 1] = thi;
  }
}

// Tile-wise gather (+ kick and drift) over the primary entries of each tile, from a shared copy
// of the tile's force values with a one-cell halo on the upper side of every axis: 3 components x
// (T+1)^2 rows of TZ + 1 floats, rows padded to kHp (16 bytes).
constexpr int kHx = kT + 1, kHp = (kTz + 1 + 3) & ~3;
constexpr int kGatherFloats = 3 * kHx * kHx * kHp;
constexpr int kBulkWaitLimit = 1 << 22;   // polls of the staging barrier before the CTA gives up

// Stage a tile's forces: one cp.async.bulk of the tile's z extent (64 cells, fewer in the last tile; a
// multiple of 4: the mesh side is, where this kernel runs) per force row, all completing on the mbarrier
// at bar_sa, plus each row's periodic halo cell by a 4-byte cp.async (committed as one group).  Rows start
// 16-byte aligned (z0 a multiple of 64, rows of 2 pc floats with pc even).  Called by every thread of the
// block; contains a barrier.
__device__ __forceinline__ void gather_stage(float* fsm, unsigned bar_sa, int nm, int x0, int y0, int z0,
                                             const float* f0, const float* f1,
                                             const float* f2, long long rs) {
  const int tx = nm - x0 < kT ? nm - x0 : kT, ty = nm - y0 < kT ? nm - y0 : kT, tz = nm - z0 < kTz ? nm - z0 : kTz;
  if (threadIdx.x == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(bar_sa) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    asm volatile("{\n .reg .b64 st;\n mbarrier.arrive.expect_tx.shared::cta.b64 st, [%0], %1;\n}\n" ::"r"(bar_sa),
                 "r"(3 * (tx + 1) * (ty + 1) * tz * 4)
                 : "memory");
  }
  __syncthreads();   // the barrier expects every row's bytes before any copy is issued
  const int gzz = z0 + tz == nm ? 0 : z0 + tz;
  for (int r = threadIdx.x; r < 3 * kHx * kHx; r += kGatherThreads) {
    const int comp = r / (kHx * kHx), col = r - comp * kHx * kHx;
    const int lx = col / kHx, ly = col - lx * kHx;
    if (lx > tx || ly > ty) continue;   // beyond a cut-off tile's halo
    const int gx = x0 + lx == nm ? 0 : x0 + lx, gy = y0 + ly == nm ? 0 : y0 + ly;
    const float* f = comp == 0 ? f0 : (comp == 1 ? f1 : f2);
    const float* row = f + ((long long)gx * nm + gy) * rs;
    const unsigned sa = (unsigned)__cvta_generic_to_shared(fsm + r * kHp);
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(sa),
                 "l"(row + z0), "r"(tz * 4), "r"(bar_sa)
                 : "memory");
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(sa + 4u * tz), "l"(row + gzz) : "memory");
  }
  asm volatile("cp.async.commit_group;\n" ::: "memory");
}

// Bounded wait for phase `parity` of the mbarrier at bar_sa; false if the limit was reached.
__device__ __forceinline__ bool bulk_wait(unsigned bar_sa, unsigned parity) {
  for (int it = 0; it < kBulkWaitLimit; ++it) {
    unsigned done;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(done)
        : "r"(bar_sa), "r"(parity)
        : "memory");
    if (done) return true;
  }
  return false;
}

// The values of one particle that the gather reads.
template <bool KICK>
struct GatherPart {
  unsigned e;
  float s[3], v[3], p1[3], p2[3];
  __device__ __forceinline__ void load(const ParticleGeom& pg, unsigned ent, const float* sp, const float* vp,
                                       const float* psi1, const float* psi2) {
    e = ent;
    int q[3];
    long long id;
    unpack_q(ent, pg.np, q, &id);
    const long long n = pg.npart;
#pragma unroll
    for (int a = 0; a < 3; ++a) s[a] = sp[a * n + id];
    if (KICK) {
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        p1[a] = *(psi1 + a * n + id);
        p2[a] = *(psi2 + a * n + id);
        v[a] = vp[a * n + id];
      }
    }
  }
};

// One CTA per tile.  Bound by the latency of its dependent loads (tile offsets, entries, particles): the
// forces are staged and the first particles' values loaded at the same time, and each later particle's
// entry and values are loaded while the one before is interpolated.
template <bool KICK, bool F32>
__global__ void __launch_bounds__(kGatherThreads, 2) k_gather_tiles(ParticleGeom pg, BinGeom b, FixedGeo fg,
                                                             const unsigned* off_p,
                                                             const unsigned* ent_p,
                                                             const float* f0, const float* f1,
                                                             const float* f2, long long rs,
                                                             const float* s_in, float* force_out,
                                                             float* s, float* v, const float* psi1,
                                                             const float* psi2, KickDrift kd, int* flags) {
  after_previous();
  extern __shared__ __align__(16) float fsm[];
  const int tile = blockIdx.x;
  const unsigned e0 = off_p[tile], e1 = off_p[tile + 1];
  if (e0 == e1) return;                          // empty (uniform across the block)
  const int bz = tile % b.nz, bxy = tile / b.nz;
  const int bx = bxy / b.nt, by = bxy - bx * b.nt;
  const int x0 = bx << kLt, y0 = by << kLt, z0 = bz << kLz;
  const unsigned bar_sa = (unsigned)__cvta_generic_to_shared(fsm + kGatherFloats);
  const float* sp = KICK ? s : s_in;
  const unsigned first = e0 + threadIdx.x;
  unsigned ent = first < e1 ? *(ent_p + first) : 0u;
  unsigned ent_next = first + kGatherThreads < e1 ? *(ent_p + first + kGatherThreads) : 0u;
  gather_stage(fsm, bar_sa, pg.n, x0, y0, z0, f0, f1, f2, rs);
  GatherPart<KICK> cur;
  if (first < e1) cur.load(pg, ent, sp, v, psi1, psi2);
  asm volatile("cp.async.wait_group 0;\n" ::: "memory");
  const bool ok = bulk_wait(bar_sa, 0);
  if (__syncthreads_or(!ok)) {
    // the staging never completed (not expected): report, give the copies one more bounded wait, stop
    if (threadIdx.x == 0) atomicOr(flags, 4);
    bulk_wait(bar_sa, 0);
    return;
  }
  if (threadIdx.x == 0) asm volatile("mbarrier.inval.shared::cta.b64 [%0];\n" ::"r"(bar_sa) : "memory");
  const long long n = pg.npart;
  const float inv_one = 1.0f / kWeightOne;
  bool bad = false;
  for (unsigned e = first; e < e1; e += kGatherThreads) {
    GatherPart<KICK> nxt;
    if (e + kGatherThreads < e1) nxt.load(pg, ent_next, sp, v, psi1, psi2);
    ent_next = e + 2 * kGatherThreads < e1 ? *(ent_p + e + 2 * kGatherThreads) : 0u;
    int q[3], c[3];
    long long id;
    unpack_q(cur.e, pg.np, q, &id);
    float w1[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      int f;
      cell_frac<F32>(q[a], cur.s[a], fg, &c[a], &f);
      w1[a] = (float)f * inv_one;
    }
    const int lx = c[0] - x0, ly = c[1] - y0, lz = c[2] - z0;   // base cell inside the tile
    float fr[3] = {0.f, 0.f, 0.f};
#pragma unroll
    for (int dx = 0; dx < 2; ++dx) {
      const float wx = dx ? w1[0] : 1.0f - w1[0];
#pragma unroll
      for (int dy = 0; dy < 2; ++dy) {
        const float wxy = wx * (dy ? w1[1] : 1.0f - w1[1]);
        const int o = ((lx + dx) * kHx + (ly + dy)) * kHp + lz;
#pragma unroll
        for (int comp = 0; comp < 3; ++comp) {
          const float* p = fsm + comp * (kHx * kHx * kHp) + o;
          fr[comp] += wxy * ((1.0f - w1[2]) * p[0] + w1[2] * p[1]);
        }
      }
    }
    if (!KICK) {
      force_out[id] = fr[0];
      force_out[n + id] = fr[1];
      force_out[2 * n + id] = fr[2];
    } else {
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        const float p1 = cur.p1[a], p2 = cur.p2[a];
        const float fres = fr[a] - (kd.c1 * p1 + kd.c2 * p2);
        const float vn = cur.v[a] + kd.kick * fres;
        const float sn = cur.s[a] + kd.drift * vn + kd.dd1 * p1 + kd.dd2 * p2;
        v[a * n + id] = vn;
        s[a * n + id] = sn;
        bad |= !isfinite(vn) || !isfinite(sn);
      }
    }
    cur = nxt;
  }
  if (KICK && __syncthreads_or(bad) && threadIdx.x == 0) atomicOr(flags, 2);
}

}  // namespace

bool bin_geometry(int nmesh, int np, BinGeom* b) {
  if (np > 1024) return false;                       // packed 10-bit lattice coordinates
  b->nt = (nmesh + kT - 1) >> kLt;
  b->nz = (nmesh + kTz - 1) >> kLz;
  b->tiles = b->nt * b->nt * b->nz;                  // <= 2^25 (nmesh <= 4096)
  b->bulk = nmesh % 4 == 0;
  return true;
}

// Where the binned deposit and the tile gather pay (us per COLA step, direct / binned + direct gather /
// binned + tile gather, r = mesh side over particle side):
//   192^3: r = 1 759/973/832, 1.5 359/407/368, 2 267/308/293;  216^3: 1086/1191/973, 521/566/508, 380/408/393;
//   240^3: 1390/1480/1195, 679/697/614, 487/495/477;  384^3: 5707/5664/4291, 2649/2506/2157, 1946/1820/1691;
//   r = 3, 288^3 651/670/687, 384^3 1519/1431/1470, 480^3 2914/2794/2884.
// A direct deposit's atomics run in L2 while the 64-bit mesh fits beside what else is there (72 MB, 208^3).
// Above that dense tiles (256 particles on average, r up to 2.5) pay for the binning and the staging;
// sparse ones for the binning alone, once the mesh is some twice the L2.
void particle_schedule(const BinGeom& b, int nmesh, long long npart, bool* binned, bool* tile_gather) {
  const double mesh_mb = 8e-6 * nmesh * nmesh * nmesh;
  *tile_gather = b.bulk && mesh_mb > 72.0 && npart >= 256LL * b.tiles;
  *binned = *tile_gather || mesh_mb > 256.0;
}

int launch_excl_scan(const unsigned* cnt, int m, unsigned* seg, unsigned* off, cudaStream_t st) {
  const int nseg = (m + kScanSeg - 1) / kScanSeg;
  launch_after(k_scan_sums, dim3(nseg, 1), kScanThreads, 0, st, cnt, nullptr, m, seg);
  launch_after(k_scan_segs, 1, kScanThreads, 0, st, seg, nseg);
  launch_after(k_scan_apply, dim3(nseg, 1), kScanThreads, 0, st, cnt, nullptr, m, seg, off, nullptr, nullptr);
  return check_launch("excl_scan");
}

int launch_binning(const ParticleGeom& pg, const BinGeom& b, const float* s, BinBuffers& bb, cudaStream_t st) {
  const RowBlocks rb = row_blocks(pg.np);
  const unsigned blocks = rb.grid.x * rb.grid.y, grid = blocks < 152u * 64u ? blocks : 152u * 64u;
  unsigned mul = (unsigned)(0.382 * pg.np) | 1u;   // np has no prime factor above 5
  while (mul % 3 == 0 || mul % 5 == 0) mul += 2;
  const RowWalk walk{(unsigned)pg.np, mul};
  const FixedGeo fg = fixed_geo(pg.n, pg.r_fixed);
  // the two count arrays are adjacent: one clear of both
  if (cudaMemsetAsync(bb.cnt_p, 0, (size_t)(bb.cnt_s - bb.cnt_p + b.tiles) * sizeof(unsigned), st) != cudaSuccess)
    return COLA_ERR_CUDA;
  auto* count = pg.n < 2048 ? k_bin_count<true> : k_bin_count<false>;
  launch_after(count, grid, rb.block, 0, st, pg, b, fg, walk, s, bb.cnt_p, bb.cnt_s, bb.rec);
  int e = check_launch("bin_count");
  if (e != COLA_OK) return e;
  const int nseg = (b.tiles + kScanSeg - 1) / kScanSeg;
  if (nseg <= kScanOneSegs) {
    launch_after(k_scan_one, dim3(nseg, 2), kScanThreads, 0, st, bb.cnt_p, bb.cnt_s, b.tiles, bb.off_p, bb.off_s, bb.cur_s);
  } else {
    launch_after(k_scan_sums, dim3(nseg, 2), kScanThreads, 0, st, bb.cnt_p, bb.cnt_s, b.tiles, bb.seg);
    launch_after(k_scan_segs, 2, kScanThreads, 0, st, bb.seg, nseg);
    launch_after(k_scan_apply, dim3(nseg, 2), kScanThreads, 0, st, bb.cnt_p, bb.cnt_s, b.tiles, bb.seg, bb.off_p, bb.off_s, bb.cur_s);
  }
  if ((e = check_launch("bin_scan")) != COLA_OK) return e;
  launch_after(k_bin_scatter, grid, rb.block, 0, st, pg, b, walk, bb.rec, bb.off_p, bb.cur_s, bb.ent_p, bb.ent_s);
  return check_launch("bin_scatter");
}

int launch_deposit_tiles(const ParticleGeom& pg, const BinGeom& b, const float* s, const BinBuffers& bb,
                         unsigned long long* rho, cudaStream_t st, float* delta_out, float scale,
                         unsigned long long* tile_mass) {
  if (delta_out && !tile_mass) return COLA_ERR_INVALID;
  const FixedGeo fg = fixed_geo(pg.n, pg.r_fixed);
  auto* k = pg.n < 2048 ? k_deposit_tiles<true> : k_deposit_tiles<false>;
  launch_after(k, b.tiles, kDepositThreads, 0, st, pg, b, fg, s, bb.off_p, bb.ent_p, bb.off_s, bb.ent_s, rho, delta_out, scale, tile_mass);
  return check_launch("deposit_tiles");
}

namespace {
constexpr int kGatherSmem = kGatherFloats * (int)sizeof(float) + 16;   // + mbarrier
template <class K>
void gather_smem_limit(K kernel) {
  once_on_device(reinterpret_cast<const void*>(kernel), [](const void* k) {
    cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, kGatherSmem);
  });
}
}  // namespace

int launch_gather_tiles(const ParticleGeom& pg, const BinGeom& b, const BinBuffers& bb, const float* const f[3],
                        long long rs, const float* s_in, float* force_out, float* s, float* v, const float* psi1,
                        const float* psi2, const KickDrift* kd, int* flags, cudaStream_t st) {
  if (!b.bulk) return COLA_ERR_INVALID;   // 16-byte staging copies along z
  const FixedGeo fg = fixed_geo(pg.n, pg.r_fixed);
  const bool f32 = pg.n < 2048;
  if (kd) {
    auto* k = f32 ? k_gather_tiles<true, true> : k_gather_tiles<true, false>;
    gather_smem_limit(k);
    launch_after(k, b.tiles, kGatherThreads, kGatherSmem, st, pg, b, fg, bb.off_p, bb.ent_p, f[0], f[1], f[2], rs, nullptr, nullptr, s, v, psi1, psi2, *kd, flags);
  } else {
    auto* k = f32 ? k_gather_tiles<false, true> : k_gather_tiles<false, false>;
    gather_smem_limit(k);
    launch_after(k, b.tiles, kGatherThreads, kGatherSmem, st, pg, b, fg, bb.off_p, bb.ent_p, f[0], f[1], f[2], rs, s_in, force_out, nullptr, nullptr, nullptr, nullptr, KickDrift{}, flags);
  }
  return check_launch("gather_tiles");
}

}  // namespace cola
