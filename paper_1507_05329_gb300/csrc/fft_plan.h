// Radix plans of the FFT passes, evaluated at compile time by the kernels of a length and at run time
// by the host (twiddle tables).
//
// A length is a product of elementary Stockham stages (factor_radices).  Adjacent stages whose product
// is at most 16 form one group: a thread that holds the R1 R2 values of both runs them back to back in
// registers, with the same butterflies and twiddles as two separate stages and one pass over shared
// memory fewer (360 = 8 5 3 3 runs as 8, 5, 3x3; 1000 = 8 5 5 5 is the longest, with four groups).
#pragma once

#ifdef __CUDACC__
#define COLA_HOST_DEVICE __host__ __device__
#else
#define COLA_HOST_DEVICE
#endif

namespace cola {

constexpr int kMaxStages = 12;

struct Radices {
  int m = 0;
  int r[kMaxStages] = {};
  bool ok = false;
};

// 2^a 3^b 5^c into stages: the powers of two first, in the fewest stages of radix <= 16, as even as
// possible, then the fives, then the threes.  One factor 3 and no 5: when the powers of two would need
// one stage more for their last factor 2 (a = 1 mod 4, e.g. 1536 = 8 8 8 3), that 2 joins the 3 in a
// last radix-6 stage (16 16 6).
constexpr Radices factor_radices(int n) {
  Radices out;
  if (n < 2) return out;
  int m = n, p2 = 0, n5 = 0, n3 = 0;
  while (m % 2 == 0) { m /= 2; ++p2; }
  while (m % 5 == 0) { m /= 5; ++n5; }
  while (m % 3 == 0) { m /= 3; ++n3; }
  if (m != 1) return out;
  const bool radix6 = n3 == 1 && n5 == 0 && p2 % 4 == 1;
  if (radix6) {
    --p2;
    n3 = 0;
  }
  const int nst = (p2 + 3) / 4;
  if (nst + n5 + n3 + (radix6 ? 1 : 0) > kMaxStages) return out;
  int left = p2;
  for (int s = 0; s < nst; ++s) {
    const int e = (left + (nst - s) - 1) / (nst - s);
    out.r[out.m++] = 1 << e;
    left -= e;
  }
  for (int i = 0; i < n5; ++i) out.r[out.m++] = 5;
  for (int i = 0; i < n3; ++i) out.r[out.m++] = 3;
  if (radix6) out.r[out.m++] = 6;
  out.ok = true;
  return out;
}

constexpr int kMaxGroups = 6;
constexpr int kMaxGroupRadix = 16;

// Groups of a length's stages: radices r1 x r2 (r2 = 1: a single stage), the product ns of the radices
// before the group, and the offsets of its stages' twiddles in the length's stage-major table
// (stage_twiddle): entry off + (r - 1) ns_stage + k is exp(-2 pi i r k / (ns_stage R)), n - 1 entries in
// all.  rev: the same groups in reverse order (the inverse transforms of the Green pass, whose first
// group then reads the registers the forward's last group wrote).
struct Groups {
  int n = 0, m = 0;
  int r1[kMaxGroups] = {}, r2[kMaxGroups] = {}, ns[kMaxGroups] = {}, off1[kMaxGroups] = {}, off2[kMaxGroups] = {};
  int max_radix = 0;
  bool ok = false;
};

constexpr Groups make_groups(int n, bool rev) {
  Groups g;
  g.n = n;
  const Radices f = factor_radices(n);
  if (!f.ok) return g;
  // fewest groups, then the smallest sum of squared group radices (even groups), from the last stage back
  int cnt[kMaxStages + 1] = {}, sq[kMaxStages + 1] = {}, take[kMaxStages + 1] = {};
  for (int i = f.m - 1; i >= 0; --i) {
    cnt[i] = cnt[i + 1] + 1;
    sq[i] = sq[i + 1] + f.r[i] * f.r[i];
    take[i] = 1;
    if (i + 1 < f.m) {
      const int p = f.r[i] * f.r[i + 1], c2 = cnt[i + 2] + 1, s2 = sq[i + 2] + p * p;
      if (p <= kMaxGroupRadix && (c2 < cnt[i] || (c2 == cnt[i] && s2 < sq[i]))) {
        cnt[i] = c2;
        sq[i] = s2;
        take[i] = 2;
      }
    }
  }
  if (cnt[0] > kMaxGroups) return g;
  for (int i = 0; i < f.m; i += take[i]) {
    g.r1[g.m] = f.r[i];
    g.r2[g.m] = take[i] == 2 ? f.r[i + 1] : 1;
    ++g.m;
  }
  if (rev) {
    for (int i = 0; i < g.m / 2; ++i) {
      const int a = g.r1[i], b = g.r2[i], j = g.m - 1 - i;
      g.r1[i] = g.r1[j];
      g.r2[i] = g.r2[j];
      g.r1[j] = a;
      g.r2[j] = b;
    }
  }
  int ns = 1, off = 0;
  for (int i = 0; i < g.m; ++i) {
    g.ns[i] = ns;
    g.off1[i] = off;
    off += (g.r1[i] - 1) * ns;
    ns *= g.r1[i];
    g.off2[i] = off;
    off += (g.r2[i] - 1) * ns;
    ns *= g.r2[i];
    const int r = g.r1[i] * g.r2[i];
    if (r > g.max_radix) g.max_radix = r;
  }
  g.ok = true;
  return g;
}

// Index t (of exp(-2 pi i t / n)) of entry e of the stage-major twiddle table of g, 0 <= e < n - 1.
COLA_HOST_DEVICE constexpr int stage_twiddle(const Groups& g, int e) {
  for (int i = 0; i < g.m; ++i) {
    const int ns = g.ns[i], n1 = ns * g.r1[i];
    if (e < g.off2[i]) {
      const int r = (e - g.off1[i]) / ns + 1, k = (e - g.off1[i]) % ns;
      return r * k * (g.n / n1);
    }
    if (e < g.off2[i] + (g.r2[i] - 1) * n1) {
      const int r = (e - g.off2[i]) / n1 + 1, k = (e - g.off2[i]) % n1;
      return r * k * (g.n / (n1 * g.r2[i]));
    }
  }
  return 0;
}

}  // namespace cola
