// expansion_mi.cuh -- multi-indices of the general-order expansion.
#pragma once

namespace amfmm {

constexpr int kMaxP = 8;

// Position of (a0, a1, a2): those of order n start at n (n+1) (n+2) / 6, ordered
// a0 = n..0 and then a1 = n - a0 .. 0.
__host__ __device__ constexpr int mi_off(int n) { return n * (n + 1) * (n + 2) / 6; }
__host__ __device__ constexpr int mi_idx(int a0, int a1, int a2) {
  const int n = a0 + a1 + a2, s = a1 + a2;
  return mi_off(n) + s * (s + 1) / 2 + a2;
}

struct MultiIndices {
  unsigned char a[mi_off(kMaxP + 1)][4];  // a0, a1, a2, order
  double fact[mi_off(kMaxP + 1)], inv_fact[mi_off(kMaxP + 1)];  // a!, 1 / a!
};
constexpr MultiIndices make_multi_indices() {
  MultiIndices t{};
  double f[kMaxP + 1] = {1.0};
  for (int n = 1; n <= kMaxP; ++n) f[n] = n * f[n - 1];
  int i = 0;
  for (int n = 0; n <= kMaxP; ++n)
    for (int a0 = n; a0 >= 0; --a0)
      for (int a1 = n - a0; a1 >= 0; --a1, ++i) {
        const int a2 = n - a0 - a1;
        t.a[i][0] = static_cast<unsigned char>(a0);
        t.a[i][1] = static_cast<unsigned char>(a1);
        t.a[i][2] = static_cast<unsigned char>(a2);
        t.a[i][3] = static_cast<unsigned char>(n);
        t.fact[i] = f[a0] * f[a1] * f[a2];
        t.inv_fact[i] = 1.0 / (f[a0] * f[a1] * f[a2]);
      }
  return t;
}

// Reduced indices.  The derivatives D^g of 1/R and every local expansion made of
// them satisfy D^(g+2x) + D^(g+2y) + D^(g+2z) = 0, so those with g_z <= 1
// determine all others:  D^(t,u,s+2q) = (-1)^q sum_j C(q,j) D^(t+2j,u+2(q-j),s).
// An order n has 2n + 1 of them, from position n^2: (n-u, u, 0), u = 0..n, then
// (n-1-u, u, 1), u = 0..n-1.
__host__ __device__ constexpr int red_idx(int t, int u, int s) {
  const int n = t + u + s;
  return n * n + (s ? n + 1 : 0) + u;
}
__host__ __device__ constexpr int choose(int n, int k) {
  int c = 1;
  for (int i = 1; i <= k; ++i) c = c * (n - k + i) / i;
  return c;
}
// doubles per slot of reduced locals (orders 1..P) and per cell of reduced
// moments (orders 0..P), both rounded up to whole 16-byte words
__host__ __device__ constexpr int red_loc_stride(int P) { return ((P + 1) * (P + 1)) & ~1; }
__host__ __device__ constexpr int red_mom_stride(int P) { return ((P + 1) * (P + 1) + 1) & ~1; }

}  // namespace amfmm
