// down.cu -- a9: downward pass.  The local expansion of a cell, written about
// its centre of mass Z (Eqs. 3 and 4 are polynomials in the offset from Z), is
// the sum of its own interactions and its parent's expansion shifted to Z
// (L2L, exact for a polynomial): with s = Z_child - Z_parent,
//     C_i'   = C_i + C_ij s_j + C_ijk s_j s_k / 2
//     C_ij'  = C_ij + C_ijk s_k
//     C_ijk' = C_ijk.
// Every body of a leaf then receives a = -(C_i + C_ij x_j + C_ijk x_j x_k / 2)
// with x = X - Z_leaf (L2P), plus its near-field sum; fmm_forces scatters the
// result to the caller's order and multiplies by G.
#include "internal.cuh"

namespace amfmm {
namespace {

// symmetric index helpers for the local layout
// C_ij: xx xy xz yy yz zz -> 3..8 ; C_ijk: xxx xxy xxz xyy xyz xzz yyy yyz yzz zzz -> 9..18
__device__ __forceinline__ int i2(int i, int j) {
  const int a = min(i, j), b = max(i, j);
  return a == 0 ? b : (a == 1 ? 2 + b : 5);
}
__device__ __forceinline__ int i3(int i, int j, int k) {
  // sort the three indices
  int a = i, b = j, c = k, t;
  if (a > b) { t = a; a = b; b = t; }
  if (b > c) { t = b; b = c; c = t; }
  if (a > b) { t = a; a = b; b = t; }
  if (a == 0) {
    if (b == 0) return c;          // xxx xxy xxz
    if (b == 1) return 2 + c;      // xyy xyz
    return 5;                      // xzz
  }
  if (a == 1) return b == 1 ? 5 + c : 8;  // yyy yyz | yzz
  return 9;                               // zzz
}

// With h_ij = C_ijk s_k:  C_i' = C_i + (C_ij + h_ij / 2) s_j.  Both kernels spell out
// every operation, so that it makes no difference which of them takes a level (it
// follows from the number of cells, in a forest of all systems).
__device__ __forceinline__ double dot3(double a0, double a1, double a2, double s0, double s1, double s2) {
  return fma(a2, s2, fma(a1, s1, __dmul_rn(a0, s0)));
}

// A thread per child where a level fills the GPU: 58 FP64 instructions for 32
// children.  An FP64 instruction holds its pipe for 64 cycles whatever number
// of lanes work, so on a small level those 58 are a chain of 2 us; there a
// warp takes one child, a lane per coefficient, with a chain of 9.
__global__ void k_l2l(int32_t c0, int32_t c1, const int32_t *parent,
                      const double *Z, double *__restrict__ loc) {
  pdl_wait();
  const int c = c0 + blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= c1) return;
  const int p = parent[c];
  const double s[3] = {Z[3 * c] - Z[3 * p], Z[3 * c + 1] - Z[3 * p + 1], Z[3 * c + 2] - Z[3 * p + 2]};
  const double *P = loc + static_cast<int64_t>(p) * kLocStride;
  double *C = loc + static_cast<int64_t>(c) * kLocStride;
  double Pl[19], h[6];
#pragma unroll
  for (int q = 0; q < 19; ++q) Pl[q] = P[q];
#pragma unroll
  for (int q = 0; q < 10; ++q) C[9 + q] += Pl[9 + q];
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = i; j < 3; ++j) {
      const int q = i2(i, j);
      h[q] = dot3(Pl[9 + i3(i, j, 0)], Pl[9 + i3(i, j, 1)], Pl[9 + i3(i, j, 2)], s[0], s[1], s[2]);
      C[3 + q] = __dadd_rn(C[3 + q], __dadd_rn(Pl[3 + q], h[q]));
      h[q] = fma(0.5, h[q], Pl[3 + q]);
    }
#pragma unroll
  for (int i = 0; i < 3; ++i)
    C[i] = __dadd_rn(C[i], __dadd_rn(Pl[i], dot3(h[i2(i, 0)], h[i2(i, 1)], h[i2(i, 2)], s[0], s[1], s[2])));
}

constexpr int kL2LWarps = 4;

__global__ void __launch_bounds__(kL2LWarps * 32) k_l2l_warp(int32_t c0, int32_t c1,
                                                             const int32_t *parent,
                                                             const double *Z, double *__restrict__ loc) {
  pdl_wait();
  __shared__ double sp[kL2LWarps][kLocStride], sh[kL2LWarps][6];
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  const int c = c0 + blockIdx.x * kL2LWarps + w;
  if (c >= c1) return;  // whole warp
  const int p = parent[c];
  double own = 0.0, up = 0.0;
  if (l < 19) {
    own = loc[static_cast<int64_t>(c) * kLocStride + l];
    sp[w][l] = up = loc[static_cast<int64_t>(p) * kLocStride + l];
  }
  double s = 0.0;
  if (l < 3) s = Z[3 * c + l] - Z[3 * p + l];
  const double s0 = __shfl_sync(0xffffffffu, s, 0), s1 = __shfl_sync(0xffffffffu, s, 1),
               s2 = __shfl_sync(0xffffffffu, s, 2);
  __syncwarp();
  const int q = l - 3;                             // this lane's C_ij
  const int i = q < 3 ? 0 : q < 5 ? 1 : 2;
  const int j = q < 3 ? q : q < 5 ? q - 2 : 2;
  if (q >= 0 && q < 6) {
    const double h = dot3(sp[w][9 + i3(i, j, 0)], sp[w][9 + i3(i, j, 1)], sp[w][9 + i3(i, j, 2)], s0, s1, s2);
    sh[w][q] = fma(0.5, h, up);
    up = __dadd_rn(up, h);
  }
  __syncwarp();
  if (l < 3) up = __dadd_rn(up, dot3(sh[w][i2(l, 0)], sh[w][i2(l, 1)], sh[w][i2(l, 2)], s0, s1, s2));
  if (l < 19) loc[static_cast<int64_t>(c) * kLocStride + l] = __dadd_rn(own, up);
}

// (39 FP64 operations per body through the contraction with x / 2, 68 us at N =
// 1M; 127 us with every product x_j x_k x_ijk formed on its own)
__global__ void k_l2p(int64_t n, const int32_t *leaf_of, const double *Z,
                      const double *loc, const double *X,
                      const double *Y, const double *Zb,
                      const double *near, double *__restrict__ acc) {
  pdl_wait();
  const int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
  if (i >= n) return;
  const int L = leaf_of[i];
  const double x[3] = {X[i] - Z[3 * L], Y[i] - Z[3 * L + 1], Zb[i] - Z[3 * L + 2]};
  const double2 *Cp = reinterpret_cast<const double2 *>(loc + static_cast<int64_t>(L) * kLocStride);
  double C[kLocStride];
#pragma unroll
  for (int q = 0; q < kLocStride / 2; ++q) {
    const double2 v = Cp[q];
    C[2 * q] = v.x;
    C[2 * q + 1] = v.y;
  }
  // with y = x / 2:  C_i + (C_ij + C_ijk y_k) x_j
  const double y[3] = {0.5 * x[0], 0.5 * x[1], 0.5 * x[2]};
  double h[6];
#pragma unroll
  for (int d = 0; d < 3; ++d)
#pragma unroll
    for (int j = d; j < 3; ++j) {
      double v = C[3 + i2(d, j)];
#pragma unroll
      for (int k = 0; k < 3; ++k) v = fma(C[9 + i3(d, j, k)], y[k], v);
      h[i2(d, j)] = v;
    }
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    double v = C[d];
#pragma unroll
    for (int j = 0; j < 3; ++j) v = fma(h[i2(d, j)], x[j], v);
    acc[d * n + i] = near[d * n + i] - v;
  }
}

__global__ void k_unpermute(int64_t n, const int32_t *order, const double *acc,
                            double G, double *__restrict__ ax, double *__restrict__ ay,
                            double *__restrict__ az) {
  pdl_wait();
  const int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
  if (i >= n) return;
  const int o = order[i];
  ax[o] = G * acc[i];
  ay[o] = G * acc[n + i];
  az[o] = G * acc[2 * n + i];
}

}  // namespace

int downward(fmm_ctx *c) {
  const int64_t n = c->sz.n;
  AMFMM_TRY(ensure<double>(c, c->acc, 3 * n));
  if (c->opts.order_P != 3) return downward_general(c);
  const int64_t fill = std::max(1, c->num_sms);
  for (int lev = 1; lev <= c->sz.depth; ++lev) {
    const int64_t c0 = c->sz.lvl_off[lev], c1 = c->sz.lvl_off[lev + 1];
    if (c1 <= c0) continue;
    const bool many = c1 - c0 >= 16 * fill;  // then a thread per child has fewer instructions in all
    const auto down = many ? k_l2l : k_l2l_warp;
    const int threads = many ? 128 : kL2LWarps * 32;
    launch(c, down, grid_for(c1 - c0, many ? 128 : kL2LWarps), threads, 0, static_cast<int32_t>(c0),
           static_cast<int32_t>(c1), ptr<int32_t>(c->parent), ptr<double>(c->Z), ptr<double>(c->loc));
    AMFMM_TRY(launched(c, "l2l"));
  }
  launch(c, k_l2p, grid_for(n, 256), 256, 0, n, ptr<int32_t>(c->leaf_of), ptr<double>(c->Z), ptr<double>(c->loc),
         ptr<double>(c->X), ptr<double>(c->Y), ptr<double>(c->Zb), ptr<double>(c->near), ptr<double>(c->acc));
  return launched(c, "l2p");
}

int forces(fmm_ctx *c, double *ax, double *ay, double *az) {
  const int64_t n = c->sz.n;
  launch(c, k_unpermute, grid_for(n, 256), 256, 0, n, ptr<int32_t>(c->order), ptr<double>(c->acc), c->opts.G, ax, ay,
         az);
  return launched(c, "unpermute");
}

}  // namespace amfmm
