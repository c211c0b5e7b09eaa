// expansion.cu -- a7': the general-order expansion of App. A on the GPU, orders
// P = 4 .. 8, FP64, on the tree, walk and near field of the order-3 path.  In
// multi-index notation (a, b, g exponent triples, |a| the order, a! the product
// of the factorials):
//   P2M: M^a = sum mu x^a about each leaf's centre of mass
//   M2M: M^a += sum_{b<=a} C(a,b) M_child^b s^(a-b), s = Z_child - Z
//   M2L: expansion_m2l.cu
//   L2L: L'^a += sum_g L^(a+g) s^g / g!, s = Z_child - Z_parent
//   L2P: g_k = -sum_a L^(a+e_k) x^a / a!
// FP64 warp instructions hold their pipe for 64 cycles whatever lanes work, so
// every kernel spreads its sums over all lanes and factorises them by
// coordinate: a monomial as x^a0 times y^a1 z^a2, a shift as three shifts along
// one axis each (P + 1 terms at most per coefficient instead of up to 84 at P =
// 6).  Every sum has a fixed order.
// Measured: P2M and M2M 0.22 ms at 65,536 bodies and P = 5 (1.92 with a thread per
// cell), 0.18 at 16,384 and P = 6 (2.70 with one lane for the centre of mass and
// unfactorised sums); L2L and L2P 0.13 (0.27) and 0.10 (0.22) ms.
#include "expansion_mi.cuh"
#include "internal.cuh"

namespace amfmm {
namespace {

#include "expansion_gen.cuh"

__device__ const MultiIndices d_mi = make_multi_indices();

constexpr int kWarps = 4;

// One warp per leaf.  Centre of mass: products in parallel, sums in body order,
// one lane per component.  Moments: per body the powers mu x^i and the products
// y^j z^k, then one lane per moment, bodies in order, one FMA per body.
template <int P>
constexpr int kP2MRows = P + 1 + (P + 1) * (P + 2) / 2;

template <int P>
__global__ void __launch_bounds__(kWarps * 32) k_p2m(
    int32_t nleaf, const int32_t *leaves, const int32_t *begin,
    const int32_t *count, const double *X, const double *Y,
    const double *Zb, const double *Mb, double *__restrict__ S, double *__restrict__ M,
    double *__restrict__ Z, double *__restrict__ invM, double *__restrict__ mom) {
  pdl_wait();
  constexpr int NM = mi_off(P + 1), kRounds = (NM + 31) / 32, kRows = kP2MRows<P>;
  extern __shared__ double rows_all[];  // [kWarps][kRows][33]
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  double(*row)[33] = reinterpret_cast<double(*)[33]>(rows_all + static_cast<size_t>(w) * kRows * 33);
  const int q = blockIdx.x * kWarps + w;
  if (q >= nleaf) return;  // whole warp
  const int c = leaves[q], b = begin[c], cnt = count[c];
  double s = 0.0;
  for (int t0 = 0; t0 < cnt; t0 += 32) {
    if (t0 + l < cnt) {
      const int i = b + t0 + l;
      const double mu = Mb[i];
      row[0][l] = __dmul_rn(mu, X[i]);
      row[1][l] = __dmul_rn(mu, Y[i]);
      row[2][l] = __dmul_rn(mu, Zb[i]);
      row[3][l] = mu;
    }
    __syncwarp();
    if (l < 4)
      for (int k = 0; k < min(32, cnt - t0); ++k) s = __dadd_rn(s, row[l][k]);
    __syncwarp();
  }
  const double mm = __shfl_sync(0xffffffffu, s, 3);
  const double z = __ddiv_rn(l == 3 ? 1.0 : s, mm);
  if (l < 3) {
    S[3 * c + l] = s;
    Z[3 * c + l] = z;
  } else if (l == 3) {
    M[c] = mm;
    invM[c] = z;
  }
  const double z0 = __shfl_sync(0xffffffffu, z, 0), z1 = __shfl_sync(0xffffffffu, z, 1),
               z2 = __shfl_sync(0xffffffffu, z, 2);
  int rx[kRounds], ryz[kRounds];
  double acc[kRounds];
#pragma unroll
  for (int r = 0; r < kRounds; ++r) {
    const int i = min(l + 32 * r, NM - 1), a1 = d_mi.a[i][1], a2 = d_mi.a[i][2], h = a1 + a2;
    rx[r] = d_mi.a[i][0];
    ryz[r] = P + 1 + h * (h + 1) / 2 + a2;
    acc[r] = 0.0;
  }
  for (int t0 = 0; t0 < cnt; t0 += 32) {
    if (t0 + l < cnt) {
      const int i = b + t0 + l;
      const double x = X[i] - z0, y = Y[i] - z1, zz = Zb[i] - z2;
      double v = Mb[i];
      row[0][l] = v;
#pragma unroll
      for (int a = 1; a <= P; ++a) row[a][l] = v *= x;
      double yz[P + 1];  // y^(h-k) z^k of one order h
      yz[0] = 1.0;
      row[P + 1][l] = 1.0;
#pragma unroll
      for (int h = 1; h <= P; ++h) {
        yz[h] = yz[h - 1] * zz;
#pragma unroll
        for (int k = h - 1; k >= 0; --k) yz[k] *= y;
#pragma unroll
        for (int k = 0; k <= h; ++k) row[P + 1 + h * (h + 1) / 2 + k][l] = yz[k];
      }
    }
    __syncwarp();
    const int num = min(32, cnt - t0);
#pragma unroll
    for (int r = 0; r < kRounds; ++r) {
      const double *px = row[rx[r]], *pyz = row[ryz[r]];
      for (int k = 0; k < num; ++k) acc[r] = fma(px[k], pyz[k], acc[r]);
    }
    __syncwarp();
  }
#pragma unroll
  for (int r = 0; r < kRounds; ++r) {
    const int i = l + 32 * r;
    if (i < NM) mom[static_cast<int64_t>(c) * NM + i] = i == 0 ? mm : acc[r];
  }
}

// One block per parent (a warp on each partition of the SM): the eight children
// side by side, their moments over a! shifted axis by axis, then added in octant
// order.  Every warp takes the centre of mass for itself.
template <int P>
__global__ void __launch_bounds__(kWarps * 32) k_m2m(int32_t c0, const int32_t *first_child,
                                                     const int32_t *nchild, double *__restrict__ S,
                                                     double *__restrict__ M, double *__restrict__ Z,
                                                     double *__restrict__ invM, double *__restrict__ mom) {
  pdl_wait();
  constexpr int NM = mi_off(P + 1);
  __shared__ double buf[2][8 * NM], sf[8][3][P + 1];
  const int t = threadIdx.x, l = t & 31;
  const int c = c0 + blockIdx.x;
  const int nch = nchild[c];
  if (nch == 0) return;  // whole block
  const int f = first_child[c];
  // lane 4 k + d: component d of child k (d = 3: the mass)
  const int ck = l >> 2, d = l & 3;
  const double v = ck < nch ? (d < 3 ? S[3 * (f + ck) + d] : M[f + ck]) : 0.0;
  double s = 0.0;
  for (int k = 0; k < nch; ++k) s = __dadd_rn(s, __shfl_sync(0xffffffffu, v, 4 * k + d));
  const double mm = __shfl_sync(0xffffffffu, s, 3);
  const double z = __ddiv_rn(d == 3 ? 1.0 : s, mm);
  if (t < 4) {
    if (d < 3) {
      S[3 * c + d] = s;
      Z[3 * c + d] = z;
    } else {
      M[c] = mm;
      invM[c] = z;
    }
  }
  if (t < 32 && ck < nch && d < 3) {
    const double sv = Z[3 * (f + ck) + d] - z;  // s^p / p!
    double p = 1.0;
    sf[ck][d][0] = 1.0;
#pragma unroll
    for (int a = 1; a <= P; ++a) {
      p *= sv;
      sf[ck][d][a] = p * d_mi.inv_fact[mi_off(a)];
    }
  }
  const int work = nch * NM;
  for (int e = t; e < work; e += kWarps * 32) buf[0][e] = mom[static_cast<int64_t>(f) * NM + e] * d_mi.inv_fact[e % NM];
  __syncthreads();
#pragma unroll
  for (int axis = 0; axis < 3; ++axis) {
    const double *in = buf[axis & 1];
    for (int e = t; e < work; e += kWarps * 32) {
      const int k = e / NM, i = e - k * NM;
      const int a0 = d_mi.a[i][0], a1 = d_mi.a[i][1], a2 = d_mi.a[i][2];
      const int a = axis == 0 ? a0 : axis == 1 ? a1 : a2;
      const double *src = in + k * NM, *pw = sf[k][axis];
      double acc = 0.0;
      for (int b = 0; b <= a; ++b) {
        const int j = axis == 0 ? mi_idx(b, a1, a2) : axis == 1 ? mi_idx(a0, b, a2) : mi_idx(a0, a1, b);
        acc = fma(src[j], pw[a - b], acc);
      }
      buf[(axis & 1) ^ 1][e] = acc;
    }
    __syncthreads();
  }
  for (int i = t; i < NM; i += kWarps * 32) {
    double acc = 0.0;
    for (int k = 0; k < nch; ++k) acc += buf[1][k * NM + i];
    mom[static_cast<int64_t>(c) * NM + i] = i == 0 ? mm : acc * d_mi.fact[i];
  }
}

// One warp per child, axis by axis.
template <int P>
__global__ void __launch_bounds__(kWarps * 32) k_l2l_general(int32_t c0, int32_t c1,
                                                             const int32_t *parent,
                                                             const double *Z, double *__restrict__ loc) {
  pdl_wait();
  constexpr int NM = mi_off(P + 1), NL = NM - 1;
  __shared__ double buf_all[kWarps][2][NM], sf_all[kWarps][3][P + 1];
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  const int c = c0 + blockIdx.x * kWarps + w;
  if (c >= c1) return;  // whole warp
  double(*buf)[NM] = buf_all[w];
  const int p = parent[c];
  if (l < 3) {
    const double sv = Z[3 * c + l] - Z[3 * p + l];
    double v = 1.0;
    sf_all[w][l][0] = 1.0;
#pragma unroll
    for (int a = 1; a <= P; ++a) {
      v *= sv;
      sf_all[w][l][a] = v * d_mi.inv_fact[mi_off(a)];
    }
  }
  for (int i = l; i < NM; i += 32) buf[0][i] = i > 0 ? loc[static_cast<int64_t>(p) * NL + i - 1] : 0.0;
  __syncwarp();
#pragma unroll
  for (int axis = 0; axis < 3; ++axis) {
    const double *in = buf[axis & 1], *pw = sf_all[w][axis];
    for (int i = l; i < NM; i += 32) {
      const int a0 = d_mi.a[i][0], a1 = d_mi.a[i][1], a2 = d_mi.a[i][2], top = P - d_mi.a[i][3];
      double acc = 0.0;
      for (int g = 0; g <= top; ++g) {
        const int j = axis == 0 ? mi_idx(a0 + g, a1, a2) : axis == 1 ? mi_idx(a0, a1 + g, a2) : mi_idx(a0, a1, a2 + g);
        acc = fma(in[j], pw[g], acc);
      }
      if (axis < 2) buf[(axis & 1) ^ 1][i] = acc;
      else if (i > 0) loc[static_cast<int64_t>(c) * NL + i - 1] += acc;
    }
    __syncwarp();
  }
}

template <int P>
__global__ void k_l2p_general(int64_t n, const int32_t *leaf_of, const double *Z,
                              const double *loc, const double *X,
                              const double *Y, const double *Zb,
                              const double *near, double *__restrict__ acc) {
  pdl_wait();
  const int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
  if (i >= n) return;
  const int L = leaf_of[i];
  const double x[3] = {X[i] - Z[3 * L], Y[i] - Z[3 * L + 1], Zb[i] - Z[3 * L + 2]};
  double g[3];
  BodyField<P>::eval(loc + static_cast<int64_t>(L) * (mi_off(P + 1) - 1), x, g);
#pragma unroll
  for (int d = 0; d < 3; ++d) acc[d * n + i] = near[d * n + i] + g[d];
}

template <int P>
int upward_p(fmm_ctx *c) {
  constexpr int kShared = static_cast<int>(sizeof(double)) * kWarps * kP2MRows<P> * 33;
  if (kShared > 48 * 1024)
    AMFMM_CUDA(c, cudaFuncSetAttribute(k_p2m<P>, cudaFuncAttributeMaxDynamicSharedMemorySize, kShared));
  launch(c, k_p2m<P>, grid_for(c->sz.nleaf, kWarps), kWarps * 32, kShared, static_cast<int32_t>(c->sz.nleaf),
         ptr<int32_t>(c->leaves), ptr<int32_t>(c->begin), ptr<int32_t>(c->count), ptr<double>(c->X), ptr<double>(c->Y),
         ptr<double>(c->Zb), ptr<double>(c->Mb), ptr<double>(c->S), ptr<double>(c->M), ptr<double>(c->Z),
         ptr<double>(c->invM), ptr<double>(c->mom));
  AMFMM_TRY(launched(c, "p2m"));
  for (int lev = c->sz.depth - 1; lev >= 0; --lev) {
    const int64_t c0 = c->sz.lvl_off[lev], c1 = c->sz.lvl_off[lev + 1];
    if (c1 <= c0) continue;
    launch(c, k_m2m<P>, static_cast<unsigned>(c1 - c0), kWarps * 32, 0, static_cast<int32_t>(c0),
           ptr<int32_t>(c->first_child), ptr<int32_t>(c->nchild), ptr<double>(c->S), ptr<double>(c->M),
           ptr<double>(c->Z), ptr<double>(c->invM), ptr<double>(c->mom));
    AMFMM_TRY(launched(c, "m2m"));
  }
  return FMM_OK;
}

template <int P>
int downward_p(fmm_ctx *c) {
  const int64_t n = c->sz.n;
  for (int lev = 1; lev <= c->sz.depth; ++lev) {
    const int64_t c0 = c->sz.lvl_off[lev], c1 = c->sz.lvl_off[lev + 1];
    if (c1 <= c0) continue;
    launch(c, k_l2l_general<P>, grid_for(c1 - c0, kWarps), kWarps * 32, 0, static_cast<int32_t>(c0),
           static_cast<int32_t>(c1), ptr<int32_t>(c->parent), ptr<double>(c->Z), ptr<double>(c->loc));
    AMFMM_TRY(launched(c, "l2l_general"));
  }
  launch(c, k_l2p_general<P>, grid_for(n, 128), 128, 0, n, ptr<int32_t>(c->leaf_of), ptr<double>(c->Z),
         ptr<double>(c->loc), ptr<double>(c->X), ptr<double>(c->Y), ptr<double>(c->Zb), ptr<double>(c->near),
         ptr<double>(c->acc));
  return launched(c, "l2p_general");
}

}  // namespace

int mom_stride(int P) { return (P + 1) * (P + 2) * (P + 3) / 6; }
int loc_stride(int P) { return P == 3 ? kLocStride : mom_stride(P) - 1; }

int upward_general(fmm_ctx *c) {
  switch (c->opts.order_P) {
    case 4: return upward_p<4>(c);
    case 5: return upward_p<5>(c);
    case 6: return upward_p<6>(c);
    case 7: return upward_p<7>(c);
    default: return upward_p<8>(c);
  }
}

int downward_general(fmm_ctx *c) {
  switch (c->opts.order_P) {
    case 4: return downward_p<4>(c);
    case 5: return downward_p<5>(c);
    case 6: return downward_p<6>(c);
    case 7: return downward_p<7>(c);
    default: return downward_p<8>(c);
  }
}

}  // namespace amfmm
