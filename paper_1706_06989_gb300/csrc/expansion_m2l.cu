// expansion_m2l.cu -- M2L of the general-order expansion (App. A), P = 4 .. 8,
// FP64.  Notation as in expansion.cu; with r = Z_A - Z_B, n = r / R and the
// derivatives D^g = d^g (-1/R) = R^-(|g|+1) U^g(n):
//   field of B at A:  L_A^a = sum_b (-1)^|b| D^(a+b) M_B^b / b!,  |a| + |b| <= P
//   field of A at B:  L_B^b = (-1)^|b| sum_a D^(a+b) M_A^a / a!
//   correction:       F_k = - sum_{|a|+|b|=P} (-1)^|b| M_A^a M_B^b D^(a+b+e_k) / (a! b!),
//                     -F/M_A on A, +F/M_B on B; TCO: F - n (n.F)
//
// FP64 instructions are what this costs (64 cycles of their pipe per warp), so
// their number is kept small by the reduced indices: the moments of a cell are
// folded onto them once, M'^b' = the sum of M^b / b! over the b that the trace
// relation sends to b', with its sign and count, and the sums over a and b run
// over 2n + 1 indices per order instead of (n+1)(n+2)/2.  The correction uses
//   V^a' = sum_{|b|=P+1-|a'|} U^(a'+b) M'_B^b,   F_k = - sum_a M'_A^a V^(a+e_k)
// which continues the field's own sums by one order.  P = 5: about 1,400
// instructions per pair instead of 2,700 (full indices, straight-line code);
// P = 6: 2,100 instead of 7,000 (full indices, a warp per pair with tables).
//
// One thread per pair: every lane works in every instruction, and values that
// exceed the registers go to local memory, whose traffic the slow FP64 pipe
// hides.  The slots hold reduced locals; the per-cell sums restore the others.
// Measured: 1.5M pairs at P = 5 in 3.19 ms (6.97 with full indices), 152,000 at
// P = 6 in 0.54 ms (3.65 with a warp per pair); the sums in 0.27 (0.70) and 0.06
// (0.27) ms.
#include <type_traits>
#include <utility>

#include "expansion_mi.cuh"
#include "internal.cuh"

namespace amfmm {
namespace {

__device__ const MultiIndices d_mi = make_multi_indices();

template <int I>
using Int = std::integral_constant<int, I>;
// f(Int<B>{}), ..., f(Int<E - 1>{})
template <int B, class F, int... I>
__device__ __forceinline__ void for_each_int(F &&f, std::integer_sequence<int, I...>) {
  (f(Int<B + I>{}), ...);
}
template <int B, int E, class F>
__device__ __forceinline__ void static_for(F &&f) {
  if constexpr (B < E) for_each_int<B>(f, std::make_integer_sequence<int, E - B>{});
}

constexpr int isqrt(int r) {
  int n = 0;
  while ((n + 1) * (n + 1) <= r) ++n;
  return n;
}
// the exponents of reduced index r
struct Red {
  int n, t, u, s;
};
constexpr Red red(int r) {
  const int n = isqrt(r), k = r - n * n, s = k > n ? 1 : 0, u = s ? k - n - 1 : k;
  return Red{n, n - s - u, u, s};
}
constexpr int tri(int t, int u) { return (t + u) * (t + u + 1) / 2 + u; }
constexpr int tri_count(int n) { return (n + 1) * (n + 2) / 2; }  // t + u <= n

// U^(t,u,s), t + u + s <= N, s <= 2, by the recurrences of the derivatives of
// f_m = (1/R d/dR)^m (-1/R) at R = 1 (d_x f_m = x f_(m+1)), level by level down
// to m = 0.
template <int N>
struct UnitDerivs {
  double u0[tri_count(N)], u1[tri_count(N - 1)], u2[tri_count(N - 2)];
  __device__ __forceinline__ void fill(double x, double y, double z) {
    double up[tri_count(N)];
    static_for<0, N + 1>([&](auto im) {
      constexpr int m = N - im;
      double now[tri_count(N)];
      double f = m % 2 ? 1.0 : -1.0;  // -(-1)^m (2m-1)!!
      static_for<1, m + 1>([&](auto k) { f *= 2 * k - 1; });
      now[0] = f;
      static_for<1, N - m + 1>([&](auto t) {
        now[tri(t, 0)] = x * up[tri(t - 1, 0)];
        if constexpr (t > 1) now[tri(t, 0)] += (t - 1) * up[tri(t > 1 ? t - 2 : 0, 0)];
      });
      static_for<1, N - m + 1>([&](auto u) {
        static_for<0, N - m - u + 1>([&](auto t) {
          now[tri(t, u)] = y * up[tri(t, u - 1)];
          if constexpr (u > 1) now[tri(t, u)] += (u - 1) * up[tri(t, u > 1 ? u - 2 : 0)];
        });
      });
      static_for<0, tri_count(N - m)>([&](auto q) { up[q] = now[q]; });
      if constexpr (m == 1) static_for<0, tri_count(N - 1)>([&](auto q) { u1[q] = z * now[q]; });
      if constexpr (m == 0) static_for<0, tri_count(N)>([&](auto q) { u0[q] = now[q]; });
    });
    static_for<0, N - 1>([&](auto t) {
      static_for<0, N - 1 - t>([&](auto u) { u2[tri(t, u)] = -(u0[tri(t + 2, u)] + u0[tri(t, u + 2)]); });
    });
  }
  template <int T, int U, int S>
  __device__ __forceinline__ double get() const {
    if constexpr (S == 0) return u0[tri(T, U)];
    else if constexpr (S == 1) return u1[tri(T, U)];
    else return u2[tri(T, U)];
  }
  // sum over reduced b of orders [M0, M1] of U^(a+b) m[b], a the reduced index R
  template <int R, int M0, int M1>
  __device__ __forceinline__ double contract(const double *m) const {
    constexpr Red a = red(R);
    double acc = 0.0;
    static_for<M0 * M0, (M1 + 1) * (M1 + 1)>([&](auto ib) {
      constexpr Red b = red(ib);
      acc = fma(get<a.t + b.t, a.u + b.u, a.s + b.s>(), m[ib], acc);
    });
    return acc;
  }
};

// moments folded onto the reduced indices, divided by b!
template <int P>
__global__ void __launch_bounds__(128) k_fold_moments(int32_t ncell, const double *mom,
                                                      double *__restrict__ out) {
  pdl_wait();
  constexpr int NM = mi_off(P + 1), NR = (P + 1) * (P + 1), NS = red_mom_stride(P);
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= ncell) return;
  const double *m = mom + static_cast<int64_t>(c) * NM;
  double acc[NS];
#pragma unroll
  for (int q = 0; q < NS; ++q) acc[q] = 0.0;
  static_for<0, P + 1>([&](auto a2) {
    static_for<0, P + 1 - a2>([&](auto a1) {
      static_for<0, P + 1 - a2 - a1>([&](auto a0) {
        constexpr int q = a2 / 2;
        constexpr double f[9] = {1.0, 1.0, 2.0, 6.0, 24.0, 120.0, 720.0, 5040.0, 40320.0};
        const double v = m[mi_idx(a0, a1, a2)] * (1.0 / (f[a0] * f[a1] * f[a2]));
        static_for<0, q + 1>([&](auto j) {
          acc[red_idx(a0 + 2 * j, a1 + 2 * (q - j), a2 % 2)] += (q % 2 ? -choose(q, j) : choose(q, j)) * v;
        });
      });
    });
  });
  double2 *o = reinterpret_cast<double2 *>(out + static_cast<int64_t>(c) * NS);
#pragma unroll
  for (int q = 0; q < NS / 2; ++q) o[q] = make_double2(acc[2 * q], 2 * q + 1 < NR ? acc[2 * q + 1] : 0.0);
}

template <int P>
__global__ void __launch_bounds__(128, 2) k_m2l_general(int64_t K, int variant, const int2 *pairs,
                                                        const double *Z, const double *invM,
                                                        const double *fold,
                                                        const int32_t *pos, double *__restrict__ slots) {
  pdl_wait();
  constexpr int NR = (P + 1) * (P + 1), NL = red_loc_stride(P), NS = red_mom_stride(P);
  const int64_t k = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
  if (k >= K) return;
  const int A = pairs[k].x, B = pairs[k].y;
  double2 *LA = reinterpret_cast<double2 *>(slots + static_cast<int64_t>(pos[2 * k]) * NL);
  double2 *LB = reinterpret_cast<double2 *>(slots + static_cast<int64_t>(pos[2 * k + 1]) * NL);
  const double r0 = Z[3 * A] - Z[3 * B], r1 = Z[3 * A + 1] - Z[3 * B + 1], r2 = Z[3 * A + 2] - Z[3 * B + 2];
  const double R2 = r0 * r0 + r1 * r1 + r2 * r2;
  if (!(R2 > 0.0)) {
    for (int q = 0; q < NL / 2; ++q) LA[q] = LB[q] = make_double2(0.0, 0.0);
    return;
  }
  const double Ri = rsqrt(R2), nx = r0 * Ri, ny = r1 * Ri, nz = r2 * Ri;
  double ri[P + 2];
  ri[0] = 1.0;
#pragma unroll
  for (int q = 1; q < P + 2; ++q) ri[q] = ri[q - 1] * Ri;
  UnitDerivs<P + 1> U;
  U.fill(nx, ny, nz);
  // moments times R^-|b|; B's with (-1)^|b|
  double mA[NS], mB[NS];
  const double2 *fA = reinterpret_cast<const double2 *>(fold + static_cast<int64_t>(A) * NS);
  const double2 *fB = reinterpret_cast<const double2 *>(fold + static_cast<int64_t>(B) * NS);
#pragma unroll
  for (int q = 0; q < NS / 2; ++q) {
    const double2 a = fA[q], b = fB[q];
    mA[2 * q] = a.x;
    mA[2 * q + 1] = a.y;
    mB[2 * q] = b.x;
    mB[2 * q + 1] = b.y;
  }
  static_for<1, NR>([&](auto q) {
    constexpr int n = red(q).n;
    mA[q] *= ri[n];
    mB[q] *= n % 2 ? -ri[n] : ri[n];
  });
  // A's locals, and the correction's sums
  double first[3], keep = 0.0, f0 = 0.0, f1 = 0.0, f2 = 0.0;
  const bool torque = variant != FMM_UC;
  static_for<1, (P + 2) * (P + 2)>([&](auto ir) {
    constexpr Red a = red(ir);
    if constexpr (a.n <= P) {
      const double v = ri[a.n + 1 <= P + 1 ? a.n + 1 : 0] * U.template contract<ir, 0, P - a.n>(mB);
      constexpr int q = ir - 1;
      if constexpr (q < 3) first[q] = v;
      else if constexpr (q == 3) reinterpret_cast<double *>(LA)[3] = v;
      else if constexpr (q % 2 == 0 && q + 1 < NR - 1) keep = v;
      else if constexpr (q % 2 == 0) LA[q / 2] = make_double2(v, 0.0);
      else LA[q / 2] = make_double2(keep, v);
    }
    if (torque) {
      // V^a' meets M'_A^(a'-e_k); for a with s = 1, a + e_z has s = 2:
      // V^(t,u,2) = -V^(t+2,u,0) - V^(t,u+2,0)
      const double v = U.template contract<ir, P + 1 - a.n, P + 1 - a.n>(mB);
      if constexpr (a.t > 0) f0 = fma(mA[red_idx(a.t - 1, a.u, a.s)], v, f0);
      if constexpr (a.u > 0) f1 = fma(mA[red_idx(a.t, a.u - 1, a.s)], v, f1);
      if constexpr (a.s > 0) f2 = fma(mA[red_idx(a.t, a.u, 0)], v, f2);
      if constexpr (a.s == 0 && a.t > 1) f2 = fma(-mA[red_idx(a.t - 2, a.u, 1)], v, f2);
      if constexpr (a.s == 0 && a.u > 1) f2 = fma(-mA[red_idx(a.t, a.u - 2, 1)], v, f2);
    }
  });
  f0 *= -ri[2];
  f1 *= -ri[2];
  f2 *= -ri[2];
  if (variant == FMM_TCO) {
    const double nf = nx * f0 + ny * f1 + nz * f2;
    f0 -= nx * nf;
    f1 -= ny * nf;
    f2 -= nz * nf;
  }
  const double iA = invM[A], iB = invM[B];
  LA[0] = make_double2(first[0] - f0 * iA, first[1] - f1 * iA);
  reinterpret_cast<double *>(LA)[2] = first[2] - f2 * iA;
  static_for<1, NR>([&](auto ir) {
    constexpr Red a = red(ir);
    constexpr int q = ir - 1;
    double v = (a.n % 2 ? -ri[a.n + 1] : ri[a.n + 1]) * U.template contract<ir, 0, P - a.n>(mA);
    if constexpr (q == 0) v += f0 * iB;
    if constexpr (q == 1) v += f1 * iB;
    if constexpr (q == 2) v += f2 * iB;
    if constexpr (q % 2 == 0 && q + 1 < NR - 1) keep = v;
    else if constexpr (q % 2 == 0) LB[q / 2] = make_double2(v, 0.0);
    else LB[q / 2] = make_double2(keep, v);
  });
}

// Every cell sums its slots (in groups of slots, each in the order of the sort;
// the groups' sums are added in order), and the trace relation gives the local
// coefficients that the slots leave out.
constexpr int kSumBlock = 128;

template <int P>
__global__ void __launch_bounds__(kSumBlock) k_reduce_general(const int32_t *off,
                                                              const double *slots,
                                                              double *__restrict__ loc) {
  pdl_wait();
  constexpr int NS = red_loc_stride(P), NR = (P + 1) * (P + 1) - 1, NL = mi_off(P + 1) - 1;
  constexpr int kGroups = kSumBlock / NS;
  __shared__ double part[kGroups][NS];
  const int c = blockIdx.x, t = threadIdx.x, g = t / NS, q = t - g * NS;
  const int s0 = off[c], s1 = off[c + 1];
  if (g < kGroups && q < NR) {
    double acc = 0.0;
    int s = s0 + g;
    for (; s + 3 * kGroups < s1; s += 4 * kGroups) {
      double v[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) v[u] = slots[static_cast<int64_t>(s + u * kGroups) * NS + q];
#pragma unroll
      for (int u = 0; u < 4; ++u) acc += v[u];
    }
    for (; s < s1; s += kGroups) acc += slots[static_cast<int64_t>(s) * NS + q];
    part[g][q] = acc;
  }
  __syncthreads();
  if (t < NR) {
    double acc = part[0][t];
    for (int k = 1; k < kGroups; ++k) acc += part[k][t];
    part[0][t] = acc;
  }
  __syncthreads();
  for (int i = t; i < NL; i += kSumBlock) {
    const int a0 = d_mi.a[i + 1][0], a1 = d_mi.a[i + 1][1], a2 = d_mi.a[i + 1][2], h = a2 / 2;
    double v = 0.0;
    for (int j = 0; j <= h; ++j) v += choose(h, j) * part[0][red_idx(a0 + 2 * j, a1 + 2 * (h - j), a2 % 2) - 1];
    loc[static_cast<int64_t>(c) * NL + i] = h % 2 ? -v : v;
  }
}

template <int P>
int m2l_p(fmm_ctx *c) {
  const int64_t K = c->sz.n_m2l, nc = c->sz.ncell;
  AMFMM_TRY(ensure<double>(c, c->gen_fold, static_cast<size_t>(red_mom_stride(P)) * nc));
  launch(c, k_fold_moments<P>, grid_for(nc, 128), 128, 0, static_cast<int32_t>(nc), ptr<double>(c->mom),
         ptr<double>(c->gen_fold));
  AMFMM_TRY(launched(c, "fold_moments"));
  launch(c, k_m2l_general<P>, grid_for(K, 128), 128, 0, K, c->opts.variant, ptr<int2>(c->m2l), ptr<double>(c->Z),
         ptr<double>(c->invM), ptr<double>(c->gen_fold), ptr<int32_t>(c->m2l_pos), ptr<double>(c->m2l_slots));
  return launched(c, "m2l_general");
}

template <int P>
int reduce_p(fmm_ctx *c) {
  launch(c, k_reduce_general<P>, static_cast<unsigned>(c->sz.ncell), kSumBlock, 0, ptr<int32_t>(c->m2l_off),
         ptr<double>(c->m2l_slots), ptr<double>(c->loc));
  return launched(c, "reduce_general");
}

}  // namespace

int slot_stride_general(int P) { return red_loc_stride(P); }

int m2l_general(fmm_ctx *c) {
  if (c->sz.n_m2l == 0) return FMM_OK;
  switch (c->opts.order_P) {
    case 4: return m2l_p<4>(c);
    case 5: return m2l_p<5>(c);
    case 6: return m2l_p<6>(c);
    case 7: return m2l_p<7>(c);
    default: return m2l_p<8>(c);
  }
}

int reduce_general(fmm_ctx *c) {
  if (c->sz.n_m2l == 0) {
    AMFMM_CUDA(c, cudaMemsetAsync(c->loc.p, 0, sizeof(double) * loc_stride(c->opts.order_P) * c->sz.ncell, c->stream));
    return FMM_OK;
  }
  switch (c->opts.order_P) {
    case 4: return reduce_p<4>(c);
    case 5: return reduce_p<5>(c);
    case 6: return reduce_p<6>(c);
    case 7: return reduce_p<7>(c);
    default: return reduce_p<8>(c);
  }
}

}  // namespace amfmm
