// p2p64.cu -- a8 in the FP64 form: near-field sums in 64-bit fixed point
// (fix64.cuh).
//
// On this GPU an FP64 instruction holds its partition's pipe for 64 cycles per
// warp, an integer product for four.  In FP64 arithmetic the near field ran at
// the FP64 pipe's rate (20 instructions per body pair, the pipe 90% busy) with
// every other unit idle: 16.1 ms at N = 1,048,576 (Plummer, theta = 0.5, 421M
// body pairs), 4.45 ms at 262,144, 1.21 ms at 2,000.  In fixed point: 7.22,
// 1.99 and 0.08 ms.  It is bound by the integer pipes and the latencies around
// them (four resident blocks per SM; with three 8.4 ms at N = 1,048,576, with five,
// which spill registers, 7.5), and no less exact: a pair's factor is good to
// 2^-54.6 (FP64: about 2^-52), and a term rounds once.
//
// One-sided: each leaf gathers from its own bodies and from every leaf paired
// with it, on either side.  A pair is then evaluated twice, but the sums live
// in registers (the mutual form kept a third of its traffic in shared-memory
// partials, and wrote and read 24 bytes per body and pair), and the
// preparation needs one sort of the leaf pairs instead of two, no slot offsets
// and no column arrays.  The two forces of a pair are rounded independently, from
// the same separation; the net force stays at rounding level (5.6e-18 of the sum of
// the magnitudes at N = 1,048,576).
//
// Work item: 16 bodies (rows) of a leaf at most, and a group of 32 entries of
// the leaf's list (itself first, then its partners in the stable order of the
// sort); groups keep a leaf with very many partners from serialising the
// kernel.  One warp per item, drawn from a queue.  Lanes are (row, subset):
// with nr rows, 32 / nr subsets share a batch of source bodies.  A batch is 32
// source bodies: each lane converts one to the batch's window and leaves its
// digits in shared memory.
//
// The sums' unit follows the heaviest source of what is being summed, a body at
// the row's own place apart: a unit set by a body that adds no term there would
// round the others' terms away.  A batch is therefore taken in classes of mass: the
// sources within 2^kClassSpan of its heaviest, then those of the rest, and so on
// (one class unless the masses differ by more).  N = 262,144 with half of the masses
// 1e-10 of the others: 4.35 ms (FP64 arithmetic 5.85); spread evenly over 2^90, five
// classes a batch, 17.0 (13.1).
//
// Every sum has a fixed order and every result is independent of which warp
// takes an item.
#include <limits.h>

#include "fix64.cuh"
#include "internal.cuh"

namespace amfmm {
namespace {

constexpr int kWarps = 4;
constexpr int kGroup = 32;  // list entries per work item
constexpr int kRows = 16;   // rows per work item: 32 / rows subsets share a batch, and leaves of 17 to 25 bodies
                            // (half of the work at n_crit = 25) would fill 53 to 78% of one warp's lanes

// Positions and mass of a body in the fixed formats, 48 bytes.
struct Rec {
  uint4 a, b, c;  // x0 x1 x2 y0 | y1 y2 z0 z1 | z2 m1 m0 (mass exponent, extent exponent << 16)
};

__global__ void k_body_fixed(int64_t n, const double *X, const double *Y,
                             const double *Zb, const double *Mb,
                             const double *box, const int32_t *order,
                             const int32_t *sysid, Rec *__restrict__ rec) {
  pdl_wait();
  const int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
  if (i >= n) return;
  const int ex = fix::extent_exponent(box[(sysid ? 4 * sysid[order[i]] : 0) + 3]);
  const fix::W96 x = fix::fixed96(X[i], ex - 95), y = fix::fixed96(Y[i], ex - 95), z = fix::fixed96(Zb[i], ex - 95);
  uint64_t M;
  int em;
  fix::mantissa64(Mb[i], &M, &em);
  Rec r;
  r.a = make_uint4(x.w[0], x.w[1], x.w[2], y.w[0]);
  r.b = make_uint4(y.w[1], y.w[2], z.w[0], z.w[1]);
  r.c = make_uint4(z.w[2], static_cast<uint32_t>(M >> 32), static_cast<uint32_t>(M),
                   (static_cast<uint32_t>(em) & 0xffffu) | (static_cast<uint32_t>(ex) << 16));
  rec[i] = r;
}

__device__ __forceinline__ void unpack(const Rec &r, fix::W96 o[3]) {
  o[0] = fix::W96{{r.a.x, r.a.y, r.a.z}};
  o[1] = fix::W96{{r.a.w, r.b.x, r.b.y}};
  o[2] = fix::W96{{r.b.z, r.b.w, r.c.x}};
}

// A body's position relative to another's (its leaf's first row), the unit of
// both, and its mass's exponent.
__device__ __forceinline__ void offset(const Rec &r, const Rec &origin, fix::W96 o[3], int *g, int *em) {
  fix::W96 ref[3];
  unpack(origin, ref);
  unpack(r, o);
#pragma unroll
  for (int c = 0; c < 3; ++c) o[c] = fix::sub96(o[c], ref[c]);
  *g = (static_cast<int32_t>(r.c.w) >> 16) - 95;
  *em = static_cast<int16_t>(r.c.w & 0xffffu);
}

// Pairs without digits (positions that agree to 2^-42 of the system's extent,
// close softened pairs, any pair when eps^2 overflows): the direct sum's formula
// in FP64.
__device__ __forceinline__ double3 pair64(double dx, double dy, double dz, double m, double eps2) {
  const double d2 = fma(dz, dz, fma(dy, dy, dx * dx));
  if (d2 == 0.0) return make_double3(0.0, 0.0, 0.0);
  const double ri = rsqrt(d2 + eps2);
  const double s = m * (ri * ri * ri);
  return make_double3(s * dx, s * dy, s * dz);
}

struct WarpSmem {
  int4 h[32];   // Hx Hy Hz Lx
  int4 l[32];   // Ly Lz m1 m0
  int2 x[32];   // mass exponent, body index
  double f[3][32];  // per lane: FP64 sums
};

// Adds the sums to the lane's FP64 ones and clears them.
__device__ __forceinline__ void flush(fix::Acc &acc, int &terms, WarpSmem &sm, int l) {
  fix::acc_carry(acc, terms);
#pragma unroll
  for (int c = 0; c < 3; ++c)
    sm.f[c][l] += scalbn(fma(static_cast<double>(acc.a2[c]), 536870912.0, static_cast<double>(acc.a1[c])),
                         acc.Ua + 2 * fix::kDig);
  fix::acc_clear(acc);
  terms = 0;
}

// SOFT: softening added to r^2 in fixed point.
template <bool SOFT>
__global__ void __launch_bounds__(kWarps * 32, 4) k_p2p64(
    int32_t nitem, int64_t n, const int4 *items, const int32_t *begin,
    const int32_t *count, const int32_t *off, const uint32_t *partner,
    const Rec *rec, const double *X,
    const double *Y, const double *Zb, const double *Mb, double eps2, double *__restrict__ near,
    double *__restrict__ extra, int *__restrict__ queue) {
  pdl_wait();
  __shared__ WarpSmem smem[kWarps];
  const int l = threadIdx.x & 31;
  WarpSmem &sm = smem[threadIdx.x >> 5];
  constexpr unsigned kAll = 0xffffffffu;
  for (;;) {
    int q = 0;
    if (l == 0) q = atomicAdd(queue, 1);
    q = __shfl_sync(kAll, q, 0);
    if (q >= nitem) break;
    const int4 it = items[q];  // leaf, first row, entry group, offset of the partial sums (-1: near)
    const int L = it.x;
    const int nA = count[L], bA = begin[L] + it.y;
    const int nr = min(kRows, nA - it.y);
    const int nsub = 32 / nr;
    const int sub = l / nr, row = l - sub * nr;
    const bool active = sub < nsub;
    const int i = bA + (active ? row : 0);
    int g0;  // unit of the positions
    uint32_t rmag;
    {
      fix::W96 o[3];
      int em;
      offset(rec[i], rec[bA], o, &g0, &em);
      rmag = max(max(fix::top_mag(o[0]), fix::top_mag(o[1])), fix::top_mag(o[2]));
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) sm.f[c][l] = 0.0;
    const bool all64 = SOFT && !isfinite(eps2);
    rmag = __reduce_max_sync(kAll, rmag);
    fix::Acc acc;
    fix::acc_clear(acc);
    int steps = 0, terms = 0;  // since the last carry: steps of the warp, terms of the lane
    // this group's entries, one per lane (entry 0 of group 0: the leaf itself)
    const int e = it.z * kGroup + l - 1, e0 = off[L], e1 = off[L + 1];
    int pb = 0, pc = 0;
    if (e < 0) {
      pb = begin[L];
      pc = nA;
    } else if (e0 + e < e1) {
      const int P = static_cast<int>(partner[e0 + e]);
      pb = begin[P];
      pc = count[P];
    }
    int incl = pc;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int y = __shfl_up_sync(kAll, incl, d);
      if (l >= d) incl += y;
    }
    const int total = __shfl_sync(kAll, incl, 31);
    const int bodyBase = pb - (incl - pc);  // body of column j of this entry: bodyBase + j
    int shPrev = -1;       // window of the digits
    int unit = INT_MIN / 2;  // the sums' unit, less what acc_carry raises it by
    int32_t H[3], Lo[3];
    bool rounded = false;
    fix::Soft soft{};
    for (int j0 = 0; j0 < total; j0 += 32) {
      const int j = min(j0 + l, total - 1);
      int own = 0;  // entry of column j: the number of entries that end at or before it
#pragma unroll
      for (int step = 16; step > 0; step >>= 1) {
        const int y = __shfl_sync(kAll, incl, own + step - 1);
        if (y <= j) own += step;
      }
      const int jb = __shfl_sync(kAll, bodyBase, own) + j;
      const Rec rj = rec[jb];
      fix::W96 s[3];
      int gj, emj;
      offset(rj, rec[bA], s, &gj, &emj);
      const uint32_t cmag =
          __reduce_max_sync(kAll, max(max(fix::top_mag(s[0]), fix::top_mag(s[1])), fix::top_mag(s[2])));
      const int sh = fix::window_shift(rmag, cmag);
      const int gd = g0 + sh;
      if (sh != shPrev) {
        fix::W96 o[3];
        int g, er;
        offset(rec[i], rec[bA], o, &g, &er);
        rounded = false;
#pragma unroll
        for (int c = 0; c < 3; ++c) rounded |= fix::digits(o[c], sh, &H[c], &Lo[c]);
        shPrev = sh;
        if (SOFT && !all64) soft = fix::soft_window(eps2, gd);
      }
      const int ncol = min(32, total - j0);
      int4 dh, dl;
      int32_t close;
      {
        int32_t h[3], lo[3];
        bool r = rounded;
#pragma unroll
        for (int c = 0; c < 3; ++c) r |= fix::digits(s[c], sh, &h[c], &lo[c]);
        close = __any_sync(kAll, r) ? fix::kCloseRounded : fix::kCloseExact;
        if (SOFT) close = all64 ? 0x7fffffff : fix::kCloseRounded;
        dh = make_int4(h[0], h[1], h[2], lo[0]);
        dl = make_int4(lo[1], lo[2], static_cast<int>(rj.c.y), static_cast<int>(rj.c.z));
      }
      unsigned rest = 0xffffffffu >> (32 - ncol);
#pragma unroll 1
      do {  // classes of mass
        const bool there = (rest >> l) & 1u;
        int top = __shfl_sync(kAll, emj, __ffs(static_cast<int>(rest)) - 1);
        if (__any_sync(kAll, there && emj != top)) top = __reduce_max_sync(kAll, there ? emj : INT_MIN);
        const bool in = there && emj >= top - (SOFT ? fix::kSoftClassSpan : fix::kClassSpan);
        const unsigned cls = __ballot_sync(kAll, in), tops = __ballot_sync(kAll, in && emj == top);
        const int nc = __popc(cls);
        rest &= ~cls;
        __syncwarp();  // every lane is done with the class before
        if (in) {
          const int at = __popc(cls & ((1u << l) - 1));
          sm.h[at] = dh;
          sm.l[at] = dl;
          sm.x[at] = make_int2(emj, jb);
        }
        __syncwarp();
        int em = top;
        if (!SOFT && (tops & (tops - 1)) == 0) {
          // a single heaviest body: not a source of the row where it is (itself,
          // or a body at its place)
          const int second = __reduce_max_sync(kAll, in && emj != top ? emj : INT_MIN);
          const int at = __popc(cls & (tops - 1));
          const int4 th = sm.h[at], tl = sm.l[at];
          if (th.x == H[0] && th.y == H[1] && th.z == H[2] && th.w == Lo[0] && tl.x == Lo[1] && tl.y == Lo[2])
            em = second;
        }
        if (em != INT_MIN) {  // (else nothing but that body)
          const int u = SOFT ? fix::unit_soft(gd, em, soft) : fix::unit_guess(gd, em);
          if (abs(u - unit) > (SOFT ? fix::kSoftUnitSpan : fix::kUnitSpan)) {  // (also at the first class)
            flush(acc, terms, sm, l);
            acc.Ua = unit = u;
          }
        }
        const int kb = fix::k_base(acc.Ua, gd) + 3 * soft.t;
        // The loop has no branch: close pairs, and those whose factor leaves the
        // sums' range, add nothing here and are marked for the loop below.  (Two
        // steps at a time where the registers allow: 7.22 against 7.35 ms at N = 1M,
        // 0.48 against 0.57 for one leaf of 4,096; softened 8.15 against 8.0.)
        unsigned mark = 0, bit = 1;
        constexpr int kUnroll = SOFT ? 1 : 2;
#pragma unroll kUnroll
        for (int c = active ? sub : 32; c < nc; c += nsub) {
          const int4 hh = sm.h[c], ll = sm.l[c];
          const int32_t dH[3] = {H[0] - hh.x, H[1] - hh.y, H[2] - hh.z};
          const int32_t dL[3] = {Lo[0] - hh.w, Lo[1] - ll.x, Lo[2] - ll.y};
          int64_t hi;
          uint32_t rem;
          fix::square(dH, dL, &hi, &rem);
          const bool apart = !fix::is_close(hi, close);
          if constexpr (SOFT) fix::soften(soft, &hi, &rem);
          int s2;
          const uint64_t w = fix::inv_cube(hi, rem, &s2);
          const uint64_t q = fix::times_mass(w, static_cast<uint32_t>(ll.z), static_cast<uint32_t>(ll.w));
          int k = kb - sm.x[c].x - 3 * s2;
          if (!apart || static_cast<unsigned>(k) >= fix::kShiftEnd) {
            k = fix::kNoTerm;
            mark |= bit;
          }
          bit <<= 1;
          int32_t qd[3];
          fix::factor_digits(q, k, qd);
          fix::acc_add(acc, qd, dH, dL);
        }
        terms += 31 - __clz(static_cast<int>(bit)) - __popc(mark);
        for (; mark; mark &= mark - 1) {
          const int c = sub + nsub * (__ffs(static_cast<int>(mark)) - 1);
          const int2 xx = sm.x[c];
          if (xx.y == i) continue;
          if constexpr (!SOFT) {
            fix::W96 a[3], b[3];
            unpack(rec[i], a);
            unpack(rec[xx.y], b);
            int32_t dH[3], dL[3], qd[3];
            const int shc = fix::close_digits(a, b, dH, dL);
            int64_t hi;
            uint32_t rem;
            int s2;
            fix::square(dH, dL, &hi, &rem);
            const uint64_t w = fix::inv_cube(hi, rem, &s2);
            const uint64_t q =
                fix::times_mass(w, static_cast<uint32_t>(sm.l[c].z), static_cast<uint32_t>(sm.l[c].w));
            const int k = kb + 2 * (shc - sh) - xx.x - 3 * s2;
            if (shc != fix::kNoDigits && static_cast<unsigned>(k) < fix::kShiftEnd) {
              fix::factor_digits(q, k, qd);
              fix::acc_add(acc, qd, dH, dL);
              ++terms;
              continue;
            }
          }
          const double3 f = pair64(X[i] - X[xx.y], Y[i] - Y[xx.y], Zb[i] - Zb[xx.y], Mb[xx.y], eps2);
          sm.f[0][l] += f.x;
          sm.f[1][l] += f.y;
          sm.f[2][l] += f.z;
        }
        // at most kMaxTerms steps between two carries
        steps += (nc + nsub - 1) / nsub;
        if (steps + (32 + nsub - 1) / nsub > fix::kMaxTerms) {
          fix::acc_carry(acc, terms);
          steps = terms = 0;
        }
      } while (rest);
    }
    flush(acc, terms, sm, l);
    double v[3] = {sm.f[0][l], sm.f[1][l], sm.f[2][l]};
    // sums of a row's subsets, pairwise in a fixed order
    int span = 1;
    while (span < nsub) span <<= 1;
    for (span >>= 1; span >= 1; span >>= 1) {
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const double y = __shfl_down_sync(kAll, v[c], static_cast<unsigned>(span * nr) & 31u);
        if (sub < span && sub + span < nsub) v[c] += y;
      }
    }
    if (l < nr) {
      // a_i = sum_j m_j (X_j - X_i) / r^3: the digits hold X_i - X_j
      if (it.w < 0) {
#pragma unroll
        for (int c = 0; c < 3; ++c) near[c * n + bA + l] = -v[c];
      } else {
#pragma unroll
        for (int c = 0; c < 3; ++c) extra[it.w + 3 * (it.y + l) + c] = -v[c];
      }
    }
  }
}

// Entry groups of a leaf (its own entry and ne partners)
__device__ __forceinline__ int groups_of(int ne) { return (ne + kGroup) / kGroup; }

// Work items and partial sums of every leaf; the near-field work, n_A n_B per
// leaf pair plus n (n - 1) / 2 per leaf, and the totals of the work items and of
// the partial sums in 64 bits (one atomic per block each, integer: exact).
constexpr int kCountBlock = 256;
__global__ void k_items64_count(int32_t nleaf, const int32_t *leaves, const int32_t *count,
                                const int32_t *off, const uint32_t *partner,
                                int32_t *__restrict__ nitems, int32_t *__restrict__ nextra,
                                unsigned long long *__restrict__ work, unsigned long long *__restrict__ extot,
                                unsigned long long *__restrict__ ittot) {
  pdl_wait();
  // one warp per leaf
  __shared__ unsigned long long sum[3][kCountBlock / 32];
  const int q = static_cast<int>((blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x) >> 5);
  const int l = threadIdx.x & 31, w = threadIdx.x >> 5;
  unsigned long long pairs = 0, parts = 0, items = 0;
  if (q == nleaf && l == 0) nitems[q] = nextra[q] = 0;  // closes the scans
  if (q < nleaf) {
    const int L = leaves[q], a = count[L];
    const int e0 = off[L], e1 = off[L + 1];
    unsigned long long cols = 0;
    for (int e = e0 + l; e < e1; e += 32) {
      const int P = static_cast<int>(partner[e]);
      if (P > L) cols += static_cast<unsigned long long>(count[P]);  // each pair once
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) cols += __shfl_xor_sync(0xffffffffu, cols, o);
    const int g = groups_of(e1 - e0), nb = (a + kRows - 1) / kRows;
    pairs = a * cols + static_cast<unsigned long long>(a) * (a - 1) / 2;
    parts = static_cast<unsigned long long>(g - 1) * 3 * a;
    items = static_cast<unsigned long long>(g) * nb;
    if (l == 0) {
      nitems[q] = static_cast<int32_t>(items);
      nextra[q] = static_cast<int32_t>(parts);
    }
  }
  if (l == 0) {
    sum[0][w] = pairs;
    sum[1][w] = parts;
    sum[2][w] = items;
  }
  __syncthreads();
  if (threadIdx.x < 3) {
    unsigned long long v = 0;
    for (int k = 0; k < kCountBlock / 32; ++k) v += sum[threadIdx.x][k];
    if (v) atomicAdd(threadIdx.x == 0 ? work : threadIdx.x == 1 ? extot : ittot, v);
  }
}

__global__ void k_items64_fill(int32_t nleaf, const int32_t *leaves, const int32_t *count,
                               const int32_t *off, const int32_t *itemOff,
                               const int32_t *extraOff, int4 *__restrict__ items) {
  pdl_wait();
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= nleaf) return;
  const int L = leaves[q], a = count[L];
  const int g = groups_of(off[L + 1] - off[L]), nb = (a + kRows - 1) / kRows;
  int o = itemOff[q];
  for (int k = 0; k < g; ++k)
    for (int b = 0; b < nb; ++b)
      items[o++] = make_int4(L, kRows * b, k, k == 0 ? -1 : extraOff[q] + (k - 1) * 3 * a);
}

// Adds the partial sums of a leaf's later entry groups, in group order (one
// warp per leaf).
__global__ void k_p2p64_groups(int32_t nleaf, int64_t n, const int32_t *leaves,
                               const int32_t *begin, const int32_t *count,
                               const int32_t *off, const int32_t *extraOff,
                               const double *extra, double *__restrict__ near) {
  pdl_wait();
  const int q = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int l = threadIdx.x & 31;
  if (q >= nleaf) return;
  const int L = leaves[q];
  const int g = groups_of(off[L + 1] - off[L]);
  if (g < 2) return;
  const int bA = begin[L], nA = count[L];
  const double *e = extra + extraOff[q];
  for (int t = l; t < 3 * nA; t += 32) {
    const int64_t o = static_cast<int64_t>(t % 3) * n + bA + t / 3;
    double s = near[o];
    for (int k = 0; k < g - 1; ++k) s += e[static_cast<int64_t>(k) * 3 * nA + t];
    near[o] = s;
  }
}

}  // namespace

int p2p64_prepare(fmm_ctx *c) {
  const int64_t K = c->sz.n_p2p, nc = c->sz.ncell, n = c->sz.n;
  const int32_t nleaf = static_cast<int32_t>(c->sz.nleaf);
  if (2 * K > 0x7fffffffLL) return set_error(c, FMM_EUNSUPPORTED, "too many leaf pairs (%lld)", (long long)K);
  AMFMM_TRY(ensure<double>(c, c->near, 3 * n));
  AMFMM_TRY(ensure<int32_t>(c, c->p2p_offA, nc + 1));
  AMFMM_TRY(ensure<int32_t>(c, c->p2p_itemOff, nleaf + 1));
  AMFMM_TRY(ensure<int32_t>(c, c->p2p_extraOff, nleaf + 1));
  AMFMM_TRY(ensure<int32_t>(c, c->incl, std::max<int64_t>(nc + 1, n + 1)));
  AMFMM_TRY(ensure<Rec>(c, c->p2p_rec, n));
  const bool forest = c->sz.nsys > 1;
  launch(c, k_body_fixed, grid_for(n, 256), 256, 0, n, ptr<double>(c->X), ptr<double>(c->Y), ptr<double>(c->Zb),
         ptr<double>(c->Mb), forest ? ptr<double>(c->sbox) : ptr<double>(c->bbox), ptr<int32_t>(c->order),
         forest ? ptr<int32_t>(c->sysid) : nullptr, ptr<Rec>(c->p2p_rec));
  AMFMM_TRY(launched(c, "p2p_body_fixed"));
  // every leaf's partners, in the stable order of the pair list
  int32_t *off = ptr<int32_t>(c->p2p_offA);
  AMFMM_TRY(partner_lists(c, ptr<int2>(c->p2p), K, c->pkey, c->pval, off, &c->p2p_which));
  // work items; totals: [33] items, [34] partial sums, stat: body pairs, [12] partial sums and [13] items in 64 bits
  int32_t *itot = ptr<int32_t>(c->totals) + 33, *etot = ptr<int32_t>(c->totals) + 34;
  unsigned long long *stat = ptr<unsigned long long>(c->totals) + 8;
  unsigned long long *ext64 = ptr<unsigned long long>(c->totals) + 12, *it64 = ext64 + 1;
  int32_t *icnt = ptr<int32_t>(c->incl), *ecnt = ptr<int32_t>(c->flag);  // free scratch of >= nleaf + 1
  int32_t *itemOff = ptr<int32_t>(c->p2p_itemOff), *extraOff = ptr<int32_t>(c->p2p_extraOff);
  launch(c, k_items64_count, grid_for(32 * (static_cast<int64_t>(nleaf) + 1), kCountBlock), kCountBlock, 0, nleaf,
         ptr<int32_t>(c->leaves), ptr<int32_t>(c->count), off, K > 0 ? ptr<uint32_t>(c->pval[c->p2p_which]) : nullptr,
         icnt, ecnt, stat, ext64, it64);
  AMFMM_TRY(launched(c, "p2p64_item_counts"));
  AMFMM_TRY(exclusive_scan_i32(c, icnt, itemOff, nleaf + 1, itot));
  AMFMM_TRY(exclusive_scan_i32(c, ecnt, extraOff, nleaf + 1, etot));
  int64_t *h = static_cast<int64_t *>(c->hpin);
  const HostRead rb{h, ext64, 2 * sizeof(int64_t)};
  AMFMM_TRY(read_back(c, &rb, 1));
  if (capturing(c)) {
    Expect e;
    for (int k = 0; k < 2; ++k) e.add64(ext64 + k, static_cast<uint64_t>(h[k]));
    AMFMM_TRY(graph_expect(c, e));
  }
  const int64_t nextra = h[0], nitem = h[1];
  if (nextra > 0x7fffffffLL || nitem > 0x7fffffffLL)
    return set_error(c, FMM_EUNSUPPORTED, "too many near-field work items (%lld) or partial sums (%lld)",
                     (long long)nitem, (long long)nextra);
  c->sz.p2p_items = nitem;
  AMFMM_TRY(ensure<int4>(c, c->p2p_items, nitem + 1));
  AMFMM_TRY(ensure<double>(c, c->p2p_extra, nextra + 1));
  launch(c, k_items64_fill, grid_for(nleaf, 256), 256, 0, nleaf, ptr<int32_t>(c->leaves), ptr<int32_t>(c->count), off,
         itemOff, extraOff, ptr<int4>(c->p2p_items));
  return launched(c, "p2p64_item_fill");
}

int p2p64_run(fmm_ctx *c) {
  const int32_t nitem = static_cast<int32_t>(c->sz.p2p_items), nleaf = static_cast<int32_t>(c->sz.nleaf);
  auto kern = c->eps2 == 0.0 ? k_p2p64<false> : k_p2p64<true>;
  int per_sm = 0;
  AMFMM_CUDA(c, cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kWarps * 32, 0));
  const int64_t resident = static_cast<int64_t>(std::max(1, per_sm)) * std::max(1, c->num_sms);
  const unsigned grid = static_cast<unsigned>(std::min<int64_t>(grid_for(nitem, kWarps), resident));
  int *queue = ptr<int32_t>(c->totals) + 40;
  launch(c, kern, grid, kWarps * 32, 0, nitem, c->sz.n, ptr<int4>(c->p2p_items), ptr<int32_t>(c->begin),
         ptr<int32_t>(c->count), ptr<int32_t>(c->p2p_offA),
         c->sz.n_p2p > 0 ? ptr<uint32_t>(c->pval[c->p2p_which]) : nullptr, ptr<Rec>(c->p2p_rec), ptr<double>(c->X),
         ptr<double>(c->Y), ptr<double>(c->Zb), ptr<double>(c->Mb), c->eps2, ptr<double>(c->near), ptr<double>(c->p2p_extra), queue);
  AMFMM_TRY(launched(c, "p2p"));
  if (c->sz.n_p2p == 0) return FMM_OK;
  launch(c, k_p2p64_groups, grid_for(static_cast<int64_t>(nleaf) * 32, 256), 256, 0, nleaf, c->sz.n,
         ptr<int32_t>(c->leaves), ptr<int32_t>(c->begin), ptr<int32_t>(c->count), ptr<int32_t>(c->p2p_offA),
         ptr<int32_t>(c->p2p_extraOff), ptr<double>(c->p2p_extra), ptr<double>(c->near));
  return launched(c, "p2p_groups");
}

}  // namespace amfmm
