// p2p.cu -- a8 in the mixed form: mutual near-field sums in FP32 (Sec. 2:
// "the force contributions from any remaining nearby particles are computed
// directly").  The FP64 form is p2p64.cu.
//
// For every leaf pair (A, B) each body pair (i in A, j in B) is evaluated
// once: with d = X_j - X_i and s = 1/|d|^3,
//     a_i += m_j s d,    a_j -= m_i s d,
// so the two contributions are equal and opposite (linear momentum is
// conserved pair by pair).  With Plummer softening, s = 1/(|d|^2 + eps^2)^(3/2).  A leaf with itself sums every ordered pair i != j
// once on the side of i.  A pair at zero separation contributes nothing.
//
// Work layout: one warp per leaf A.  Its columns are A's own bodies (summed
// one-sided, i != j) followed by the bodies of every leaf B paired with A as
// the smaller id (pairs sorted by A, stable), packed 32 columns to a step so
// that small leaves still fill the warp.  Each lane owns one column body j and
// loops over the rows i of A: the B-side sum b_j = sum_i m_i s_ij (X_i - X_j)
// stays in a register and is complete when the loop ends; the A-side term
// -m_j s_ij (X_i - X_j) goes to a per-(row, lane) partial in shared memory,
// summed over the lanes in lane order once per leaf.  b_j is written to the
// slot of (pair, body j); each body then adds its slots in the order of the
// stable sort.  Every sum has a fixed order; no atomics.
//
// Coordinates are relative to Z_A, formed from hi and lo floats; pair terms and
// the short sums (over the rows of one leaf, over one lane's columns) are FP32,
// every longer sum (lanes, slots, partners) FP64.
#include "internal.cuh"

namespace amfmm {
namespace {

// float -> double by integer operations (exact; subnormals, which this file
// flushes, as zero): the conversion instruction shares the slow FP64 path (sums of
// the partners' partials 184 -> 155 us at N = 1M, 734 -> 633 for a disc of 4M).
__device__ __forceinline__ double widen(float f) {
  const unsigned u = __float_as_uint(f), m = u & 0x7fffffffu;
  const unsigned off = m >= 0x7f800000u ? 0x70000000u : 0x38000000u;
  const unsigned hi = m < 0x00800000u ? 0u : (m >> 3) + off;
  return __hiloint2double(static_cast<int>(hi | (u & 0x80000000u)), static_cast<int>(m < 0x00800000u ? 0u : u << 29));
}

constexpr int kWarps = 4;
// Rows of A held in shared memory per pass (the leaf tile): 8, 16 or 32,
// chosen per context (fmm_set_tile, fmm_autotune).  16 measured best on a
// Plummer sphere of N = 1M: against 32 it halves the shared memory per warp
// and doubles the resident warps (1.68 -> 1.10 ms); 8 costs more column passes
// than it gains (1.22 ms).  Ensembles of small systems may prefer another tile.

// Shared memory per warp: the rows (bodies of A) and, per row and component,
// one running partial of the A-side sum for every lane.
template <int ROWS>
struct P2PSmem {
  alignas(16) float row[ROWS][4];  // x, y, z, m of the current row chunk (16-byte loads)
  float acc[ROWS * 3][32];         // A-side partial sums, [3 i + d][lane]
};
template <int ROWS>
__device__ __forceinline__ void acc_zero(P2PSmem<ROWS> &sm, int nr, int l) {
  for (int v = 0; v < 3 * nr; ++v) sm.acc[v][l] = 0.f;
}
// partial of row i, lane l -= s (dx, dy, dz).  (One float4 per (row, lane),
// one 16-byte load and store per update, measured 1% slower at N = 1M than
// these three scalar updates.)
template <int ROWS>
__device__ __forceinline__ void acc_sub(P2PSmem<ROWS> &sm, int i, int l, float s, float dx, float dy, float dz) {
  sm.acc[3 * i][l] = fmaf(-s, dx, sm.acc[3 * i][l]);
  sm.acc[3 * i + 1][l] = fmaf(-s, dy, sm.acc[3 * i + 1][l]);
  sm.acc[3 * i + 2][l] = fmaf(-s, dz, sm.acc[3 * i + 2][l]);
}

// below this squared separation two bodies count as coincident (their 1/r^3
// would leave the FP32 range)
constexpr float kMinR2 = 1e-30f;

// R consecutive rows i.. against one column body: the B-side sum
// in row order, then the A-side partials.
template <int R, int ROWS>
__device__ __forceinline__ void rows32(P2PSmem<ROWS> &sm, int i, int l, bool valid, bool mutual, float xj,
                                       float yj, float zj, float mj, float eps2, float &bx, float &by,
                                       float &bz) {
  float dx[R], dy[R], dz[R], r3[R];
#pragma unroll
  for (int u = 0; u < R; ++u) {
    const float4 rw = *reinterpret_cast<const float4 *>(sm.row[i + u]);
    dx[u] = rw.x - xj;
    dy[u] = rw.y - yj;
    dz[u] = rw.z - zj;
    const float r2 = fmaf(dz[u], dz[u], fmaf(dy[u], dy[u], fmaf(dx[u], dx[u], eps2)));
    const bool ok = valid && r2 > kMinR2;
    const float ri = ok ? rsqrtf(r2) : 0.f;
    r3[u] = ri * ri * ri;
    const float si = rw.w * r3[u];
    bx = fmaf(si, dx[u], bx);
    by = fmaf(si, dy[u], by);
    bz = fmaf(si, dz[u], bz);
  }
  if (mutual) {
#pragma unroll
    for (int u = 0; u < R; ++u) acc_sub(sm, i + u, l, mj * r3[u], dx[u], dy[u], dz[u]);
  }
}

// Bodies and the leaf centre are hi + lo floats, so an offset
// (x_hi - z_hi) + (x_lo - z_lo) is formed with FP32 operations only (FP64
// costs 64 FP32 operations on this GPU) and keeps FP32 relative accuracy.
__device__ __forceinline__ float3 offset32(const BodyF &b, const float4 zh, const float4 zl) {
  return make_float3((b.h.x - zh.x) + (b.l.x - zl.x), (b.h.y - zh.y) + (b.l.y - zl.y),
                     (b.h.z - zh.z) + (b.l.z - zl.z));
}

// Work items: the column stream of a leaf is cut into chunks of at most
// `chunk` columns (the first chunk also holds all of the leaf's own bodies,
// so that the one-sided self sums stay in one warp).  One warp per chunk
// keeps a leaf that the walk paired with millions of bodies (a large sparse
// leaf next to a dense region) from serialising the kernel.  Leaf order: there
// neighbouring warps share partner columns in cache.
//
// A leaf with a good part of what an average warp gets in all would still be what
// the kernel ends on, and a chunk cannot be made smaller: every lane's FP32 sum
// over a chunk's columns is one rounding sequence.  But the A side's rows are
// independent of one another, and so are the B side's columns: such a heavy
// leaf's chunks become items of kItemRows rows (A side only) and items of
// kItemCols columns (B side only), which evaluate its pairs twice, in the same
// order within every sum.  The line is half of the average work of the warps that run
// at once, in body pairs of a chunk, and at least 512 columns; and where not even a
// whole chunk of a whole leaf exceeds the average, no leaf is what the kernel ends on
// (262,144 bodies in leaves of up to 256: 5.4 ms, with half of the work in parts 6.3).
// Near field (us) without the rule, and with the line at the average itself, half, a
// third and a sixth of it: N = 65,536 (outlying leaves with up to 65,000 columns) 350,
// 141, 132, 136, 136;
// a forest of 48 systems 547, 543, 490, 496, 513; 200,000 bodies of two clusters 460,
// 292, 294, 290, 306; a disc of 262,144 518, 452, 377, 374, 395; N = 1M 803, 794, 773,
// 771, 802; leaves of up to 128 bodies at 1M 5,043, 5,154, 5,058, 5,276, 6,519, of up to
// 512 34,516, 34,442, 34,471, 34,560, 37,427 (54,362 with a line in columns, which
// made every large leaf heavy).
constexpr int kChunk = 4096;
constexpr int kItemRows = 4;
constexpr int kItemCols = 512;
constexpr int kHeavyMin = 512;
constexpr int kHeavyPart = 2;
// items {leaf, first column, end column, -1 or place in `extra`}; an item of a
// heavy leaf has the complement of the end column, and its first row, or -1 for
// the B side, in item_rows.  A heavy leaf's places: its self sums, then the
// A-side sums of every chunk.

__device__ __forceinline__ int chunks_of(int ncol, int nself) {
  const int first = max(kChunk, nself);
  return ncol <= first ? 1 : 1 + (ncol - first + kChunk - 1) / kChunk;
}
__device__ __forceinline__ int2 chunk_range(int j, int cb, int ce, int nself) {
  const int first = max(kChunk, nself);
  if (j == 0) return make_int2(cb, min(ce, cb + first));
  const int c0 = cb + first + (j - 1) * kChunk;
  return make_int2(c0, min(ce, c0 + kChunk));
}
// (counts of places and items in 64 bits: both are refused beyond 2^31 - 1)
// `pairs`: body pairs of all leaves; `warps`: that run at once; `full`: body pairs of
// a whole chunk of a whole leaf
__device__ __forceinline__ bool is_heavy(int ncol, int nA, const unsigned long long *pairs, int warps,
                                         long long full) {
  const long long chunk = static_cast<long long>(min(ncol, max(kChunk, nA))) * nA;
  const long long average = static_cast<long long>(*pairs) / warps;
  return ncol > kHeavyMin && chunk > average / kHeavyPart && max(chunk, full) > average;
}

__global__ void k_item_counts(int32_t nleaf, const int32_t *leaves, const int32_t *count,
                              const int32_t *colOff, const unsigned long long *pairs, int warps, long long full,
                              int32_t *__restrict__ nitems, int32_t *__restrict__ nextra, int *__restrict__ nheavy,
                              unsigned long long *__restrict__ wide) {
  pdl_wait();
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  unsigned long long items = 0, places = 0;
  if (q < nleaf) {
    if (q == 0) nitems[nleaf] = nextra[nleaf] = 0;
    const int L = leaves[q], cb = colOff[L], ce = colOff[L + 1], nA = count[L];
    const int k = chunks_of(ce - cb, nA);
    if (!is_heavy(ce - cb, nA, pairs, warps, full)) {
      items = k;
      places = (k - 1) * 3ull * nA;
    } else {
      for (int j = 0; j < k; ++j) {
        const int2 c = chunk_range(j, cb, ce, nA);
        items += (nA + kItemRows - 1) / kItemRows + (c.y - c.x + kItemCols - 1) / kItemCols;
      }
      atomicAdd(nheavy, 1);
      places = (k + 1) * 3ull * nA;
    }
    nitems[q] = static_cast<int32_t>(items);
    nextra[q] = static_cast<int32_t>(places);
  }
  // the totals: one addition per warp, exact in any order
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    items += __shfl_xor_sync(0xffffffffu, items, o);
    places += __shfl_xor_sync(0xffffffffu, places, o);
  }
  if ((threadIdx.x & 31) == 0) {
    if (items) atomicAdd(wide, items);
    if (places) atomicAdd(wide + 1, places);
  }
}

__global__ void k_item_fill(int32_t nleaf, const int32_t *leaves, const int32_t *count,
                            const int32_t *colOff, const unsigned long long *pairs, int warps, long long full,
                            const int32_t *itemOff, const int32_t *extraOff,
                            int4 *__restrict__ items, int32_t *__restrict__ item_rows) {
  pdl_wait();
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= nleaf) return;
  const int L = leaves[q];
  const int cb = colOff[L], ce = colOff[L + 1], nA = count[L];
  const int k = chunks_of(ce - cb, nA);
  const bool heavy = is_heavy(ce - cb, nA, pairs, warps, full);
  int o = itemOff[q];
  for (int j = 0; j < k; ++j) {
    const int2 c = chunk_range(j, cb, ce, nA);
    if (!heavy) {
      items[o++] = make_int4(L, c.x, c.y, j == 0 ? -1 : extraOff[q] + (j - 1) * 3 * nA);
      continue;
    }
    for (int r = 0; r < nA; r += kItemRows) {
      item_rows[o] = r;
      items[o++] = make_int4(L, c.x, ~c.y, extraOff[q] + (j + 1) * 3 * nA);
    }
    for (int b = c.x; b < c.y; b += kItemCols) {
      item_rows[o] = -1;
      items[o++] = make_int4(L, b, ~min(c.y, b + kItemCols), extraOff[q]);
    }
  }
}

// A leaf whose column stream was split adds the A-side partials of its later
// chunks, in chunk order, once every chunk is done (one thread per body); a
// heavy leaf its self sums and those of all chunks.
__global__ void k_p2p_chunks(int32_t nleaf, int64_t n, const int32_t *leaves,
                             const int32_t *begin, const int32_t *count,
                             const int32_t *colOff, const unsigned long long *pairs, int warps, long long full,
                             const int32_t *extraOff, const double *extra,
                             double *__restrict__ near) {
  pdl_wait();
  const int q = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int l = threadIdx.x & 31;
  if (q >= nleaf) return;
  const int e0 = extraOff[q], e1 = extraOff[q + 1];
  if (e0 == e1) return;
  const int L = leaves[q];
  const int bA = begin[L], nA = count[L];
  const bool heavy = is_heavy(colOff[L + 1] - colOff[L], nA, pairs, warps, full);
  for (int r = l; r < nA; r += 32) {
    double a0 = 0.0, a1 = 0.0, a2 = 0.0;
    if (!heavy) {
      a0 = near[bA + r];
      a1 = near[n + bA + r];
      a2 = near[2 * n + bA + r];
    }
    for (int k = e0; k < e1; k += 3 * nA) {
      const double *e = extra + k + 3 * r;
      a0 += e[0];
      a1 += e[1];
      a2 += e[2];
    }
    near[bA + r] = a0;
    near[n + bA + r] = a1;
    near[2 * n + bA + r] = a2;
  }
}

// The FP64 sums of a body have one order, however its leaf is worked on (the line
// of heavy leaves depends on the whole call, and a system solved alone and in a
// forest must agree): the self sums of all passes over the leaf's rows, then the A
// side of its chunks in order.  A leaf of several passes keeps the first chunk's
// A-side sums in `late` until the last.
// HEAVY: there are items of heavy leaves (the test for them costs 1% otherwise).
template <int ROWS, bool HEAVY>
__global__ void __launch_bounds__(kWarps * 32) k_p2p(
    int32_t nitem, int64_t n, const int4 *items, const int32_t *item_rows,
    const int32_t *begin, const int32_t *count, const double *Zc, const int2 *cols,
    double *__restrict__ near, double *__restrict__ late, double *__restrict__ extra, float *__restrict__ slots,
    const BodyF *bodyf, float eps2, int *__restrict__ queue) {
  pdl_wait();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  P2PSmem<ROWS> &sm = reinterpret_cast<P2PSmem<ROWS> *>(smem_raw)[w];
  // Work items differ in size by orders of magnitude, so warps draw them
  // from a queue until it is empty instead of taking a fixed one: a block's
  // warps then never wait for one another's items (the grid is as large as
  // fits on the GPU at once).  Which warp takes an item does not change what
  // it computes or where it writes.
  for (;;) {
  int q = 0;
  if (l == 0) q = atomicAdd(queue, 1);
  q = __shfl_sync(0xffffffffu, q, 0);
  if (q >= nitem) break;
  // work item: leaf, column range; w < 0 marks the leaf's first chunk (which
  // owns the near-field sums of the leaf), w >= 0 the offset of a later
  // chunk's A-side partials in `extra`
  const int4 it = items[q];
  const int L = it.x;
  const bool first = it.w < 0;
  const int bA = begin[L], nA = count[L];
  // an item of a heavy leaf (see k_item_fill): rows [ra, rb) on the A side, or the
  // columns' B side
  const bool heavy = HEAVY && it.z < 0;
  const int part = heavy ? item_rows[q] : 0;
  const bool sideA = !heavy || part >= 0, sideB = !heavy || part < 0;
  const int ra = heavy && sideA ? part : 0, rb = heavy && sideA ? min(nA, part + kItemRows) : nA;
  const double zx = Zc[3 * L], zy = Zc[3 * L + 1], zz = Zc[3 * L + 2];
  const float4 zh = make_float4(static_cast<float>(zx), static_cast<float>(zy), static_cast<float>(zz), 0.f);
  const float4 zl =
      make_float4(static_cast<float>(zx - zh.x), static_cast<float>(zy - zh.y), static_cast<float>(zz - zh.z), 0.f);
  const int cb = it.y, ce = heavy ? ~it.z : it.z;
  if (first) {
    for (int t = l; t < nA; t += 32) {
      near[bA + t] = 0.0;
      near[n + bA + t] = 0.0;
      near[2 * n + bA + t] = 0.0;
    }
  }
  __syncwarp();
  constexpr int kRows = ROWS;
  for (int r0 = ra; r0 < rb; r0 += kRows) {
    const int nr = min(kRows, rb - r0);
    if (l < nr) {
      const int i = bA + r0 + l;
      const BodyF b = bodyf[i];
      const float3 o = offset32(b, zh, zl);
      sm.row[l][0] = o.x;
      sm.row[l][1] = o.y;
      sm.row[l][2] = o.z;
      sm.row[l][3] = b.h.w;
    }
    acc_zero(sm, nr, l);
    __syncwarp();
    // columns: A's own bodies (one-sided, self) then the bodies of every
    // partner leaf B with A < B, packed 32 to a step.  Loads run ahead: the
    // column entry two steps ahead, the body of the next step.
    int2 colN = cb + l < ce ? cols[cb + l] : make_int2(0, -2);
    BodyF rbN{};
    if (cb + l < ce) rbN = bodyf[colN.x];
    int2 colNN = cb + 32 + l < ce ? cols[cb + 32 + l] : make_int2(0, -2);
    for (int c0 = cb; c0 < ce; c0 += 32) {
      const bool valid = c0 + l < ce;
      const int2 col = colN;
      const BodyF rb = rbN;
      colN = colNN;
      if (c0 + 32 + l < ce) rbN = bodyf[colN.x];
      colNN = c0 + 64 + l < ce ? cols[c0 + 64 + l] : make_int2(0, -2);
      float xj = 0.f, yj = 0.f, zj = 0.f, mj = 0.f;
      if (valid) {
        const float3 o = offset32(rb, zh, zl);
        xj = o.x;
        yj = o.y;
        zj = o.z;
        mj = rb.h.w;
      }
      const bool mutual = col.y >= 0 && sideA;
      float bx = 0.f, by = 0.f, bz = 0.f;
      // eight rows per step, then four and two: independent dependency chains
      // for the pipelines and less loop control per pair
      int i = 0;
      for (; i + 7 < nr; i += 8) rows32<8, ROWS>(sm, i, l, valid, mutual, xj, yj, zj, mj, eps2, bx, by, bz);
      for (; i + 3 < nr; i += 4) rows32<4, ROWS>(sm, i, l, valid, mutual, xj, yj, zj, mj, eps2, bx, by, bz);
      for (; i + 1 < nr; i += 2) rows32<2, ROWS>(sm, i, l, valid, mutual, xj, yj, zj, mj, eps2, bx, by, bz);
      for (; i < nr; ++i) {
        const float dx = sm.row[i][0] - xj, dy = sm.row[i][1] - yj, dz = sm.row[i][2] - zj;
        // softening enters as the addend of the first product (no extra
        // operation; eps2 = 0 gives the unsoftened sum)
        const float r2 = fma(dz, dz, fma(dy, dy, fma(dx, dx, eps2)));
        if (valid && r2 > kMinR2) {
          const float ri = rsqrtf(r2);
          const float r3 = ri * ri * ri;
          const float si = sm.row[i][3] * r3;
          bx = fmaf(si, dx, bx);
          by = fmaf(si, dy, by);
          bz = fmaf(si, dz, bz);
          if (mutual) {
            const float sj = mj * r3;
            acc_sub(sm, i, l, sj, dx, dy, dz);
          }
        }
      }
      if (valid && sideB) {
        if (col.y >= 0) {
          float *o = slots + 3 * static_cast<int64_t>(col.y);
          if (r0 == 0) {
            o[0] = bx;
            o[1] = by;
            o[2] = bz;
          } else {
            o[0] += bx;
            o[1] += by;
            o[2] += bz;
          }
        } else if (heavy) {
          double *o = extra + it.w + 3 * (col.x - bA);
          const bool set = r0 == 0;
          o[0] = (set ? 0.0 : o[0]) + static_cast<double>(bx);
          o[1] = (set ? 0.0 : o[1]) + static_cast<double>(by);
          o[2] = (set ? 0.0 : o[2]) + static_cast<double>(bz);
        } else {
          near[col.x] += static_cast<double>(bx);
          near[n + col.x] += static_cast<double>(by);
          near[2 * n + col.x] += static_cast<double>(bz);
        }
      }
    }
    __syncwarp();
    // A-side: every row's partials summed over the lanes in a fixed order,
    // pairwise in FP32, then one FP64 addition
    for (int v = l; sideA && v < 3 * nr; v += 32) {
      float g[4];
#pragma unroll
      for (int h = 0; h < 4; ++h) {
        float a[8];
#pragma unroll
        for (int t = 0; t < 8; ++t) a[t] = sm.acc[v][8 * h + t];
        g[h] = ((a[0] + a[1]) + (a[2] + a[3])) + ((a[4] + a[5]) + (a[6] + a[7]));
      }
      const double s = static_cast<double>((g[0] + g[1]) + (g[2] + g[3]));
      const int64_t body = static_cast<int64_t>(v % 3) * n + bA + r0 + v / 3;
      if (first && nA <= kRows) near[body] += s;
      else if (first) late[body] = s;
      else extra[it.w + 3 * (r0 + v / 3) + v % 3] = s;
    }
    __syncwarp();
  }
  if (first && nA > kRows)
    for (int t = l; t < nA; t += 32)
#pragma unroll
      for (int d = 0; d < 3; ++d) near[d * n + bA + t] += late[d * n + bA + t];
  }
}

// Each body adds, in sorted order, the partials that the pairs in which its
// leaf is the larger id left for it.
__global__ void k_p2p_reduce(int64_t n, const int32_t *leaf_of, const int32_t *begin,
                             const int32_t *offB, const int64_t *poff,
                             const float *slots, double *__restrict__ near) {
  pdl_wait();
  const int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
  if (i >= n) return;
  const int L = leaf_of[i];
  const int t = static_cast<int>(i - begin[L]);
  double a0 = near[i], a1 = near[n + i], a2 = near[2 * n + i];
  int e = offB[L];
  const int e1 = offB[L + 1];
  // FP32 partials: sums of eight in FP32 (fixed order), accumulated in FP64
  for (; e + 8 <= e1; e += 8) {
    float s0 = 0.f, s1 = 0.f, s2 = 0.f;
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const float *p = slots + poff[e + u] + 3 * t;
      s0 += p[0];
      s1 += p[1];
      s2 += p[2];
    }
    a0 += widen(s0);
    a1 += widen(s1);
    a2 += widen(s2);
  }
  for (; e < e1; ++e) {
    const float *p = slots + poff[e] + 3 * t;
    a0 += widen(p[0]);
    a1 += widen(p[1]);
    a2 += widen(p[2]);
  }
  near[i] = a0;
  near[n + i] = a1;
  near[2 * n + i] = a2;
}

// the sorted (A, B) as pairs, and every pair's column count n_B (and a zero for
// the total of the scan)
__global__ void k_sorted_pairs(int64_t K, const uint32_t *key, const uint32_t *val,
                               const int32_t *count, int2 *__restrict__ out, int32_t *__restrict__ nb) {
  pdl_wait();
  const int64_t s = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
  if (s >= K) return;
  const int2 p = make_int2(static_cast<int>(key[s]), static_cast<int>(val[s]));
  out[s] = p;
  nb[s] = count[p.y];
  if (s == 0) nb[K] = 0;
}

// pos[s] = CSR position of sorted pair s on its B side; len[e] = 3 n_B
__global__ void k_b_positions(int64_t K, const uint32_t *key, const uint32_t *sval,
                              const int32_t *count, int32_t *__restrict__ pos,
                              int64_t *__restrict__ len) {
  pdl_wait();
  const int64_t e = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
  if (e >= K) return;
  pos[sval[e]] = static_cast<int32_t>(e);
  len[e] = 3 * static_cast<int64_t>(count[key[e]]);
}

int bits_for(int64_t v) {
  int b = 1;
  while ((int64_t(1) << b) <= v) ++b;
  return b;
}

// Columns of every leaf: first its own bodies (marked -1: one-sided), then the
// bodies of its partner leaves in the A-sorted pair order, each with the slot
// that receives its B-side partial.
// Column count of every leaf A: its own bodies plus, from the prefix sums
// pre of the partners' sizes over the A-sorted pairs, the bodies of its
// partners.  Also the near-field work: n_A n_B per leaf pair plus
// n (n - 1) / 2 per leaf (one atomic per warp, integer: exact).
__global__ void k_leaf_cols(int32_t nleaf, const int32_t *leaves, const int32_t *count,
                            const int32_t *offA, const int32_t *pre,
                            int32_t *__restrict__ ccount, unsigned long long *__restrict__ work) {
  pdl_wait();
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  unsigned long long v = 0;
  if (q < nleaf) {
    const int L = leaves[q];
    const int a = count[L];
    const int cols = pre ? pre[offA[L + 1]] - pre[offA[L]] : 0;
    ccount[L] = a + cols;
    v = static_cast<unsigned long long>(a) * cols + static_cast<unsigned long long>(a) * (a - 1) / 2;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0 && v) atomicAdd(work, v);
}

__global__ void k_cols_self(int32_t nleaf, const int32_t *leaves, const int32_t *begin,
                            const int32_t *count, const int32_t *colOff,
                            int2 *__restrict__ cols) {
  pdl_wait();
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= nleaf) return;
  const int L = leaves[q];
  const int b = begin[L], c0 = colOff[L];
  for (int t = 0; t < count[L]; ++t) cols[c0 + t] = make_int2(b + t, -1);
}

__global__ void k_cols_pairs(int64_t K, const int2 *pairs, const int32_t *begin,
                             const int32_t *count, const int32_t *colOff,
                             const int32_t *offA, const int32_t *pre,
                             const int32_t *pos, const int64_t *poff,
                             int2 *__restrict__ cols) {
  pdl_wait();
  // A warp writes the runs of its 32 pairs together: entry j of the warp's
  // concatenated runs goes to lane j mod 32, which finds the pair owning it
  // by a binary search over the warp's prefix sums, so consecutive lanes
  // store consecutive entries of a run.
  const int64_t k = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
  const int lane = threadIdx.x & 31;
  int nB = 0, base = 0, bB = 0;
  long long o = 0;
  if (k < K) {
    const int2 p = pairs[k];
    base = colOff[p.x] + count[p.x] + (pre[k] - pre[offA[p.x]]);
    bB = begin[p.y];
    o = poff[pos[k]];
    nB = count[p.y];
  }
  int incl = nB;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, incl, d);
    if (lane >= d) incl += y;
  }
  const int excl = incl - nB;
  const int total = __shfl_sync(0xffffffffu, incl, 31);
  for (int j0 = 0; j0 < total; j0 += 32) {
    const int j = j0 + lane;
    int own = 0;  // number of lanes whose run ends at or before j
#pragma unroll
    for (int step = 16; step > 0; step >>= 1) {
      const int e = __shfl_sync(0xffffffffu, incl, own + step - 1);
      if (e <= j) own += step;
    }
    own = min(own, 31);
    const int b = __shfl_sync(0xffffffffu, base, own), x = __shfl_sync(0xffffffffu, excl, own);
    const int bb = __shfl_sync(0xffffffffu, bB, own);
    const long long oo = __shfl_sync(0xffffffffu, o, own);
    if (j < total) {
      const int t = j - x;
      // the slot's index (its offset / 3): 3x the range of an int32 offset
      cols[b + t] = make_int2(bb + t, static_cast<int32_t>(oo / 3 + t));
    }
  }
}

// the warps that the rule of heavy leaves counts with (16 run per SM at the
// default tile; the rule must be the same in every stage of a solve)
int heavy_warps(const fmm_ctx *c) { return 16 * std::max(1, c->num_sms); }
long long full_chunk(const fmm_ctx *c) {
  const long long rows = std::min<int64_t>(c->opts.n_crit, c->sz.n);
  return std::max<long long>(kChunk, rows) * rows;
}

template <int ROWS, bool HEAVY>
int launch_p2p_rows(fmm_ctx *c) {
  const int64_t n = c->sz.n;
  const int32_t nleaf = static_cast<int32_t>(c->sz.nleaf);
  const size_t shm = kWarps * sizeof(P2PSmem<ROWS>);
  // per function and device, so set on every launch (a host-side call)
  AMFMM_CUDA(c, cudaFuncSetAttribute(k_p2p<ROWS, HEAVY>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     static_cast<int>(shm)));
  const int32_t nitem = static_cast<int32_t>(c->sz.p2p_items);
  int per_sm = 0;
  AMFMM_CUDA(c, cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_p2p<ROWS, HEAVY>, kWarps * 32, shm));
  const int64_t resident = static_cast<int64_t>(std::max(1, per_sm)) * std::max(1, c->num_sms);
  const unsigned grid = static_cast<unsigned>(std::min<int64_t>(grid_for(nitem, kWarps), resident));
  int *queue = ptr<int32_t>(c->totals) + 40;
  launch(c, k_p2p<ROWS, HEAVY>, grid, kWarps * 32, shm, nitem, n, ptr<int4>(c->p2p_items), ptr<int32_t>(c->p2p_rowpart),
         ptr<int32_t>(c->begin), ptr<int32_t>(c->count), ptr<double>(c->Z), ptr<int2>(c->p2p_cols), ptr<double>(c->near),
         ptr<double>(c->acc), ptr<double>(c->p2p_extra), static_cast<float *>(c->p2p_slots.p), ptr<BodyF>(c->bodyf),
         static_cast<float>(c->eps2), queue);
  AMFMM_TRY(launched(c, "p2p"));
  if (nitem > nleaf) {
    launch(c, k_p2p_chunks, grid_for(static_cast<int64_t>(nleaf) * 32, 256), 256, 0, nleaf, n, ptr<int32_t>(c->leaves),
           ptr<int32_t>(c->begin), ptr<int32_t>(c->count), ptr<int32_t>(c->p2p_colOff),
           ptr<unsigned long long>(c->totals) + 8, heavy_warps(c), full_chunk(c), ptr<int32_t>(c->p2p_extraOff),
           ptr<double>(c->p2p_extra), ptr<double>(c->near));
    AMFMM_TRY(launched(c, "p2p_chunks"));
  }
  return FMM_OK;
}

}  // namespace

int p2p_prepare(fmm_ctx *c) {
  cudaStream_t st = c->stream;
  const int64_t K = c->sz.n_p2p, nc = c->sz.ncell, n = c->sz.n;
  const int32_t nleaf = static_cast<int32_t>(c->sz.nleaf);
  AMFMM_TRY(ensure<double>(c, c->near, 3 * n));
  AMFMM_TRY(ensure<double>(c, c->acc, 3 * n));  // A-side sums of leaves of several passes; the downward pass writes it
  AMFMM_TRY(ensure<int32_t>(c, c->p2p_offA, nc + 1));
  AMFMM_TRY(ensure<int32_t>(c, c->p2p_offB, nc + 1));
  AMFMM_TRY(ensure<int32_t>(c, c->p2p_colOff, nc + 1));
  AMFMM_TRY(ensure<int64_t>(c, c->p2p_poff, K + 1));
  AMFMM_TRY(ensure<int32_t>(c, c->p2p_pos, K + 1));
  AMFMM_TRY(ensure<int2>(c, c->p2p_A, K + 1));
  AMFMM_TRY(ensure<int32_t>(c, c->incl, std::max<int64_t>(nc + 1, n + 1)));
  int32_t *cnt = ptr<int32_t>(c->incl);
  int32_t *offA = ptr<int32_t>(c->p2p_offA), *offB = ptr<int32_t>(c->p2p_offB);
  int32_t *colOff = ptr<int32_t>(c->p2p_colOff);
  unsigned long long *stat = ptr<unsigned long long>(c->totals) + 8;
  int32_t *ctot = ptr<int32_t>(c->totals) + 32;
  AMFMM_TRY(ensure<int32_t>(c, c->p2p_nb, K + 1));
  AMFMM_TRY(ensure<int32_t>(c, c->p2p_pre, K + 1));
  int32_t *nb = ptr<int32_t>(c->p2p_nb), *pre = ptr<int32_t>(c->p2p_pre);
  int64_t *h = static_cast<int64_t *>(c->hpin);
  h[0] = 0;
  if (K > 0) {
    // group by A (stable), with the column counts n_B
    int which = 0;
    AMFMM_TRY(sort_pairs(c, ptr<int2>(c->p2p), K, false, c->pkey, c->pval, bits_for(nc), &which));
    AMFMM_TRY(segment_offsets(c, K, ptr<uint32_t>(c->pkey[which]), offA));
    launch(c, k_sorted_pairs, grid_for(K, 256), 256, 0, K, ptr<uint32_t>(c->pkey[which]),
           ptr<uint32_t>(c->pval[which]), ptr<int32_t>(c->count), ptr<int2>(c->p2p_A), nb);
    AMFMM_TRY(launched(c, "p2p_sorted_pairs"));
    // CSR on the B side; slot offsets: 3 n_B floats per pair, in that order
    AMFMM_TRY(sort_pairs(c, ptr<int2>(c->p2p_A), K, true, c->pkey, c->pval, bits_for(nc), &which));
    AMFMM_TRY(segment_offsets(c, K, ptr<uint32_t>(c->pkey[which]), offB));
    AMFMM_TRY(ensure<int64_t>(c, c->p2p_len, K + 1));
    int64_t *len = ptr<int64_t>(c->p2p_len);
    launch(c, k_b_positions, grid_for(K, 256), 256, 0, K, ptr<uint32_t>(c->pkey[which]), ptr<uint32_t>(c->pval[which]),
           ptr<int32_t>(c->count), ptr<int32_t>(c->p2p_pos), len);
    AMFMM_TRY(launched(c, "p2p_bpos"));
    int64_t *ptot = ptr<int64_t>(c->totals) + 12;
    AMFMM_TRY(exclusive_scan_i64(c, len, ptr<int64_t>(c->p2p_poff), K, ptot));
  }
  // column stream per leaf: pre = prefix sums of n_B over the A-sorted pairs
  // (K + 1 entries, so pre[K] is the total)
  if (K > 0) {
    AMFMM_TRY(exclusive_scan_i32(c, nb, pre, K + 1, nullptr));
  }
  AMFMM_CUDA(c, cudaMemsetAsync(cnt, 0, sizeof(int32_t) * (nc + 1), st));
  launch(c, k_leaf_cols, grid_for(nleaf, 256), 256, 0, nleaf, ptr<int32_t>(c->leaves), ptr<int32_t>(c->count), offA,
         K > 0 ? pre : nullptr, cnt, stat);
  AMFMM_TRY(launched(c, "p2p_leaf_cols"));
  AMFMM_TRY(exclusive_scan_i32(c, cnt, colOff, nc + 1, ctot));
  // work items: chunks of the column streams
  AMFMM_TRY(ensure<int32_t>(c, c->p2p_itemOff, nleaf + 1));
  AMFMM_TRY(ensure<int32_t>(c, c->p2p_extraOff, nleaf + 1));
  int32_t *itemOff = ptr<int32_t>(c->p2p_itemOff), *extraOff = ptr<int32_t>(c->p2p_extraOff);
  // totals: [32] columns, [33] work items, [34] extra partials, [35] heavy leaves (int32 slots), and
  // [13] work items, [14] extra partials in 64 bits
  int32_t *itot = ptr<int32_t>(c->totals) + 33, *etot = ptr<int32_t>(c->totals) + 34;
  int32_t *nheavy = ptr<int32_t>(c->totals) + 35;
  unsigned long long *wide = ptr<unsigned long long>(c->totals) + 13;
  int32_t *icnt = cnt, *ecnt = ptr<int32_t>(c->flag);  // free scratch of >= nleaf + 1
  launch(c, k_item_counts, grid_for(nleaf, 256), 256, 0, nleaf, ptr<int32_t>(c->leaves), ptr<int32_t>(c->count),
         colOff, stat, heavy_warps(c), full_chunk(c), icnt, ecnt, nheavy, wide);
  AMFMM_TRY(launched(c, "p2p_item_counts"));
  AMFMM_TRY(exclusive_scan_i32(c, icnt, itemOff, nleaf + 1, itot));
  AMFMM_TRY(exclusive_scan_i32(c, ecnt, extraOff, nleaf + 1, etot));
  int64_t *hw = h + 1;
  int32_t *hc = reinterpret_cast<int32_t *>(h + 3);
  {
    // (totals[12], the slot total, is not written after its scan)
    const int64_t *ptot = ptr<int64_t>(c->totals) + 12;
    HostRead rb[3];
    int nr = 0;
    if (K > 0) rb[nr++] = HostRead{h, ptot, sizeof(int64_t)};
    rb[nr++] = HostRead{hw, wide, 2 * sizeof(int64_t)};
    rb[nr++] = HostRead{hc, ctot, 4 * sizeof(int32_t)};
    AMFMM_TRY(read_back(c, rb, nr));
    if (capturing(c)) {
      Expect e;
      if (K > 0) e.add64(ptot, static_cast<uint64_t>(h[0]));
      for (int k = 0; k < 2; ++k) e.add64(wide + k, static_cast<uint64_t>(hw[k]));
      for (int k = 0; k < 4; ++k) e.add(ctot + k, static_cast<uint32_t>(hc[k]));
      AMFMM_TRY(graph_expect(c, e));
      st = c->stream;
    }
  }
  const int64_t nslot = h[0], ncol = hc[0];
  const int64_t nitem = hc[1], nextra = hc[2];
  // the columns (one per body of A and per slot: n + nslot / 3) are counted
  // by int32 scans and a slot is named by its int32 index: refuse before
  // anything is sized or launched from these totals
  if (nslot / 3 + n + 1 > 0x7fffffffLL)
    return set_error(c, FMM_EUNSUPPORTED, "too many near-field slots (%lld values)", (long long)nslot);
  if (hw[0] > 0x7fffffffLL || hw[1] > 0x7fffffffLL)
    return set_error(c, FMM_EUNSUPPORTED, "too many near-field work items (%lld) or partial sums (%lld)",
                     (long long)hw[0], (long long)hw[1]);
  c->sz.p2p_items = nitem;
  c->sz.p2p_heavy_leaves = hc[3];
  AMFMM_TRY(ensure<int4>(c, c->p2p_items, nitem + 1));
  AMFMM_TRY(ensure<double>(c, c->p2p_extra, nextra + 1));
  AMFMM_TRY(ensure<int32_t>(c, c->p2p_rowpart, nitem + 1));
  launch(c, k_item_fill, grid_for(nleaf, 256), 256, 0, nleaf, ptr<int32_t>(c->leaves), ptr<int32_t>(c->count), colOff,
         stat, heavy_warps(c), full_chunk(c), itemOff, extraOff, ptr<int4>(c->p2p_items), ptr<int32_t>(c->p2p_rowpart));
  AMFMM_TRY(launched(c, "p2p_item_fill"));
  AMFMM_TRY(ensure_bytes(c, c->p2p_slots, static_cast<size_t>(nslot + 3) * sizeof(float)));
  AMFMM_TRY(ensure<int2>(c, c->p2p_cols, ncol + 1));
  launch(c, k_cols_self, grid_for(nleaf, 256), 256, 0, nleaf, ptr<int32_t>(c->leaves), ptr<int32_t>(c->begin),
         ptr<int32_t>(c->count), colOff, ptr<int2>(c->p2p_cols));
  AMFMM_TRY(launched(c, "p2p_cols_self"));
  if (K > 0) {
    launch(c, k_cols_pairs, grid_for(K, 256), 256, 0, K, ptr<int2>(c->p2p_A), ptr<int32_t>(c->begin),
           ptr<int32_t>(c->count), colOff, offA, pre, ptr<int32_t>(c->p2p_pos), ptr<int64_t>(c->p2p_poff),
           ptr<int2>(c->p2p_cols));
    AMFMM_TRY(launched(c, "p2p_cols_pairs"));
  }
  return FMM_OK;
}

int p2p_run(fmm_ctx *c) {
  const bool heavy = c->sz.p2p_heavy_leaves > 0;
  switch (c->p2p_rows) {
    case 8: return heavy ? launch_p2p_rows<8, true>(c) : launch_p2p_rows<8, false>(c);
    case 32: return heavy ? launch_p2p_rows<32, true>(c) : launch_p2p_rows<32, false>(c);
    default: return heavy ? launch_p2p_rows<16, true>(c) : launch_p2p_rows<16, false>(c);
  }
}

int p2p_reduce(fmm_ctx *c) {
  if (c->sz.n_p2p == 0) return FMM_OK;
  const int64_t n = c->sz.n;
  launch(c, k_p2p_reduce, grid_for(n, 256), 256, 0, n, ptr<int32_t>(c->leaf_of), ptr<int32_t>(c->begin),
         ptr<int32_t>(c->p2p_offB), ptr<int64_t>(c->p2p_poff), static_cast<float *>(c->p2p_slots.p),
         ptr<double>(c->near));
  return launched(c, "p2p_reduce");
}

}  // namespace amfmm
