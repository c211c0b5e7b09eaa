// tree.cu -- a1-a4: bounding cube, Morton keys, sort, octree, centres of mass,
// R_max and moments.
//
// Sec. 2 of the paper: the bodies are decomposed into an oct-tree whose cells
// hold at most n_crit bodies; the opening criterion uses each cell's centre
// of mass Z and R_max, the largest distance from one of its bodies to Z.
// Because the interaction lists depend on exact comparisons of Z and R_max,
// every operation on that path is an explicitly rounded FP64 operation in a
// fixed order (no FMA contraction): leaf sums run over the bodies in sorted
// order, other cells sum their children in octant order, Z = S / M, and R_max
// is the exact maximum over the cell's bodies.
#include "internal.cuh"

namespace amfmm {
namespace {

constexpr int kBlock = 256;

// ---------------------------------------------------------------------------
// a1: bounding cube and keys
// ---------------------------------------------------------------------------
// Finite doubles as integers of the same order: minima and maxima then need no
// FP64 instruction (64 cycles of their pipe per warp).
__device__ __forceinline__ long long ordered(double v) {
  const long long b = __double_as_longlong(v);
  return b < 0 ? b ^ 0x7fffffffffffffffll : b;
}
__device__ __forceinline__ double from_ordered(long long k) {
  return __longlong_as_double(k < 0 ? k ^ 0x7fffffffffffffffll : k);
}
__device__ __forceinline__ bool finite_bits(double v) { return (__double2hiint(v) & 0x7ff00000) != 0x7ff00000; }

// Extremes of coordinates, in thread 0 those of the whole block.  body_extremes
// sets bit 0 of status for a coordinate that is not finite or a mass that is not
// finite and positive.
struct Extremes {
  long long lo[3], hi[3];
  __device__ __forceinline__ void combine(int d, long long l, long long h) {
    lo[d] = min(lo[d], l);
    hi[d] = max(hi[d], h);
  }
};
__device__ __forceinline__ void block_extremes(Extremes &v) {
  __shared__ long long sh[6][kBlock / 32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    for (int o = 16; o > 0; o >>= 1)
      v.combine(d, __shfl_xor_sync(0xffffffffu, v.lo[d], o), __shfl_xor_sync(0xffffffffu, v.hi[d], o));
    if (lane == 0) {
      sh[d][w] = v.lo[d];
      sh[3 + d][w] = v.hi[d];
    }
  }
  __syncthreads();
  if (threadIdx.x == 0)
    for (int d = 0; d < 3; ++d)
      for (int q = 1; q < kBlock / 32; ++q) v.combine(d, sh[d][q], sh[3 + d][q]);
}
__device__ __forceinline__ Extremes no_extremes() {
  Extremes v;
  for (int d = 0; d < 3; ++d) {
    v.lo[d] = 0x7fffffffffffffffll;
    v.hi[d] = -0x7fffffffffffffffll - 1;
  }
  return v;
}
__device__ __forceinline__ Extremes body_extremes(const double *x, const double *y,
                                                  const double *z, const double *m,
                                                  int64_t first, int64_t end, int64_t stride, int *status) {
  Extremes v = no_extremes();
  bool bad = false;
  for (int64_t i = first; i < end; i += stride) {
    const double p[3] = {x[i], y[i], z[i]}, mi = m[i];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      bad |= !finite_bits(p[d]);
      v.combine(d, ordered(p[d]), ordered(p[d]));
    }
    bad |= __double_as_longlong(mi) <= 0 || !finite_bits(mi);
  }
  if (bad) atomicOr(status, 1);
  block_extremes(v);
  return v;
}
// box[0..2] = lo, box[3] = scale = 2^21 / ext (0 when ext == 0)
__device__ __forceinline__ void write_box(const Extremes &v, double *__restrict__ box) {
  double ext = 0.0;
  for (int d = 0; d < 3; ++d) {
    const double lo = from_ordered(v.lo[d]), e = __dsub_rn(from_ordered(v.hi[d]), lo);
    ext = d == 0 ? e : fmax(ext, e);
    box[d] = lo;
  }
  box[3] = ext > 0.0 ? __ddiv_rn(2097152.0, ext) : 0.0;
}

// Bounding cube: every block its part, the last one to finish the whole (minima
// and maxima are exact, so their order does not matter).  14 us at N = 1M; two
// launches with FP64 comparisons took 45.6 + 10.1.
__global__ void k_bbox(const double *x, const double *y, const double *z,
                       const double *m, int64_t n, long long *__restrict__ part,
                       int *__restrict__ status, unsigned *__restrict__ done, double *__restrict__ bbox) {
  pdl_wait();
  __shared__ bool last;
  Extremes v = body_extremes(x, y, z, m, blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x, n,
                             static_cast<int64_t>(gridDim.x) * blockDim.x, status);
  if (threadIdx.x == 0) {
    for (int d = 0; d < 3; ++d) {
      part[6 * blockIdx.x + d] = v.lo[d];
      part[6 * blockIdx.x + 3 + d] = v.hi[d];
    }
    __threadfence();
    last = atomicAdd(done, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  v = no_extremes();
  for (unsigned b = threadIdx.x; b < gridDim.x; b += blockDim.x)
    for (int d = 0; d < 3; ++d)
      v.combine(d, *const_cast<volatile long long *>(&part[6 * b + d]),
                *const_cast<volatile long long *>(&part[6 * b + 3 + d]));
  block_extremes(v);
  if (threadIdx.x == 0) write_box(v, bbox);
}

__device__ __forceinline__ uint64_t quantise(double v, double lo, double scale) {
  return static_cast<uint64_t>(min(__double2int_rd(__dmul_rn(__dsub_rn(v, lo), scale)), 2097151));
}

// bit b of q -> bit 3b
__device__ __forceinline__ uint64_t spread3(uint64_t q) {
  q &= 0x1fffffull;
  q = (q | (q << 32)) & 0x1f00000000ffffull;
  q = (q | (q << 16)) & 0x1f0000ff0000ffull;
  q = (q | (q << 8)) & 0x100f00f00f00f00full;
  q = (q | (q << 4)) & 0x10c30c30c30c30c3ull;
  q = (q | (q << 2)) & 0x1249249249249249ull;
  return q;
}

__global__ void k_keys(const double *x, const double *y,
                       const double *z, int64_t n, const double *bbox,
                       uint64_t *__restrict__ key, uint32_t *__restrict__ idx) {
  pdl_wait();
  int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
  if (i >= n) return;
  const double s = bbox[3];
  uint64_t qx = quantise(x[i], bbox[0], s), qy = quantise(y[i], bbox[1], s),
           qz = quantise(z[i], bbox[2], s);
  key[i] = spread3(qx) | (spread3(qy) << 1) | (spread3(qz) << 2);
  idx[i] = static_cast<uint32_t>(i);
}

// ---------------------------------------------------------------------------
// a13: a forest of independent systems (concatenated, system s owns caller
// indices [off[s], off[s+1])).  Every system gets its own bounding cube and
// keys; a second stable sort pass groups the bodies by system, so each
// system's bodies stay in key order and every root covers one system.
// ---------------------------------------------------------------------------
// one block per system: its cube (lo, scale), the system id of its bodies and
// the bad-data flag
__global__ void k_bbox_sys(const double *x, const double *y,
                           const double *z, const double *m,
                           const int64_t *off, double *__restrict__ sbox,
                           int32_t *__restrict__ sysid, int *__restrict__ status) {
  pdl_wait();
  const int s = blockIdx.x;
  const int64_t b = off[s], e = off[s + 1];
  const Extremes v = body_extremes(x, y, z, m, b + threadIdx.x, e, blockDim.x, status);
  for (int64_t i = b + threadIdx.x; i < e; i += blockDim.x) sysid[i] = s;
  if (threadIdx.x == 0) write_box(v, sbox + 4 * static_cast<int64_t>(s));
}

__global__ void k_keys_sys(const double *x, const double *y,
                           const double *z, int64_t n, const double *sbox,
                           const int32_t *sysid, uint64_t *__restrict__ key,
                           uint32_t *__restrict__ idx) {
  pdl_wait();
  int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
  if (i >= n) return;
  const double *b = sbox + 4 * sysid[i];
  uint64_t qx = quantise(x[i], b[0], b[3]), qy = quantise(y[i], b[1], b[3]), qz = quantise(z[i], b[2], b[3]);
  key[i] = spread3(qx) | (spread3(qy) << 1) | (spread3(qz) << 2);
  idx[i] = static_cast<uint32_t>(i);
}

// second pass: (system of the body at sorted position s, s)
__global__ void k_sys_keys(int64_t n, const uint32_t *idx, const int32_t *sysid,
                           uint32_t *__restrict__ skey, uint32_t *__restrict__ sval) {
  pdl_wait();
  int64_t s = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
  if (s >= n) return;
  skey[s] = static_cast<uint32_t>(sysid[idx[s]]);
  sval[s] = static_cast<uint32_t>(s);
}

__global__ void k_gather_sorted(int64_t n, const uint32_t *perm, const uint64_t *k1,
                                const uint32_t *i1, uint64_t *__restrict__ k2,
                                uint32_t *__restrict__ i2) {
  pdl_wait();
  int64_t t = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
  if (t >= n) return;
  k2[t] = k1[perm[t]];
  i2[t] = i1[perm[t]];
}

// Gather the bodies into key order, also as hi + lo floats (R_max, and the
// mixed form's near field).
__global__ void k_permute(const double *x, const double *y,
                          const double *z, const double *m,
                          const uint32_t *idx, int64_t n, double *__restrict__ X,
                          double *__restrict__ Y, double *__restrict__ Zb, double *__restrict__ Mb,
                          int32_t *__restrict__ order, BodyF *__restrict__ bodyf) {
  pdl_wait();
  int64_t s = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
  if (s >= n) return;
  const uint32_t o = idx[s];
  const double xs = x[o], ys = y[o], zs = z[o], ms = m[o];
  X[s] = xs;
  Y[s] = ys;
  Zb[s] = zs;
  Mb[s] = ms;
  order[s] = static_cast<int32_t>(o);
  bodyf[s] = split_body(xs, ys, zs, ms);
}

// ---------------------------------------------------------------------------
// a3: octree, all levels at once
// ---------------------------------------------------------------------------
// The sorted keys fix the tree without a pass per level.  A run of bodies that
// share l octal digits is a cell of level l if the run at level l - 1 is
// split, that is, holds more than n_crit bodies (and l <= 21).  A body's run
// holds more than n_crit bodies at level l exactly when some window of
// n_crit + 1 consecutive bodies around it shares l digits, and a window shares
// as many as its first and last key do.  So its leaf lies at level
//     D = min(21, 1 + max over its windows of the digits shared by their ends)
// (0 without a window), and the cells that start at the body are those of the
// levels (digits shared with its predecessor) + 1 .. D.  Counting the starts
// per level and block, one scan over (level, block) gives every cell its id
// in breadth-first order; a body's cell at any level up to D is the last
// start at or before it.  (One pass per level, five launches each: 0.45 of the
// 0.79 ms of the tree at N = 1,048,576, 0.26 of 0.50 ms at 65,536.)
constexpr int kLevels = kMaxLevel + 1;
// largest n_crit whose windows a block keeps in shared memory and each body
// scans; wider ones take the maximum by doubling, a launch per step
constexpr int kWindowMax = 2048;

// octal digits that two keys share
__device__ __forceinline__ int shared_digits(uint64_t a, uint64_t b) {
  const uint64_t d = a ^ b;
  return d == 0 ? kMaxLevel : (__clzll(static_cast<long long>(d)) - 1) / 3;
}
// system of the body at sorted position s
__device__ __forceinline__ int system_of(const int32_t *sysid, const uint32_t *idx,
                                         int64_t s) {
  return sysid ? sysid[idx[s]] : 0;
}
// digits shared by the ends of the window [j, j + w], -1 if there is none
__device__ __forceinline__ int window_digits(const uint64_t *key, const uint32_t *idx,
                                             const int32_t *sysid, int64_t n, int64_t j, int w) {
  if (j < 0 || j + w >= n || system_of(sysid, idx, j) != system_of(sysid, idx, j + w)) return -1;
  return shared_digits(key[j], key[j + w]);
}

// For n_crit beyond kWindowMax: the windows' digits, and their running maximum
// over the last 2^k window starts by doubling (out = max of in at j and at
// j - step).
__global__ void k_window_digits(const uint64_t *key, const uint32_t *idx,
                                const int32_t *sysid, int64_t n, int w, int8_t *__restrict__ out) {
  pdl_wait();
  const int64_t j = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
  if (j < n) out[j] = static_cast<int8_t>(window_digits(key, idx, sysid, n, j, w));
}
__global__ void k_window_max(int64_t n, int64_t step, const int8_t *in, int8_t *__restrict__ out) {
  pdl_wait();
  const int64_t j = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
  if (j < n) out[j] = j >= step ? max(in[j], in[j - step]) : in[j];
}

// Per body: the digits shared with its predecessor (-1 for the first of a
// system) and its leaf's level; per block and level: cells and leaves that
// start there.  wmax (n_crit > kWindowMax): the maximum over the body's
// windows.
__global__ void k_cell_levels(const uint64_t *key, const uint32_t *idx,
                              const int32_t *sysid, int64_t n, int n_crit,
                              const int8_t *wmax, char2 *__restrict__ lv, int32_t *__restrict__ cnt) {
  pdl_wait();
  extern __shared__ int8_t win[];  // kBlock + n_crit window starts
  __shared__ int32_t tot[2][kLevels];
  const int t = threadIdx.x, lane = t & 31;
  const int64_t i0 = blockIdx.x * static_cast<int64_t>(kBlock), i = i0 + t;
  if (t < 2 * kLevels) tot[t / kLevels][t % kLevels] = 0;
  if (!wmax)
    for (int q = t; q < kBlock + n_crit; q += kBlock)
      win[q] = static_cast<int8_t>(window_digits(key, idx, sysid, n, i0 - n_crit + q, n_crit));
  __syncthreads();
  int lcp = kMaxLevel, D = -1;
  if (i < n) {
    int m = -1;
    if (wmax) m = wmax[i];
    else
      for (int q = 0; q <= n_crit; ++q) m = max(m, static_cast<int>(win[t + q]));
    D = min(kMaxLevel, 1 + m);
    lcp = i == 0 || system_of(sysid, idx, i) != system_of(sysid, idx, i - 1) ? -1 : shared_digits(key[i - 1], key[i]);
    lv[i] = make_char2(static_cast<signed char>(lcp), static_cast<signed char>(D));
  }
#pragma unroll
  for (int l = 0; l < kLevels; ++l) {
    const unsigned c = __ballot_sync(0xffffffffu, l > lcp && l <= D);
    const unsigned f = __ballot_sync(0xffffffffu, l > lcp && l == D);
    if (lane == 0 && c) atomicAdd(&tot[0][l], __popc(c));
    if (lane == 0 && f) atomicAdd(&tot[1][l], __popc(f));
  }
  __syncthreads();
  if (t < 2 * kLevels) cnt[static_cast<int64_t>(t) * gridDim.x + blockIdx.x] = tot[t / kLevels][t % kLevels];
  if (blockIdx.x == 0 && t == 0) cnt[2 * kLevels * static_cast<int64_t>(gridDim.x)] = 0;  // closes the scan
}

// Emits the cells: begin, level, parent; every body's cell per level (-1 below
// its leaf), its leaf, and the leaves in id order.  lvl: first id of every
// level (23 entries) and the number of leaves.
__global__ void k_emit_cells(int64_t n, const char2 *lv, const int32_t *offs, int64_t cap,
                             int32_t *__restrict__ begin, int32_t *__restrict__ level, int32_t *__restrict__ parent,
                             int32_t *__restrict__ cell_at, int32_t *__restrict__ leaf_of,
                             int32_t *__restrict__ leaves, int32_t *__restrict__ lvl) {
  pdl_wait();
  __shared__ int32_t base[2][kLevels][kBlock / 32];
  __shared__ int32_t first[kLevels + 1];
  const int t = threadIdx.x, lane = t & 31, w = t >> 5;
  const int64_t nb = gridDim.x, i = blockIdx.x * static_cast<int64_t>(kBlock) + t;
  int lcp = kMaxLevel, D = -1;
  if (i < n) {
    const char2 v = lv[i];
    lcp = v.x;
    D = v.y;
  }
  if (t <= kLevels) first[t] = offs[t * nb];
#pragma unroll
  for (int l = 0; l < kLevels; ++l) {
    const unsigned c = __ballot_sync(0xffffffffu, l > lcp && l <= D);
    const unsigned f = __ballot_sync(0xffffffffu, l > lcp && l == D);
    if (lane == 0) {
      base[0][l][w] = __popc(c);
      base[1][l][w] = __popc(f);
    }
  }
  __syncthreads();
  if (t < 2 * kLevels) {
    int run = offs[static_cast<int64_t>(t) * nb + blockIdx.x];
    int32_t *b = base[t / kLevels][t % kLevels];
    for (int q = 0; q < kBlock / 32; ++q) {
      const int v = b[q];
      b[q] = run;
      run += v;
    }
  }
  __syncthreads();
  const int ncell = first[kLevels];
  if (blockIdx.x == 0 && t <= kLevels) lvl[t] = first[t];
  if (blockIdx.x == 0 && t == 0) lvl[kLevels + 1] = offs[2 * kLevels * nb] - ncell;
  const unsigned lt = (1u << lane) - 1;
  int up = -1;  // the body's cell of the level above
  for (int l = 0; l < kLevels && first[l] < ncell; ++l) {
    const bool starts = l > lcp && l <= D;
    const unsigned c = __ballot_sync(0xffffffffu, starts);
    const unsigned f = __ballot_sync(0xffffffffu, starts && l == D);
    if (i >= n) continue;
    const int id = l <= D ? base[0][l][w] + __popc(c & lt) + (starts ? 1 : 0) - 1 : -1;
    cell_at[static_cast<int64_t>(l) * n + i] = id;
    if (starts && id < cap) {
      begin[id] = static_cast<int32_t>(i);
      level[id] = l;
      parent[id] = up;
    }
    if (l == D) {
      leaf_of[i] = id;
      if (starts) leaves[base[1][l][w] + __popc(f & lt) - ncell] = id;
    }
    up = id;
  }
}

// Ends and children of the cells.  A cell ends where its next sibling begins,
// or with its parent; the children of a split cell are the cells of its first
// to its last body on the next level.
__global__ void k_finish_cells(int64_t n, int n_crit, int nsys, int64_t cap, const int64_t *sys_off,
                               const int32_t *lvl, const int32_t *begin,
                               const int32_t *level, const int32_t *parent,
                               const int32_t *cell_at, int32_t *__restrict__ count,
                               int32_t *__restrict__ first_child, int32_t *__restrict__ nchild) {
  pdl_wait();
  const int ncell = lvl[kLevels];
  if (ncell > cap) return;  // built again with more room
  for (int64_t id = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; id < ncell;
       id += static_cast<int64_t>(gridDim.x) * blockDim.x) {
    int64_t q = id, e = -1;
    while (e < 0) {
      const int p = parent[q];
      if (p < 0) e = sys_off[q + 1];  // the roots are the first cells
      else if (q + 1 < ncell && parent[q + 1] == p) e = begin[q + 1];
      else q = p;
    }
    const int b = begin[id], l = level[id], c = static_cast<int>(e) - b;
    int f = -1, k = 0;
    if (c > n_crit && l < kMaxLevel) {
      const int32_t *next = cell_at + static_cast<int64_t>(l + 1) * n;
      f = next[b];
      k = next[b + c - 1] - f + 1;
    }
    count[id] = c;
    first_child[id] = f;
    nchild[id] = k;
  }
}

// ---------------------------------------------------------------------------
// a4: centres of mass, moments, R_max
// ---------------------------------------------------------------------------
// Moments about Z in the order M, x, y, z, xx, xy, xz, yy, yz, zz, xxx, xxy,
// xxz, xyy, xyz, xzz, yyy, yyz, yzz, zzz.
//
// An FP64 instruction holds its pipe for 64 cycles per warp, however many of
// its lanes work, so what counts here is the number of FP64 warp instructions:
// their total where a level fills the GPU, their chain where it does not.
//
// Leaves: a warp takes G leaves and 32 of their bodies at a time.  The centre
// of mass is summed in body order (as its definition here demands), one lane
// per (leaf, component); then each lane forms its body's offset and the ten
// products of up to second order, and one lane per moment sums leaf by leaf in
// body order with one FMA per body (lanes over all (leaf, moment) instead run as
// long as the largest leaf of the tile: 178 against 164 us at N = 1M).  About 18 FP64 warp
// instructions per leaf at G = 8 against 27 with a thread per leaf, and a chain
// of about 75 instead of 1,100 for a leaf of 25 bodies.
// A moment as (base product of up to second order) x coordinate: base 0..9 =
// mu, mx, my, mz, mxx, mxy, mxz, myy, myz, mzz; coordinate 0..2, 3: one.
__constant__ signed char c_mom_base[kMomStride] = {0, 0, 0, 0, 1, 1, 1, 2, 2, 3, 4, 4, 4, 7, 5, 9, 7, 7, 9, 9};
__constant__ signed char c_mom_coord[kMomStride] = {3, 0, 1, 2, 0, 1, 2, 1, 2, 2, 0, 1, 2, 0, 2, 0, 1, 2, 1, 2};
constexpr int kUpWarps = 4;

template <int G>
__global__ void __launch_bounds__(kUpWarps * 32) k_leaf_upward(
    int32_t nleaf, const int32_t *leaves, const int32_t *begin,
    const int32_t *count, const double *X, const double *Y,
    const double *Zb, const double *Mb, double *__restrict__ S, double *__restrict__ M,
    double *__restrict__ Z, double *__restrict__ invM, double *__restrict__ mom) {
  pdl_wait();
  __shared__ double sh[kUpWarps][14][33];  // per body: ten products, x, y, z, 1 (first: mu x, mu y, mu z, mu)
  __shared__ double com[kUpWarps][G][4];
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  const int q0 = (blockIdx.x * kUpWarps + w) * G;
  if (q0 >= nleaf) return;  // whole warp
  const int ng = min(G, nleaf - q0);
  const int c = l < ng ? leaves[q0 + l] : 0;
  const int b = l < ng ? begin[c] : 0, cnt = l < ng ? count[c] : 0;
  int end = cnt;  // inclusive prefix: leaf g owns concatenated bodies [end - cnt, end)
#pragma unroll
  for (int o = 1; o < G; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, end, o);
    if (l >= o) end += y;
  }
  const int total = __shfl_sync(0xffffffffu, end, ng - 1);
  // body of lane l in the tile at t0, and its leaf
  const auto locate = [&](int t0, int &g) {
    const int t = t0 + l;
    g = 0;
#pragma unroll
    for (int k = 0; k < G - 1; ++k) g += t >= __shfl_sync(0xffffffffu, end, k) ? 1 : 0;
    g = min(g, ng - 1);
    const int bg = __shfl_sync(0xffffffffu, b, g), eg = __shfl_sync(0xffffffffu, end, g),
              cg = __shfl_sync(0xffffffffu, cnt, g);
    return bg + (t - (eg - cg));
  };
  // bodies of leaf g in the tile at t0: lanes [lo, hi)
  const int cg4 = l >> 2;  // leaf of this lane's centre-of-mass component
  const int ce = __shfl_sync(0xffffffffu, end, cg4 < G ? cg4 : 0), cc = __shfl_sync(0xffffffffu, cnt, cg4 < G ? cg4 : 0);
  double s = 0.0;
  for (int t0 = 0; t0 < total; t0 += 32) {
    int g;
    const int i = locate(t0, g);
    if (t0 + l < total) {
      const double mu = Mb[i];
      sh[w][0][l] = __dmul_rn(mu, X[i]);
      sh[w][1][l] = __dmul_rn(mu, Y[i]);
      sh[w][2][l] = __dmul_rn(mu, Zb[i]);
      sh[w][3][l] = mu;
    }
    __syncwarp();
    if (cg4 < ng)
      for (int k = max(ce - cc - t0, 0); k < min(ce - t0, 32); ++k) s = __dadd_rn(s, sh[w][l & 3][k]);
    __syncwarp();
  }
  const double mm = __shfl_sync(0xffffffffu, s, (l & ~3) + 3);
  const double z = __ddiv_rn((l & 3) == 3 ? 1.0 : s, mm);
  if (cg4 < ng) {
    const int cell = leaves[q0 + cg4];
    com[w][cg4][l & 3] = (l & 3) == 3 ? mm : z;
    if ((l & 3) == 3) {
      M[cell] = mm;
      invM[cell] = z;
    } else {
      S[3 * cell + (l & 3)] = s;
      Z[3 * cell + (l & 3)] = z;
    }
  }
  __syncwarp();
  const int base = l < kMomStride ? c_mom_base[l] : 0, coord = l < kMomStride ? c_mom_coord[l] : 0;
  double acc = 0.0;  // of the leaf that the tiles have reached
  for (int t0 = 0; t0 < total; t0 += 32) {
    int g;
    const int i = locate(t0, g);
    if (t0 + l < total) {
      const double mu = Mb[i], x = X[i] - com[w][g][0], y = Y[i] - com[w][g][1], zz = Zb[i] - com[w][g][2];
      const double mx = mu * x, my = mu * y, mz = mu * zz;
      sh[w][0][l] = mu;
      sh[w][1][l] = mx;
      sh[w][2][l] = my;
      sh[w][3][l] = mz;
      sh[w][4][l] = mx * x;
      sh[w][5][l] = mx * y;
      sh[w][6][l] = mx * zz;
      sh[w][7][l] = my * y;
      sh[w][8][l] = my * zz;
      sh[w][9][l] = mz * zz;
      sh[w][10][l] = x;
      sh[w][11][l] = y;
      sh[w][12][l] = zz;
      sh[w][13][l] = 1.0;
    }
    __syncwarp();
    const double *q = sh[w][base], *xc = sh[w][10 + coord];
    for (int tg = 0; tg < ng; ++tg) {
      const int te = __shfl_sync(0xffffffffu, end, tg) - t0, tb = te - __shfl_sync(0xffffffffu, cnt, tg);
      if (te <= 0 || tb >= 32) continue;
      for (int k = max(tb, 0); k < min(te, 32); ++k) acc = fma(q[k], xc[k], acc);
      if (te <= 32) {
        if (l < kMomStride)
          mom[static_cast<int64_t>(leaves[q0 + tg]) * kMomStride + l] = l == 0 ? com[w][tg][3] : acc;
        acc = 0.0;
      }
    }
    __syncwarp();
  }
}

// One level of internal cells: S, M from the children in octant order, then
// the moments shifted from each child centre to Z (M2M, exact algebra for the
// raw moments Sum mu x^a): with s = Z_child - Z,
//   Q_ij  += Q_ij' + M' s_i s_j
//   O_ijk += O_ijk' + (Q_ij' s_k + Q_ik' s_j + Q_jk' s_i) + M' s_i s_j s_k
// The child dipoles D' (zero about a centre of mass up to rounding, Sec. 2)
// are left out of the shift; the parent's dipole is the shift of the child
// monopoles, D_i = Sum M' s_i.
// Two kernels do this, by the number of cells of the level, which in a forest is that
// of all systems; every operation is spelled out, so that a system's moments have the
// same bits alone and in a forest.
__device__ __forceinline__ double shift_quad(double q, double Ms_i, double s_j) { return fma(Ms_i, s_j, q); }
__device__ __forceinline__ double shift_oct(double o, double Qij, double Qik, double Qjk, double Ms_i, double si,
                                            double sj, double sk) {
  const double t = fma(Qjk, si, fma(Qik, sj, __dmul_rn(Qij, sk)));
  return fma(__dmul_rn(Ms_i, sj), sk, __dadd_rn(o, t));
}

// A warp takes four parents, eight lanes each, one per child: a lane shifts its
// child's moments, and one lane per (parent, moment) adds the shifted ones in
// octant order.  About 120 FP64 warp instructions for four parents; a thread per
// parent had a chain of 600 (52 us per level of 4,000 to 16,000 cells).
__global__ void __launch_bounds__(kUpWarps * 32) k_internal_upward(
    int32_t c0, int32_t c1, const int32_t *first_child, const int32_t *nchild,
    double *__restrict__ S, double *__restrict__ M, double *__restrict__ Z, double *__restrict__ invM,
    double *__restrict__ mom) {
  pdl_wait();
  constexpr int CELLS = 4, kRounds = (CELLS * kMomStride + 31) / 32;
  __shared__ double sh[kUpWarps][kMomStride][33];
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  const int64_t first = c0 + static_cast<int64_t>(blockIdx.x * kUpWarps + w) * CELLS;
  if (first >= c1) return;  // whole warp
  const int g = l >> 3, k = l & 7;
  const int64_t cc = first + g;
  const int c = static_cast<int>(cc);
  const int nch = g < CELLS && cc < c1 ? nchild[c] : 0;
  const int f = nch > 0 ? first_child[c] : 0;
  const bool child = k < nch;
  double zk[3] = {0.0, 0.0, 0.0}, q[kMomStride];
#pragma unroll
  for (int t = 0; t < kMomStride; ++t) q[t] = 0.0;
  if (child) {
    const double *qk = mom + static_cast<int64_t>(f + k) * kMomStride;
#pragma unroll
    for (int t = 0; t < kMomStride; ++t) q[t] = qk[t];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      zk[d] = Z[3 * (f + k) + d];
      sh[w][d][l] = S[3 * (f + k) + d];
    }
    sh[w][3][l] = M[f + k];
  }
  __syncwarp();
  // lane d of a group sums component d (lane 3: the mass)
  double s = 0.0;
  if (k < 4)
    for (int j = 0; j < nch; ++j) s = __dadd_rn(s, sh[w][k][8 * g + j]);
  const double mm = __shfl_sync(0xffffffffu, s, 8 * g + 3);
  const double z = __ddiv_rn(k == 3 ? 1.0 : s, mm);
  if (nch > 0 && k < 4) {
    if (k == 3) {
      M[c] = mm;
      invM[c] = z;
    } else {
      S[3 * c + k] = s;
      Z[3 * c + k] = z;
    }
  }
  double sv[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) sv[d] = zk[d] - __shfl_sync(0xffffffffu, z, 8 * g + d);
  __syncwarp();
  if (child) {
    const double Ms[3] = {__dmul_rn(q[0], sv[0]), __dmul_rn(q[0], sv[1]), __dmul_rn(q[0], sv[2])};
    const double Q[3][3] = {{q[4], q[5], q[6]}, {q[5], q[7], q[8]}, {q[6], q[8], q[9]}};
#pragma unroll
    for (int d = 0; d < 3; ++d) sh[w][1 + d][l] = Ms[d];
    const int qi[6] = {0, 0, 0, 1, 1, 2}, qj[6] = {0, 1, 2, 1, 2, 2};
#pragma unroll
    for (int t = 0; t < 6; ++t) sh[w][4 + t][l] = shift_quad(q[4 + t], Ms[qi[t]], sv[qj[t]]);
    const int oi[10] = {0, 0, 0, 0, 0, 0, 1, 1, 1, 2};
    const int oj[10] = {0, 0, 0, 1, 1, 2, 1, 1, 2, 2};
    const int ok[10] = {0, 1, 2, 1, 2, 2, 1, 2, 2, 2};
#pragma unroll
    for (int t = 0; t < 10; ++t) {
      const int a = oi[t], b = oj[t], e = ok[t];
      sh[w][10 + t][l] = shift_oct(q[10 + t], Q[a][b], Q[a][e], Q[b][e], Ms[a], sv[a], sv[b], sv[e]);
    }
  }
  __syncwarp();
#pragma unroll
  for (int r = 0; r < kRounds; ++r) {
    const int task = l + 32 * r, tg = task / kMomStride, t = task - tg * kMomStride;
    const int n = __shfl_sync(0xffffffffu, nch, tg < CELLS ? 8 * tg : 0);
    const double total = __shfl_sync(0xffffffffu, mm, tg < CELLS ? 8 * tg : 0);
    if (tg < CELLS && n > 0) {
      double a = 0.0;
      if (t > 0)
        for (int j = 0; j < n; ++j) a += sh[w][t][8 * tg + j];
      mom[(first + tg) * kMomStride + t] = t == 0 ? total : a;
    }
  }
}

// The same with a block per parent, for levels that leave the GPU idle: a thread
// per (child, moment), and every warp, on its own partition, takes the centre of
// mass for itself, so that the chain is one division and about 25 more FP64
// instructions instead of 120: upward pass 66 -> 47 us at N = 2,000, 114 -> 89 at
// 65,536, 233 -> 197 for a disc of 262,144 with 15 levels.
__constant__ signed char c_oct[10][3] = {{0, 0, 0}, {0, 0, 1}, {0, 0, 2}, {0, 1, 1}, {0, 1, 2},
                                         {0, 2, 2}, {1, 1, 1}, {1, 1, 2}, {1, 2, 2}, {2, 2, 2}};
__constant__ signed char c_quad[3][3] = {{4, 5, 6}, {5, 7, 8}, {6, 8, 9}};

__global__ void __launch_bounds__(128) k_internal_upward_block(
    int32_t c0, const int32_t *first_child, const int32_t *nchild, double *__restrict__ S,
    double *__restrict__ M, double *__restrict__ Z, double *__restrict__ invM, double *__restrict__ mom) {
  pdl_wait();
  __shared__ double q[8 * kMomStride], sh[kMomStride][9], sv[8][3];
  const int t = threadIdx.x, l = t & 31;
  const int c = c0 + blockIdx.x;
  const int nch = nchild[c];
  if (nch == 0) return;  // whole block
  const int f = first_child[c];
  for (int e = t; e < nch * kMomStride; e += 128) q[e] = mom[static_cast<int64_t>(f) * kMomStride + e];
  // lane 4 k + d: component d of child k (d = 3: the mass)
  const int ck = l >> 2, d = l & 3;
  const bool child = ck < nch;
  const double v = child ? (d < 3 ? S[3 * (f + ck) + d] : M[f + ck]) : 0.0;
  const double zk = child && d < 3 ? Z[3 * (f + ck) + d] : 0.0;
  double s = 0.0;
  for (int k = 0; k < nch; ++k) s = __dadd_rn(s, __shfl_sync(0xffffffffu, v, 4 * k + d));
  const double mm = __shfl_sync(0xffffffffu, s, 3);
  const double z = __ddiv_rn(d == 3 ? 1.0 : s, mm);
  if (t < 32 && child && d < 3) sv[ck][d] = zk - z;
  if (t < 3) {
    S[3 * c + t] = s;
    Z[3 * c + t] = z;
  } else if (t == 3) {
    M[c] = mm;
    invM[c] = z;
  }
  __syncthreads();
  if (t < 80) {
    const int k = t / 10, r = t - 10 * k;
    if (k < nch) {
      const double *m = q + kMomStride * k;
      const int a = c_oct[r][0], b = c_oct[r][1], e = c_oct[r][2];
      const double sa = sv[k][a], sb = sv[k][b], se = sv[k][e];
      sh[10 + r][k] = shift_oct(m[10 + r], m[c_quad[a][b]], m[c_quad[a][e]], m[c_quad[b][e]], __dmul_rn(m[0], sa),
                                sa, sb, se);
    }
  } else {
    const int k = (t - 80) / 6, r = t - 80 - 6 * k;
    if (k < nch) {
      const double *m = q + kMomStride * k;
      const int a = r < 3 ? 0 : r < 5 ? 1 : 2, b = r < 3 ? r : r < 5 ? r - 2 : 2;
      sh[4 + r][k] = shift_quad(m[4 + r], __dmul_rn(m[0], sv[k][a]), sv[k][b]);
      if (r < 3) sh[1 + r][k] = __dmul_rn(m[0], sv[k][r]);
    }
  }
  __syncthreads();
  if (t < kMomStride) {
    double a = 0.0;
    if (t > 0)
      for (int k = 0; k < nch; ++k) a += sh[t][k];
    mom[static_cast<int64_t>(c) * kMomStride + t] = t == 0 ? mm : a;
  }
}

// Centres as hi + lo floats for the filter of R_max, whose maxima start at zero.
__global__ void k_split_centres(int32_t ncell, const double *Z, float4 *__restrict__ zf,
                                unsigned long long *__restrict__ rmax2) {
  pdl_wait();
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= ncell) return;
  rmax2[c] = 0;
  const double x = Z[3 * c], y = Z[3 * c + 1], z = Z[3 * c + 2];
  const float hx = static_cast<float>(x), hy = static_cast<float>(y), hz = static_cast<float>(z);
  zf[2 * c] = make_float4(hx, hy, hz, 0.f);
  zf[2 * c + 1] =
      make_float4(static_cast<float>(x - hx), static_cast<float>(y - hy), static_cast<float>(z - hz), 0.f);
}

// R_max^2 of every cell, the exact maximum of the FP64 |X - Z|^2 over its
// bodies.  At every level a warp's bodies form runs of one cell.  Distances are
// first taken in FP32, from hi + lo floats: only a body whose FP32 value is
// within its error bound of its run's largest can hold the maximum (the bounds
// are those of separated_fast: each value is within 1e-6 of the exact one plus
// 3e-21 of the squared coordinates; outside the comfortable range every body
// stays).  Those, about one per run, are collected over the levels and
// evaluated in FP64 32 at a time, so the FP64 pipe sees about one round of
// eight instructions per warp instead of one per level (180 -> 60 us at N =
// 1,048,576).  The maximum is taken on the bit pattern (monotone for
// non-negative doubles); it is exact, so its order does not matter.
__global__ void __launch_bounds__(kBlock) k_rmax_bodies(
    int64_t n, int nlev, const int32_t *cell_at, const BodyF *bodyf,
    const float4 *zf, const double *X, const double *Y,
    const double *Zb, const double *Z, unsigned long long *__restrict__ rmax2) {
  pdl_wait();
  __shared__ int2 todo[kBlock / 32][64];  // (body, cell) still to be evaluated
  const int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  constexpr unsigned kAll = 0xffffffffu;
  BodyF b{};
  if (i < n) b = bodyf[i];
  const float am = fmaxf(fmaxf(fabsf(b.h.x), fabsf(b.h.y)), fabsf(b.h.z));
  int have = 0;
  const auto evaluate = [&](int first, int num) {
    if (lane < num) {
      const int2 e = todo[w][first + lane];
      const double dx = __dsub_rn(X[e.x], Z[3 * e.y]);
      const double dy = __dsub_rn(Y[e.x], Z[3 * e.y + 1]);
      const double dz = __dsub_rn(Zb[e.x], Z[3 * e.y + 2]);
      const unsigned long long d2 = static_cast<unsigned long long>(
          __double_as_longlong(__dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz))));
      if (d2 > rmax2[e.y]) atomicMax(&rmax2[e.y], d2);
    }
  };
  for (int lev = 0; lev < nlev; ++lev) {
    const int c = i < n ? cell_at[static_cast<int64_t>(lev) * n + i] : -1;
    if (!__any_sync(kAll, c >= 0)) break;  // no body of the warp reaches this level
    float d2 = -1.f, m = 0.f;
    if (c >= 0) {
      const float4 h = zf[2 * c], o = zf[2 * c + 1];
      const float dx = (b.h.x - h.x) + (b.l.x - o.x), dy = (b.h.y - h.y) + (b.l.y - o.y),
                  dz = (b.h.z - h.z) + (b.l.z - o.z);
      d2 = dx * dx + dy * dy + dz * dz;
      m = fmaxf(am, fmaxf(fmaxf(fabsf(h.x), fabsf(h.y)), fabsf(h.z)));
    }
    // largest value and bound of the run, at its first lane, then to all
    const int cprev = __shfl_up_sync(kAll, c, 1);
    const unsigned heads = __ballot_sync(kAll, lane == 0 || cprev != c);
    float best = d2, bound = m;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const float v = __shfl_down_sync(kAll, best, o), u = __shfl_down_sync(kAll, bound, o);
      const int co = __shfl_down_sync(kAll, c, o);
      if (lane + o < 32 && co == c) {
        best = fmaxf(best, v);
        bound = fmaxf(bound, u);
      }
    }
    const int head = 31 - __clz(static_cast<int>(heads & (kAll >> (31 - lane))));
    best = __shfl_sync(kAll, best, head);
    bound = __shfl_sync(kAll, bound, head);
    const bool exactly = !(best > 1e-30f && best < 1e30f);
    const bool cand = c >= 0 && (exactly || !(d2 + 1e-5f * best + 6e-21f * bound * bound < best));  // NaN: stays
    const unsigned mask = __ballot_sync(kAll, cand);
    if (cand) todo[w][have + __popc(mask & ((1u << lane) - 1))] = make_int2(static_cast<int>(i), c);
    have += __popc(mask);
    __syncwarp();
    if (have >= 32) {
      have -= 32;
      evaluate(have, 32);  // the last ones
      __syncwarp();
    }
  }
  evaluate(0, have);
}

__global__ void k_rmax_final(int32_t ncell, const unsigned long long *rmax2,
                             double *__restrict__ Rmax) {
  pdl_wait();
  int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c < ncell) Rmax[c] = __dsqrt_rn(__longlong_as_double(static_cast<long long>(rmax2[c])));
}

int ensure_cells(fmm_ctx *c, int64_t need) {
  DBuf *ib[] = {&c->begin, &c->count, &c->level, &c->parent, &c->first_child, &c->nchild};
  for (DBuf *b : ib) AMFMM_TRY(ensure<int32_t>(c, *b, need));
  return FMM_OK;
}

// device words of the tree stage: [0] bad input, [1] blocks done, [8, 32) the levels' first
// cell ids, the number of cells and of leaves
constexpr int kStatusLvl = 8;
constexpr int kStatusWords = kStatusLvl + kLevels + 2;

}  // namespace

int build_tree(fmm_ctx *c) {
  const int64_t n = c->sz.n;
  cudaStream_t st = c->stream;
  // body buffers
  AMFMM_TRY(ensure<uint64_t>(c, c->key[0], n));
  AMFMM_TRY(ensure<uint32_t>(c, c->idx[0], n));
  AMFMM_TRY(ensure<double>(c, c->X, n));
  AMFMM_TRY(ensure<double>(c, c->Y, n));
  AMFMM_TRY(ensure<double>(c, c->Zb, n));
  AMFMM_TRY(ensure<double>(c, c->Mb, n));
  AMFMM_TRY(ensure<int32_t>(c, c->order, n));
  AMFMM_TRY(ensure<BodyF>(c, c->bodyf, n));
  AMFMM_TRY(ensure<int32_t>(c, c->leaves, n + 1));
  AMFMM_TRY(ensure<int32_t>(c, c->leaf_of, n));
  AMFMM_TRY(ensure<int32_t>(c, c->cell_at, static_cast<size_t>(kMaxLevel + 1) * n));
  AMFMM_TRY(ensure<int>(c, c->status, kStatusWords));
  const int nbb = std::max(1, std::min<int>(c->num_sms * 4, static_cast<int>((n + kBlock - 1) / kBlock)));
  AMFMM_TRY(ensure<long long>(c, c->bbox_part, 6 * nbb));
  AMFMM_TRY(ensure<double>(c, c->bbox, 8));

  int *status = ptr<int>(c->status);
  AMFMM_CUDA(c, cudaMemsetAsync(status, 0, sizeof(int) * kStatusWords, st));
  const int nsys = c->sz.nsys;
  int which = 0;
  if (nsys == 1) {
    launch(c, k_bbox, nbb, kBlock, 0, c->x, c->y, c->z, c->m, n, ptr<long long>(c->bbox_part), status,
           reinterpret_cast<unsigned *>(status + 1), ptr<double>(c->bbox));
    AMFMM_TRY(launched(c, "bbox"));
    launch(c, k_keys, grid_for(n, kBlock), kBlock, 0, c->x, c->y, c->z, n, ptr<double>(c->bbox),
           ptr<uint64_t>(c->key[0]), ptr<uint32_t>(c->idx[0]));
    AMFMM_TRY(launched(c, "keys"));
    AMFMM_TRY(radix_sort_u64(c, c->key, c->idx, n, 63, &which));
  } else {
    AMFMM_TRY(ensure<double>(c, c->sbox, 4 * static_cast<size_t>(nsys)));
    AMFMM_TRY(ensure<int32_t>(c, c->sysid, n));
    launch(c, k_bbox_sys, nsys, kBlock, 0, c->x, c->y, c->z, c->m, ptr<int64_t>(c->sys_off), ptr<double>(c->sbox),
           ptr<int32_t>(c->sysid), status);
    AMFMM_TRY(launched(c, "bbox_sys"));
    launch(c, k_keys_sys, grid_for(n, kBlock), kBlock, 0, c->x, c->y, c->z, n, ptr<double>(c->sbox),
           ptr<int32_t>(c->sysid), ptr<uint64_t>(c->key[0]), ptr<uint32_t>(c->idx[0]));
    AMFMM_TRY(launched(c, "keys_sys"));
    int w1 = 0;
    AMFMM_TRY(radix_sort_u64(c, c->key, c->idx, n, 63, &w1));
    AMFMM_TRY(ensure<uint32_t>(c, c->ekey[0], n));
    AMFMM_TRY(ensure<uint32_t>(c, c->eval[0], n));
    launch(c, k_sys_keys, grid_for(n, kBlock), kBlock, 0, n, ptr<uint32_t>(c->idx[w1]), ptr<int32_t>(c->sysid),
           ptr<uint32_t>(c->ekey[0]), ptr<uint32_t>(c->eval[0]));
    AMFMM_TRY(launched(c, "sys_keys"));
    int w2 = 0, sbits = 1;
    while ((int64_t(1) << sbits) <= nsys) ++sbits;
    AMFMM_TRY(radix_sort_u32(c, c->ekey, c->eval, n, sbits, &w2));
    launch(c, k_gather_sorted, grid_for(n, kBlock), kBlock, 0, n, ptr<uint32_t>(c->eval[w2]),
           ptr<uint64_t>(c->key[w1]), ptr<uint32_t>(c->idx[w1]), ptr<uint64_t>(c->key[w1 ^ 1]),
           ptr<uint32_t>(c->idx[w1 ^ 1]));
    AMFMM_TRY(launched(c, "gather_sorted"));
    which = w1 ^ 1;
  }
  const uint64_t *skey = ptr<uint64_t>(c->key[which]);
  const uint32_t *sidx = ptr<uint32_t>(c->idx[which]);
  c->sz.key_which = which;
  launch(c, k_permute, grid_for(n, kBlock), kBlock, 0, c->x, c->y, c->z, c->m, sidx, n, ptr<double>(c->X),
         ptr<double>(c->Y), ptr<double>(c->Zb), ptr<double>(c->Mb), ptr<int32_t>(c->order), ptr<BodyF>(c->bodyf));
  AMFMM_TRY(launched(c, "permute"));

  // octree: levels of every body, ids by one scan, cells
  const int n_crit = static_cast<int>(std::min<int64_t>(c->opts.n_crit, n));
  const int32_t *sysid = nsys == 1 ? nullptr : ptr<int32_t>(c->sysid);
  const unsigned nb = grid_for(n, kBlock);
  const int64_t ncnt = 2 * kLevels * static_cast<int64_t>(nb) + 1;
  AMFMM_TRY(ensure<char2>(c, c->body_lv, n));
  AMFMM_TRY(ensure<int32_t>(c, c->flag, std::max(n, ncnt) + 1));
  AMFMM_TRY(ensure<int32_t>(c, c->incl, std::max(n, ncnt) + 1));
  int32_t *cnt = ptr<int32_t>(c->flag), *offs = ptr<int32_t>(c->incl);
  const int8_t *wmax = nullptr;
  if (n_crit > kWindowMax) {
    // windows wider than a block: maximum over the last n_crit + 1 starts by
    // doubling, then once more over the two halves that cover them
    AMFMM_TRY(ensure<int8_t>(c, c->lcp, 2 * n));
    int8_t *a = ptr<int8_t>(c->lcp), *o = a + n;
    launch(c, k_window_digits, nb, kBlock, 0, skey, sidx, sysid, n, n_crit, a);
    AMFMM_TRY(launched(c, "window_digits"));
    int64_t have = 1;
    while (have < n_crit + 1) {
      const int64_t step = std::min<int64_t>(have, n_crit + 1 - have);
      launch(c, k_window_max, nb, kBlock, 0, n, step, a, o);
      AMFMM_TRY(launched(c, "window_max"));
      std::swap(a, o);
      have += step;
    }
    wmax = a;
  }
  launch(c, k_cell_levels, nb, kBlock, wmax ? 0 : kBlock + n_crit, skey, sidx, sysid, n, n_crit, wmax,
         ptr<char2>(c->body_lv), cnt);
  AMFMM_TRY(launched(c, "cell_levels"));
  AMFMM_TRY(exclusive_scan_i32(c, cnt, offs, ncnt, nullptr));
  int32_t *lvl = reinterpret_cast<int32_t *>(status + kStatusLvl);
  int64_t cap_cells = std::max<int64_t>(std::max<int64_t>(1024, n / 2 + 64), 2 * static_cast<int64_t>(nsys));
  int32_t *h = static_cast<int32_t *>(c->hpin);
  double *hb = reinterpret_cast<double *>(h + kStatusWords);
  const double *bbox = nsys == 1 ? ptr<double>(c->bbox) : ptr<double>(c->sbox);
  for (int attempt = 0;; ++attempt) {
    AMFMM_TRY(ensure_cells(c, cap_cells));
    const int64_t cap = static_cast<int64_t>(std::min({c->begin.cap, c->count.cap, c->level.cap, c->parent.cap,
                                                       c->first_child.cap, c->nchild.cap}) /
                                             sizeof(int32_t));
    launch(c, k_emit_cells, nb, kBlock, 0, n, ptr<char2>(c->body_lv), offs, cap, ptr<int32_t>(c->begin),
           ptr<int32_t>(c->level), ptr<int32_t>(c->parent), ptr<int32_t>(c->cell_at), ptr<int32_t>(c->leaf_of),
           ptr<int32_t>(c->leaves), lvl);
    AMFMM_TRY(launched(c, "emit_cells"));
    launch(c, k_finish_cells,
           static_cast<unsigned>(std::min<int64_t>(grid_for(std::min(cap, n), kBlock), 8 * c->num_sms)), kBlock, 0, n,
           n_crit, nsys, cap, ptr<int64_t>(c->sys_off), lvl, ptr<int32_t>(c->begin), ptr<int32_t>(c->level),
           ptr<int32_t>(c->parent), ptr<int32_t>(c->cell_at), ptr<int32_t>(c->count), ptr<int32_t>(c->first_child),
           ptr<int32_t>(c->nchild));
    AMFMM_TRY(launched(c, "finish_cells"));
    const HostRead rb[2] = {{h, status, sizeof(int) * kStatusWords}, {hb, bbox, 4 * sizeof(double)}};
    AMFMM_TRY(read_back(c, rb, 2));
    if (h[kStatusLvl + kLevels] <= cap) break;
    // a tree of single-child chains can have more cells than bodies
    if (capturing(c) || attempt > 0) return set_error(c, FMM_EINVAL, "octree: cell room still short after growing");
    cap_cells = h[kStatusLvl + kLevels];
  }
  if (capturing(c)) {
    AMFMM_TRY(graph_record_bbox(c, bbox));
    Expect e;
    for (int k = 0; k < kStatusWords; ++k) e.add(status + k, static_cast<uint32_t>(h[k]));
    AMFMM_TRY(graph_expect(c, e));
  }
  const int32_t *hl = h + kStatusLvl;
  const int64_t nc = hl[kLevels];
  int depth = 0;
  while (depth + 1 < kLevels && hl[depth + 1] < nc) ++depth;
  c->sz.depth = depth;
  c->sz.ncell = nc;
  c->sz.lvl_off.assign(hl, hl + depth + 2);
  c->sz.nleaf = hl[kLevels + 1];
  for (int d = 0; d < 3; ++d) c->sz.lo[d] = hb[d];
  c->sz.scale = hb[3];
  if (h[0] != 0)
    return set_error(c, FMM_EINVAL, "a body has a non-finite coordinate or a mass that is not positive and finite");
  AMFMM_TRY(ensure<int32_t>(c, c->flag, std::max(n, nc) + 1));
  AMFMM_TRY(ensure<int32_t>(c, c->incl, std::max(n, nc) + 1));
  return FMM_OK;
}

int upward(fmm_ctx *c) {
  const int64_t n = c->sz.n, nc = c->sz.ncell;
  AMFMM_TRY(ensure<double>(c, c->S, 3 * nc));
  AMFMM_TRY(ensure<double>(c, c->M, nc));
  AMFMM_TRY(ensure<double>(c, c->Z, 3 * nc));
  AMFMM_TRY(ensure<double>(c, c->invM, nc));
  AMFMM_TRY(ensure<double>(c, c->Rmax, nc));
  AMFMM_TRY(ensure<unsigned long long>(c, c->rmax2, nc));
  AMFMM_TRY(ensure<double>(c, c->mom, static_cast<size_t>(mom_stride(c->opts.order_P)) * nc));
  if (c->opts.order_P != 3) {
    AMFMM_TRY(upward_general(c));
  } else {
  // leaves per warp: as many as leave two warps per partition of the GPU
  // (fewer FP64 instructions per leaf), down to one (a short chain)
  const int64_t nleaf = c->sz.nleaf;
  const int64_t fill = 8 * static_cast<int64_t>(std::max(1, c->num_sms));
  const auto leaf = nleaf >= 8 * fill ? k_leaf_upward<8> : nleaf >= 4 * fill ? k_leaf_upward<4>
                  : nleaf >= 2 * fill ? k_leaf_upward<2> : k_leaf_upward<1>;
  const int per = nleaf >= 8 * fill ? 8 : nleaf >= 4 * fill ? 4 : nleaf >= 2 * fill ? 2 : 1;
  launch(c, leaf, grid_for(nleaf, kUpWarps * per), kUpWarps * 32, 0, static_cast<int32_t>(nleaf),
         ptr<int32_t>(c->leaves), ptr<int32_t>(c->begin), ptr<int32_t>(c->count), ptr<double>(c->X), ptr<double>(c->Y),
         ptr<double>(c->Zb), ptr<double>(c->Mb), ptr<double>(c->S), ptr<double>(c->M), ptr<double>(c->Z),
         ptr<double>(c->invM), ptr<double>(c->mom));
  AMFMM_TRY(launched(c, "leaf_upward"));
  for (int lev = c->sz.depth - 1; lev >= 0; --lev) {
    const int64_t c0 = c->sz.lvl_off[lev], c1 = c->sz.lvl_off[lev + 1];
    // four parents per warp once that gives every partition of the GPU two warps
    // (lines at twice to eight times as many parents measured the same within 1%)
    if (c1 - c0 >= fill)
      launch(c, k_internal_upward, grid_for(c1 - c0, 4 * kUpWarps), kUpWarps * 32, 0, static_cast<int32_t>(c0),
             static_cast<int32_t>(c1), ptr<int32_t>(c->first_child), ptr<int32_t>(c->nchild), ptr<double>(c->S),
             ptr<double>(c->M), ptr<double>(c->Z), ptr<double>(c->invM), ptr<double>(c->mom));
    else
      launch(c, k_internal_upward_block, static_cast<unsigned>(c1 - c0), 128, 0, static_cast<int32_t>(c0),
             ptr<int32_t>(c->first_child), ptr<int32_t>(c->nchild), ptr<double>(c->S), ptr<double>(c->M),
             ptr<double>(c->Z), ptr<double>(c->invM), ptr<double>(c->mom));
    AMFMM_TRY(launched(c, "internal_upward"));
  }
  }
  AMFMM_TRY(ensure<float4>(c, c->cellzf, 2 * nc));
  launch(c, k_split_centres, grid_for(nc, kBlock), kBlock, 0, static_cast<int32_t>(nc), ptr<double>(c->Z),
         ptr<float4>(c->cellzf), ptr<unsigned long long>(c->rmax2));
  AMFMM_TRY(launched(c, "split_centres"));
  launch(c, k_rmax_bodies, grid_for(n, kBlock), kBlock, 0, n, c->sz.depth + 1, ptr<int32_t>(c->cell_at),
         ptr<BodyF>(c->bodyf), ptr<float4>(c->cellzf), ptr<double>(c->X), ptr<double>(c->Y), ptr<double>(c->Zb),
         ptr<double>(c->Z), ptr<unsigned long long>(c->rmax2));
  AMFMM_TRY(launched(c, "rmax_bodies"));
  launch(c, k_rmax_final, grid_for(nc, kBlock), kBlock, 0, static_cast<int32_t>(nc), ptr<unsigned long long>(c->rmax2),
         ptr<double>(c->Rmax));
  return launched(c, "rmax_final");
}

}  // namespace amfmm
