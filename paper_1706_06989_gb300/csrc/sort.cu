// sort.cu -- device primitives: exclusive prefix sums and a stable LSD radix
// sort of (key, value) pairs.  Both are deterministic: integer arithmetic
// only, and a fixed assignment of keys to ranks.
#include <algorithm>

#include "internal.cuh"

namespace amfmm {
namespace {

constexpr int kScanBlock = 256;
constexpr int kScanItems = 8;
constexpr int kScanTile = kScanBlock * kScanItems;
constexpr int kRedundantTiles = 4096;  // up to 8M elements: two launches per scan

// ---- element operations for the scans ----
__device__ __forceinline__ int32_t vadd(int32_t a, int32_t b) { return a + b; }
__device__ __forceinline__ int64_t vadd(int64_t a, int64_t b) { return a + b; }
template <class T> __device__ __forceinline__ T vzero();
template <> __device__ __forceinline__ int32_t vzero<int32_t>() { return 0; }
template <> __device__ __forceinline__ int64_t vzero<int64_t>() { return 0; }

__device__ __forceinline__ int32_t shfl_up(int32_t v, int d) { return __shfl_up_sync(0xffffffffu, v, d); }
__device__ __forceinline__ int64_t shfl_up(int64_t v, int d) {
  return static_cast<int64_t>(__shfl_up_sync(0xffffffffu, static_cast<long long>(v), d));
}
// Inclusive scan across the warp.
template <class T>
__device__ __forceinline__ T warp_inclusive(T v) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    T t = shfl_up(v, d);
    if (lane >= d) v = vadd(v, t);
  }
  return v;
}

// Exclusive scan of one value per thread over the block; returns the block total.
template <class T>
__device__ __forceinline__ T block_exclusive(T v, T *excl) {
  __shared__ T wtot[kScanBlock / 32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  T inc = warp_inclusive(v);
  if (lane == 31) wtot[w] = inc;
  __syncthreads();
  if (w == 0) {
    T s = lane < kScanBlock / 32 ? wtot[lane] : vzero<T>();
    s = warp_inclusive(s);
    if (lane < kScanBlock / 32) wtot[lane] = s;
  }
  __syncthreads();
  T before = w > 0 ? wtot[w - 1] : vzero<T>();
  T prev = shfl_up(inc, 1);
  if (lane == 0) prev = vzero<T>();
  *excl = vadd(before, prev);
  T total = wtot[kScanBlock / 32 - 1];
  __syncthreads();
  return total;
}

template <class T>
__global__ void k_tile_reduce(const T *in, int64_t n, T *__restrict__ sums) {
  pdl_wait();
  const int64_t base = static_cast<int64_t>(blockIdx.x) * kScanTile;
  T s = vzero<T>();
#pragma unroll
  for (int k = 0; k < kScanItems; ++k) {
    int64_t i = base + static_cast<int64_t>(k) * kScanBlock + threadIdx.x;
    if (i < n) s = vadd(s, in[i]);
  }
  T excl;
  T tot = block_exclusive(s, &excl);
  if (threadIdx.x == 0) sums[blockIdx.x] = tot;
}

// Exclusive scan of one tile; the tile's offset is offs[tile] when offs is
// given, else the sum of the tile sums sums[0, tile) taken by this block
// (integer addition: exact in any order), else zero.  The last tile writes
// the grand total.
template <class T>
__global__ void k_tile_scan(const T *in, T *__restrict__ out, int64_t n,
                            const T *offs, T *__restrict__ total,
                            const T *sums) {
  pdl_wait();
  const int64_t base = static_cast<int64_t>(blockIdx.x) * kScanTile;
  T pre = vzero<T>();
  if (!offs && sums) {
    for (int q = threadIdx.x; q < static_cast<int>(blockIdx.x); q += kScanBlock) pre = vadd(pre, sums[q]);
    T ignore;
    pre = block_exclusive(pre, &ignore);  // the block total of the partial sums
  }
  // each thread owns kScanItems consecutive elements
  T v[kScanItems];
  const int64_t mybase = base + static_cast<int64_t>(threadIdx.x) * kScanItems;
  T s = vzero<T>();
#pragma unroll
  for (int k = 0; k < kScanItems; ++k) {
    int64_t i = mybase + k;
    v[k] = i < n ? in[i] : vzero<T>();
    s = vadd(s, v[k]);
  }
  T excl;
  T tot = block_exclusive(s, &excl);
  T off = offs ? offs[blockIdx.x] : pre;
  T run = vadd(off, excl);
#pragma unroll
  for (int k = 0; k < kScanItems; ++k) {
    int64_t i = mybase + k;
    if (i < n) out[i] = run;
    run = vadd(run, v[k]);
  }
  if (total && blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) *total = vadd(off, tot);
}

template <class T>
int scan_impl(fmm_ctx *c, const T *in, T *out, int64_t n, T *total, size_t tmp_off) {
  if (n <= 0) {
    if (total) AMFMM_CUDA(c, cudaMemsetAsync(total, 0, sizeof(T), c->stream));
    return FMM_OK;
  }
  const int64_t nt = (n + kScanTile - 1) / kScanTile;
  if (nt == 1) {
    launch(c, k_tile_scan<T>, 1, kScanBlock, 0, in, out, n, nullptr, total, nullptr);
    return launched(c, "tile_scan");
  }
  // scratch: sums[nt], offs[nt], then the recursion's scratch
  size_t need = tmp_off + 2 * static_cast<size_t>(nt) * sizeof(T) + 256;
  if (need > c->scan_tmp.cap) {
    return set_error(c, FMM_ENOMEM, "scan scratch too small (%zu > %zu)", need, c->scan_tmp.cap);
  }
  char *base = static_cast<char *>(c->scan_tmp.p) + tmp_off;
  T *sums = reinterpret_cast<T *>(base);
  T *offs = sums + nt;
  size_t next = tmp_off + ((2 * static_cast<size_t>(nt) * sizeof(T) + 255) / 256) * 256;
  launch(c, k_tile_reduce<T>, static_cast<unsigned>(nt), kScanBlock, 0, in, n, sums);
  AMFMM_TRY(launched(c, "tile_reduce"));
  if (nt <= kRedundantTiles) {
    // few tiles: every block adds up the sums of the tiles before it (at
    // most kRedundantTiles reads, from L2) instead of a separate scan of them
    launch(c, k_tile_scan<T>, static_cast<unsigned>(nt), kScanBlock, 0, in, out, n, nullptr, total, sums);
    return launched(c, "tile_scan");
  }
  AMFMM_TRY(scan_impl<T>(c, sums, offs, nt, nullptr, next));
  launch(c, k_tile_scan<T>, static_cast<unsigned>(nt), kScanBlock, 0, in, out, n, offs, total, nullptr);
  return launched(c, "tile_scan");
}

template <class T>
int scan_entry(fmm_ctx *c, const T *in, T *out, int64_t n, T *total) {
  // scratch bound: 2 * sizeof(T) * (n/tile + n/tile^2 + ...) + alignment
  size_t need = 0;
  for (int64_t m = (n + kScanTile - 1) / kScanTile; m > 1; m = (m + kScanTile - 1) / kScanTile)
    need += ((2 * static_cast<size_t>(m) * sizeof(T) + 255) / 256) * 256 + 256;
  AMFMM_TRY(ensure_bytes(c, c->scan_tmp, need + 1024));
  return scan_impl<T>(c, in, out, n, total, 0);
}

// ---- radix sort ----
__device__ __forceinline__ unsigned lanemask_lt() {
  unsigned m;
  asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
  return m;
}

// A pass is one launch that ranks tiles of keys and writes them out.  Where a
// tile's keys go depends on the digits of the tiles before it: those of its own
// group of kGroup tiles it adds up itself, reading their counts as they appear
// (look-back over at most kGroup - 1 rows, all in flight at once); for the
// groups before there are two forms.
// - few keys (no more tiles than run at once): the digits of all passes are
//   counted in one launch (they do not depend on the order of the keys), and a
//   tile also adds up the groups' counts, which the tiles before it accumulate;
// - many: one launch per pass counts the digits of every group of tiles, one
//   turns the counts into first positions.
// Look-back over all tiles of a large input would read as many rows of counts
// as tiles are in flight (hundreds of 2 to 4 KB per tile): with four rows in
// flight, 50M keys took 5.2 ms a pass.  A block per run of consecutive tiles
// needs no look-back, but its neighbours then write far apart and their
// partial sectors do not meet in the L2: 0.48 to 0.82 ms.
// Measured on the entries of 25M cell pairs (50M keys of 18 bits, two passes):
// 38 + 11 + 291 and 40 + 11 + 221 us; with the counts of every tile scanned,
// 53 + 35 + 288 and 51 + 35 + 218, and 95 us for writing the entries first.  A
// pass moves 0.8 GB (115 us at the copy rate); it is bound by the shared-memory
// and match instructions of the ranking.  Look-back groups of 2, 4, 8 and 16
// tiles: 22 + 282, 11 + 291, 8 + 310, 6 + 335 us.  Keys here come in runs, so a
// match instruction is quick (with one vote per digit bit instead: 364 and 350
// us; random keys are the other way round, 520 against 378).
constexpr int kMaxPasses = 8;
template <bool WAVE>
constexpr int kGroup = WAVE ? 16 : 4;

// The keys of the first pass.
enum SortSource {
  kPairsKV = 0,    // key[i], val[i]
  kKeyIndex = 1,   // key[i], value i
  kBothSides = 2,  // key: flat pair element e, value: the other element of its pair
  kFirstSide = 3,  // key: pairs[i].x, value: pairs[i].y
  kSecondSide = 4  // key: pairs[i].y, value i
};
template <class K>
__device__ __forceinline__ K sort_key(const K *key, int src, int64_t i) {
  return src == kFirstSide ? key[2 * i] : src == kSecondSide ? key[2 * i + 1] : key[i];
}

// Device words of a sort.
template <int R>
struct SortCtl {
  int32_t hist[kMaxPasses][R];  // keys per digit
  int32_t base[kMaxPasses][R];  // first position of every digit (one wave)
  unsigned ticket[kMaxPasses];
  unsigned done;
};
// one wave: counts per (tile, digit), 1 + count once there; per (group, digit);
// tiles that added to a group
struct WaveRows {
  int32_t *tile;
  int32_t *group;
  unsigned *arrived;
};

constexpr int kHistBlock = 512;
constexpr int kHistLoads = 8;  // keys in flight per thread

// Adds the digits of keys [i0, i1) to cnt[p * R + digit], p < passes.
template <class K, int R>
__device__ __forceinline__ void count_digits(const K *key, int src, int64_t i0, int64_t i1, int shift0,
                                             int passes, int width, int *cnt) {
  const int t = threadIdx.x, lane = t & 31;
  const unsigned dmask = (1u << width) - 1;
  for (int64_t b = i0; b < i1; b += kHistBlock * kHistLoads) {
    K k[kHistLoads];
#pragma unroll
    for (int u = 0; u < kHistLoads; ++u) {
      const int64_t i = b + u * kHistBlock + t;
      k[u] = i < i1 ? sort_key(key, src, i) : K(0);
    }
#pragma unroll
    for (int u = 0; u < kHistLoads; ++u) {
      const bool valid = b + u * kHistBlock + t < i1;
      const unsigned m = __ballot_sync(0xffffffffu, valid);
      for (int p = 0; p < passes; ++p) {
        const unsigned d = static_cast<unsigned>(k[u] >> (shift0 + p * width)) & dmask;
        // leading digits of neighbouring keys are often equal: one addition
        const unsigned d0 = __shfl_sync(0xffffffffu, d, 0);
        if (__all_sync(0xffffffffu, !valid || d == d0)) {
          if (lane == 0 && m) atomicAdd(&cnt[p * R + d0], __popc(m));
        } else if (valid) {
          atomicAdd(&cnt[p * R + d], 1);
        }
      }
    }
  }
}

// One wave: digits of all passes.
template <class K, int R>
__global__ void __launch_bounds__(kHistBlock) k_sort_hist(const K *key, int src, int64_t n, int passes,
                                                          int width, SortCtl<R> *__restrict__ ctl) {
  pdl_wait();
  extern __shared__ int cnt[];  // [passes][R]
  __shared__ bool last;
  const int t = threadIdx.x, lane = t & 31;
  for (int d = t; d < passes * R; d += kHistBlock) cnt[d] = 0;
  __syncthreads();
  const int64_t per = (n + gridDim.x - 1) / gridDim.x, i0 = blockIdx.x * per;
  count_digits<K, R>(key, src, i0, i0 + per < n ? i0 + per : n, 0, passes, width, cnt);
  __syncthreads();
  for (int d = t; d < passes * R; d += kHistBlock)
    if (cnt[d]) atomicAdd(&ctl->hist[d / R][d % R], cnt[d]);
  __threadfence();
  __syncthreads();
  if (t == 0) last = atomicAdd(&ctl->done, 1u) == gridDim.x - 1;
  __syncthreads();
  if (!last) return;
  // the block that finishes last: first position of every digit, a warp per pass
  __threadfence();
  const int w = t >> 5;
  if (w < passes) {
    int run = 0;
    for (int d0 = 0; d0 < (1 << width); d0 += 32) {
      const int d = d0 + lane;
      const int v = d < (1 << width) ? *reinterpret_cast<volatile int32_t *>(&ctl->hist[w][d]) : 0;
      const int incl = warp_inclusive(v);
      if (d < (1 << width)) ctl->base[w][d] = run + incl - v;
      run += __shfl_sync(0xffffffffu, incl, 31);
    }
  }
}

// Many keys: digits of one pass per group, a block per tile (added up in the
// group's row), and their totals; clears the tile's row.
template <class K, int R>
__global__ void __launch_bounds__(kHistBlock) k_group_hist(const K *key, int src, int64_t n, int ktile,
                                                           int tiles, int pass, int width, SortCtl<R> *__restrict__ ctl,
                                                           WaveRows wave, int64_t ntiles) {
  pdl_wait();
  __shared__ int cnt[R];
  const int t = threadIdx.x, nd = 1 << width, shift = pass * width;
  const unsigned dmask = nd - 1;
  const int64_t tile0 = static_cast<int64_t>(blockIdx.x) * tiles;
  for (int d = t; d < nd; d += kHistBlock) cnt[d] = 0;
  for (int64_t q = 0; q < tiles && tile0 + q < ntiles; ++q)
    for (int d = t; d < nd; d += kHistBlock) wave.tile[(tile0 + q) * R + d] = 0;
  __syncthreads();
  const int64_t i0 = tile0 * ktile, i1 = i0 + static_cast<int64_t>(tiles) * ktile;
  if (src < kFirstSide && i1 <= n) {
    // whole tiles: 16-byte loads (tiles start 16-byte aligned)
    constexpr int kPer = 16 / sizeof(K);
    const uint4 *kv = reinterpret_cast<const uint4 *>(key + i0);
    const int nv = tiles * ktile / kPer;
    for (int b = t; b < nv; b += 4 * kHistBlock) {
      uint4 v[4];
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (b + u * kHistBlock < nv) v[u] = kv[b + u * kHistBlock];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        if (b + u * kHistBlock >= nv) break;
        const K *e = reinterpret_cast<const K *>(&v[u]);
#pragma unroll
        for (int j = 0; j < kPer; ++j) atomicAdd(&cnt[static_cast<unsigned>(e[j] >> shift) & dmask], 1);
      }
    }
  } else {
    for (int64_t i = i0 + t; i < i1 && i < n; i += kHistBlock)
      atomicAdd(&cnt[static_cast<unsigned>(sort_key(key, src, i) >> shift) & dmask], 1);
  }
  __syncthreads();
  for (int d = t; d < nd; d += kHistBlock)
    if (cnt[d]) {
      atomicAdd(&wave.group[tile0 / kGroup<false> * R + d], cnt[d]);
      atomicAdd(&ctl->hist[pass][d], cnt[d]);
    }
}

// rows[group][digit]: counts -> first positions.  A block takes 32 digits.
template <int R>
__global__ void __launch_bounds__(1024) k_group_scan(int ngroup, int pass, const SortCtl<R> *ctl,
                                                     int32_t *__restrict__ rows) {
  pdl_wait();
  __shared__ int part[32][33], wsum[32];
  const int x = threadIdx.x & 31, y = threadIdx.x >> 5;
  const int d0 = 32 * blockIdx.x;
  // keys of lower digits
  int low = 0;
  for (int d = threadIdx.x; d < d0; d += 1024) low += ctl->hist[pass][d];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) low += __shfl_xor_sync(0xffffffffu, low, o);
  if (x == 0) wsum[y] = low;
  const int per = (ngroup + 31) / 32, r0 = y * per, r1 = min(ngroup, r0 + per);
  int s = 0;
  for (int r = r0; r < r1; ++r) s += rows[static_cast<int64_t>(r) * R + d0 + x];
  part[y][x] = s;
  __syncthreads();
  // warp y: prefix over the row groups of digit d0 + y
  const int v = part[x][y];
  const int incl = warp_inclusive(v);
  __syncthreads();
  part[x][y] = incl - v;
  __shared__ int start[32];
  if (y == 0) {
    const int h = ctl->hist[pass][d0 + x];
    int b = warp_inclusive(h) - h;
    for (int q = 0; q < 32; ++q) b += wsum[q];
    start[x] = b;
  }
  __syncthreads();
  int run = start[x] + part[y][x];
  for (int r = r0; r < r1; ++r) {
    int32_t *p = &rows[static_cast<int64_t>(r) * R + d0 + x];
    const int q = *p;
    *p = run;
    run += q;
  }
}

// Stable scatter of tiles.  Warp w owns consecutive keys of the tile and takes
// them 32 at a time in index order: a key's rank among the warp's keys of its
// digit is the warp's running count of that digit (shared memory, updated by
// the first lane of each group of equal digits) plus its rank within the group.
// One exclusive scan over (digit, warp) gives every key its position in the
// tile's stably digit-sorted order; the tile is staged in that order in shared
// memory and written so that consecutive threads store consecutive positions.
//
// Tiles are drawn by ticket, so a tile waits only for tiles already running,
// and the wait is bounded: a block whose predecessors stay silent for
// `spins` polls counts the keys before its tile itself, so the result is right
// either way.
constexpr int kSpins = 1 << 16;

template <class K, int THREADS, int ITEMS, int RB, bool WAVE>
__global__ void __launch_bounds__(THREADS, 1024 / THREADS) k_radix_pass(
    const K *key, const uint32_t *val, int src, int64_t n, int pass, int width,
    SortCtl<(1 << RB)> *__restrict__ ctl, const int32_t *rows, WaveRows wave, int spins,
    K *__restrict__ okey, uint32_t *__restrict__ oval) {
  pdl_wait();
  constexpr int kGroup = ::amfmm::kGroup<WAVE>;
  constexpr int R = 1 << RB, kW = THREADS / 32, kTile = THREADS * ITEMS, kWarpKeys = 32 * ITEMS;
  constexpr int kD = (R + THREADS - 1) / THREADS;  // digits per thread
  constexpr int kCntStride = R + 2;
  constexpr int kCntWords = kW * kCntStride / 2;
  extern __shared__ __align__(16) unsigned char pool[];
  __shared__ int goff[R];
  __shared__ int wsum[kW];
  __shared__ unsigned s_tile;
  static_assert(kTile < 65536, "counts of a tile are 16 bits");
  uint16_t(*cnt)[kCntStride] = reinterpret_cast<uint16_t(*)[kCntStride]>(pool);
  const int t = threadIdx.x, w = t >> 5, lane = t & 31;
  const int shift = pass * width, nd = 1 << width;
  const unsigned dmask = nd - 1, lt = lanemask_lt();
  if (t == 0) s_tile = atomicAdd(&ctl->ticket[pass], 1u);
  K *sk = reinterpret_cast<K *>(pool);
  uint32_t *sv = reinterpret_cast<uint32_t *>(pool + sizeof(K) * kTile);
  for (int q = t; q < kCntWords; q += THREADS) reinterpret_cast<uint32_t *>(pool)[q] = 0;
  __syncthreads();
  const int64_t tile = s_tile, tile0 = tile * kTile;
  const int nvalid = static_cast<int>(n - tile0 < kTile ? n - tile0 : kTile);
    K k[ITEMS];
#pragma unroll
    for (int r = 0; r < ITEMS; ++r) {
      const int li = w * kWarpKeys + r * 32 + lane;
      k[r] = li < nvalid ? sort_key(key, src, tile0 + li) : K(0);
    }
    uint32_t lpos[ITEMS / 2];  // two positions per word
#pragma unroll
    for (int r = 0; r < ITEMS; ++r) {
      const bool valid = w * kWarpKeys + r * 32 + lane < nvalid;
      const int d = valid ? static_cast<int>(static_cast<unsigned>(k[r] >> shift) & dmask) : nd;
      const unsigned peers = __match_any_sync(0xffffffffu, d);
      const int wrank = __popc(peers & lt);
      const int prev = cnt[w][d];
      __syncwarp();
      if (r & 1) lpos[r / 2] |= static_cast<uint32_t>(prev + wrank) << 16;
      else lpos[r / 2] = prev + wrank;
      if (wrank == 0) cnt[w][d] = static_cast<uint16_t>(prev + __popc(peers));
      __syncwarp();
    }
    __syncthreads();
    // exclusive scan over (digit, warp), digit-major: thread t owns digits
    // [t kD, (t + 1) kD)
    int tot[kD], own = 0;
#pragma unroll
    for (int h = 0; h < kD; ++h) {
      tot[h] = 0;
      const int d = t * kD + h;
      if (d < nd) {
#pragma unroll
        for (int q = 0; q < kW; ++q) tot[h] += cnt[q][d];
        // for the tiles after it
        *reinterpret_cast<volatile int32_t *>(&wave.tile[tile * R + d]) = 1 + tot[h];
        if (WAVE && tot[h]) atomicAdd(&wave.group[tile / kGroup * R + d], tot[h]);
      }
      own += tot[h];
    }
    if (WAVE) __threadfence();  // counts before the arrival below
    int incl = own;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += y;
    }
    if (lane == 31) wsum[w] = incl;
    __syncthreads();
    if (WAVE && t == 0) atomicAdd(&wave.arrived[tile / kGroup], 1u);
    int before = incl - own;
    for (int q = 0; q < w; ++q) before += wsum[q];
    int first[kD];  // position of the digit in the sorted tile
#pragma unroll
    for (int h = 0; h < kD; ++h) {
      const int d = t * kD + h;
      first[h] = before;
      if (d < nd) {
#pragma unroll
        for (int q = 0; q < kW; ++q) {
          const int cq = cnt[q][d];
          cnt[q][d] = static_cast<uint16_t>(before);
          before += cq;
        }
      }
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < ITEMS; ++r)
      if (w * kWarpKeys + r * 32 + lane < nvalid)
        lpos[r / 2] += static_cast<uint32_t>(cnt[w][static_cast<unsigned>(k[r] >> shift) & dmask]) << (16 * (r & 1));
    __syncthreads();  // the counts are dead from here; the pool stages the tile
    const auto at = [&](int r) { return (lpos[r / 2] >> (16 * (r & 1))) & 0xffffu; };
#pragma unroll
    for (int r = 0; r < ITEMS; ++r)
      if (w * kWarpKeys + r * 32 + lane < nvalid) sk[at(r)] = k[r];
    // values: read only now, so that they hold no registers while ranking
    uint32_t v[ITEMS];
#pragma unroll
    for (int r = 0; r < ITEMS; ++r) {
      const int li = w * kWarpKeys + r * 32 + lane;
      const int64_t i = tile0 + li;
      v[r] = static_cast<uint32_t>(i);
      if (li < nvalid) {
        if (src == kPairsKV) v[r] = val[i];
        else if (src == kBothSides) v[r] = static_cast<uint32_t>(key[i ^ 1]);
        else if (src == kFirstSide) v[r] = static_cast<uint32_t>(key[2 * i + 1]);
      }
    }
#pragma unroll
    for (int r = 0; r < ITEMS; ++r)
      if (w * kWarpKeys + r * 32 + lane < nvalid) sv[at(r)] = v[r];
    // first position of the thread's digits: all tiles before this one
    const int grp = static_cast<int>(tile / kGroup), g0 = grp * kGroup;
    bool failed = spins == 0;  // (tests: every tile counts for itself)
    if (WAVE) {
      for (int g = failed ? grp : t; g < grp; g += THREADS) {
        int polls = 0;
        while (*reinterpret_cast<volatile unsigned *>(&wave.arrived[g]) < kGroup)
          if (++polls > spins) {
            failed = true;
            break;
          }
      }
      __threadfence();
      failed = __syncthreads_or(failed);
    }
    int run[kD];
#pragma unroll
    for (int h = 0; h < kD; ++h) {
      const int d = t * kD + h;
      run[h] = 0;
      if (d >= nd || failed) continue;
      if (WAVE) {
        const volatile int32_t *gp = wave.group + d;
#pragma unroll 8
        for (int g = 0; g < grp; ++g) run[h] += gp[static_cast<int64_t>(g) * R];
      }
      const volatile int32_t *tp = wave.tile + static_cast<int64_t>(g0) * R + d;
      int x[kGroup - 1];
#pragma unroll
      for (int u = 0; u < kGroup - 1; ++u) x[u] = g0 + u < tile ? tp[static_cast<int64_t>(u) * R] : 1;
#pragma unroll
      for (int u = 0; u < kGroup - 1; ++u) {
        int polls = 0;
        while (x[u] == 0) {
          x[u] = tp[static_cast<int64_t>(u) * R];
          if (++polls > spins) {
            failed = true;
            break;
          }
        }
        run[h] += x[u] - 1;
      }
    }
    if (__syncthreads_or(failed)) {
      // count them: from the group's first tile, or from the first of all
      const int64_t i0 = WAVE ? 0 : static_cast<int64_t>(g0) * kTile;
      for (int d = t; d < nd; d += THREADS) goff[d] = 0;
      __syncthreads();
      for (int64_t i = i0 + t; i < tile0; i += THREADS)
        atomicAdd(&goff[static_cast<unsigned>(sort_key(key, src, i) >> shift) & dmask], 1);
      __syncthreads();
#pragma unroll
      for (int h = 0; h < kD; ++h)
        if (t * kD + h < nd) run[h] = goff[t * kD + h];
      __syncthreads();
    }
#pragma unroll
    for (int h = 0; h < kD; ++h) {
      const int d = t * kD + h;
      if (d < nd) goff[d] = run[h] + (WAVE ? ctl->base[pass][d] : rows[static_cast<int64_t>(grp) * R + d]) - first[h];
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < ITEMS; ++r) {
      const int j = r * THREADS + t;
      if (j < nvalid) {
        const K kk = sk[j];
        const int pos = goff[static_cast<unsigned>(kk >> shift) & dmask] + j;
        okey[pos] = kk;
        oval[pos] = sv[j];
      }
    }
}

template <class K, int THREADS, int ITEMS, int RB, bool WAVE>
int radix_sort_with(fmm_ctx *c, const K *src_key, int src, DBuf key[2], DBuf val[2], int64_t n, int passes, int width,
                    int spins, int *which) {
  constexpr int kGroup = ::amfmm::kGroup<WAVE>;
  constexpr int R = 1 << RB, kW = THREADS / 32, kTile = THREADS * ITEMS;
  constexpr size_t kCntBytes = sizeof(uint16_t) * kW * (R + 2), kStageBytes = (sizeof(K) + 4) * kTile;
  constexpr int kPool = static_cast<int>(kCntBytes > kStageBytes ? kCntBytes : kStageBytes);
  using Ctl = SortCtl<R>;
  constexpr size_t kCtl = (sizeof(Ctl) + 255) / 256 * 256;
  cudaStream_t st = c->stream;
  auto *kern = k_radix_pass<K, THREADS, ITEMS, RB, WAVE>;
  if (kPool > 32 * 1024)
    AMFMM_CUDA(c, cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kPool));
  const int64_t ntiles = (n + kTile - 1) / kTile, ngroups = (ntiles + kGroup - 1) / kGroup;
  // words after the control words: tile rows (per pass in the one-wave form),
  // group rows, arrivals
  const int64_t per_pass = ntiles * R + ngroups * (R + 1);
  const size_t words = static_cast<size_t>(WAVE ? passes * per_pass : per_pass), zero = WAVE ? words : 0;
  AMFMM_TRY(ensure_bytes(c, c->sort_hist, kCtl + sizeof(int32_t) * words));
  Ctl *ctl = static_cast<Ctl *>(c->sort_hist.p);
  int32_t *rows = reinterpret_cast<int32_t *>(static_cast<char *>(c->sort_hist.p) + kCtl);
  AMFMM_CUDA(c, cudaMemsetAsync(ctl, 0, kCtl + sizeof(int32_t) * zero, st));
  if (WAVE) {
    const unsigned hg = static_cast<unsigned>(std::min<int64_t>((n + 2 * kHistBlock - 1) / (2 * kHistBlock),
                                                                2 * static_cast<int64_t>(std::max(1, c->num_sms))));
    launch(c, k_sort_hist<K, R>, hg, kHistBlock, sizeof(int) * passes * R, src_key, src, n, passes, width, ctl);
    AMFMM_TRY(launched(c, "sort_hist"));
  }
  // keys given as arrays are in buffer 0; others are first written there
  int out = src == kPairsKV ? 1 : 0;
  const K *in_key = src_key;
  const uint32_t *in_val = src == kPairsKV ? ptr<uint32_t>(val[0]) : nullptr;
  for (int p = 0; p < passes; ++p) {
    const int from = p == 0 ? src : kPairsKV;
    WaveRows wave;
    wave.tile = rows + (WAVE ? p * per_pass : 0);
    wave.group = wave.tile + ntiles * R;
    wave.arrived = reinterpret_cast<unsigned *>(wave.group + ngroups * R);
    if (!WAVE) {
      // tiles per block: a whole group only where the groups fill the GPU
      const int tiles = ngroups >= 2 * std::max(1, c->num_sms) ? kGroup : 1;
      AMFMM_CUDA(c, cudaMemsetAsync(wave.group, 0, sizeof(int32_t) * ngroups * R, st));
      launch(c, k_group_hist<K, R>, static_cast<unsigned>((ntiles + tiles - 1) / tiles), kHistBlock, 0, in_key, from,
             n, kTile, tiles, p, width, ctl, wave, ntiles);
      AMFMM_TRY(launched(c, "group_hist"));
      launch(c, k_group_scan<R>, ((1 << width) + 31) / 32, 1024, 0, static_cast<int>(ngroups), p, ctl, wave.group);
      AMFMM_TRY(launched(c, "group_scan"));
    }
    launch(c, kern, static_cast<unsigned>(ntiles), THREADS, kPool, in_key, in_val, from, n, p, width, ctl, wave.group,
           wave, spins, ptr<K>(key[out]), ptr<uint32_t>(val[out]));
    AMFMM_TRY(launched(c, "radix_pass"));
    in_key = ptr<K>(key[out]);
    in_val = ptr<uint32_t>(val[out]);
    out ^= 1;
  }
  *which = out ^ 1;
  return FMM_OK;
}

// Few keys (one wave): small tiles, so that all SMs have some; 65,536 keys take
// 11 us a pass and 12 once, 1,048,576 take 25 and 18 (four launches of 18 to 31
// us in all per pass before).  Many: large tiles, for longer runs per digit
// (tiles of 4096 keys: 298 against 291 us a pass of 50M).  Digits of 64-bit keys
// have 9 bits (63 bits in seven passes), others up to 10: 20-bit cell ids in two.
int radix_sort(fmm_ctx *c, const uint64_t *src_key, int src, DBuf key[2], DBuf val[2], int64_t n, int bits, int spins,
               int *which) {
  const int passes = (bits + 8) / 9, width = (bits + passes - 1) / passes;
  AMFMM_TRY(ensure<uint64_t>(c, key[1], n));
  AMFMM_TRY(ensure<uint32_t>(c, val[1], n));
  const int64_t sms = std::max(1, c->num_sms);
#define GO(T, I, W) return radix_sort_with<uint64_t, T, I, 9, W>(c, src_key, src, key, val, n, passes, width, spins, which)
  if (n <= 1024 * 2 * sms) GO(256, 4, true);
  if (n <= 2048 * 4 * sms) GO(256, 8, true);
  GO(256, 16, false);
#undef GO
}
int radix_sort(fmm_ctx *c, const uint32_t *src_key, int src, DBuf key[2], DBuf val[2], int64_t n, int bits, int spins,
               int *which) {
  const int passes = (bits + 9) / 10, width = (bits + passes - 1) / passes;
  AMFMM_TRY(ensure<uint32_t>(c, key[0], n));
  AMFMM_TRY(ensure<uint32_t>(c, val[0], n));
  if (src == kPairsKV || passes > 1) {
    AMFMM_TRY(ensure<uint32_t>(c, key[1], n));
    AMFMM_TRY(ensure<uint32_t>(c, val[1], n));
  }
  const int64_t sms = std::max(1, c->num_sms);
#define GO(T, I, W) return radix_sort_with<uint32_t, T, I, 10, W>(c, src_key, src, key, val, n, passes, width, spins, which)
  if (n <= 1024 * 2 * sms) GO(256, 4, true);
  if (n <= 4096 * 2 * sms) GO(256, 16, true);
  GO(512, 16, false);
#undef GO
}
template <class K>
int sort_arrays(fmm_ctx *c, DBuf key[2], DBuf val[2], int64_t n, int bits, int spins, int *which) {
  *which = 0;
  if (n <= 1 || bits <= 0) return FMM_OK;
  if (n > 0x7fffffffLL) return set_error(c, FMM_EINVAL, "radix sort: n too large");
  return radix_sort(c, ptr<K>(key[0]), kPairsKV, key, val, n, bits, spins, which);
}

}  // namespace

int exclusive_scan_i32(fmm_ctx *c, const int32_t *in, int32_t *out, int64_t n, int32_t *total) {
  return scan_entry<int32_t>(c, in, out, n, total);
}
int exclusive_scan_i64(fmm_ctx *c, const int64_t *in, int64_t *out, int64_t n, int64_t *total) {
  return scan_entry<int64_t>(c, in, out, n, total);
}
int radix_sort_u64(fmm_ctx *c, DBuf key[2], DBuf val[2], int64_t n, int bits, int *which) {
  return sort_arrays<uint64_t>(c, key, val, n, bits, kSpins, which);
}
int radix_sort_u32(fmm_ctx *c, DBuf key[2], DBuf val[2], int64_t n, int bits, int *which) {
  return sort_arrays<uint32_t>(c, key, val, n, bits, kSpins, which);
}
int sort_pair_sides(fmm_ctx *c, const int2 *pairs, int64_t K, bool partner, DBuf key[2], DBuf val[2], int bits,
                    int *which) {
  if (2 * K > 0x7fffffffLL) return set_error(c, FMM_EINVAL, "radix sort: n too large");
  return radix_sort(c, reinterpret_cast<const uint32_t *>(pairs), partner ? kBothSides : kKeyIndex, key, val, 2 * K,
                    bits, kSpins, which);
}
int sort_pairs(fmm_ctx *c, const int2 *pairs, int64_t K, bool second, DBuf key[2], DBuf val[2], int bits, int *which) {
  if (K > 0x7fffffffLL) return set_error(c, FMM_EINVAL, "radix sort: n too large");
  return radix_sort(c, reinterpret_cast<const uint32_t *>(pairs), second ? kSecondSide : kFirstSide, key, val, K, bits,
                    kSpins, which);
}

}  // namespace amfmm

using namespace amfmm;

// Test hook of the sort (no counterpart in the paper): sorts n (key, value)
// pairs given on the device with at most `spins` polls per look-back wait (0: no
// tile waits, each counts the keys before it itself).
extern "C" int fmm_debug_sort(fmm_ctx *c, int key_bytes, const void *key, const uint32_t *val, int64_t n, int bits,
                              int spins, void *okey, uint32_t *oval) {
  if (!c || (key_bytes != 4 && key_bytes != 8) || n < 1 || bits < 1 || bits > 8 * key_bytes - 1 || spins < 0)
    return FMM_EINVAL;
  DBuf k[2], v[2];
  int which = 0;
  const auto run = [&]() -> int {
    AMFMM_TRY(ensure_bytes(c, k[0], static_cast<size_t>(n) * key_bytes));
    AMFMM_TRY(ensure<uint32_t>(c, v[0], n));
    AMFMM_CUDA(c, cudaMemcpyAsync(k[0].p, key, n * key_bytes, cudaMemcpyDeviceToDevice, c->stream));
    AMFMM_CUDA(c, cudaMemcpyAsync(v[0].p, val, n * sizeof(uint32_t), cudaMemcpyDeviceToDevice, c->stream));
    AMFMM_TRY(key_bytes == 8 ? sort_arrays<uint64_t>(c, k, v, n, bits, spins, &which)
                             : sort_arrays<uint32_t>(c, k, v, n, bits, spins, &which));
    AMFMM_CUDA(c, cudaMemcpyAsync(okey, k[which].p, n * key_bytes, cudaMemcpyDeviceToDevice, c->stream));
    AMFMM_CUDA(c, cudaMemcpyAsync(oval, v[which].p, n * sizeof(uint32_t), cudaMemcpyDeviceToDevice, c->stream));
    return FMM_OK;
  };
  const int rc = run();
  cudaStreamSynchronize(c->stream);
  for (DBuf *b : {&k[0], &k[1], &v[0], &v[1]}) cudaFree(b->p);
  return rc;
}
