// geom.cuh -- the opening criterion and the records of the walk's frontier, shared
// by the walk and the learned selector.
//
// Sec. 2: the criterion compares centres of mass, so Z must come out identical
// wherever it is computed.  A leaf sums its bodies in sorted order, any other
// cell its children in octant order, Z = S / M, every step an explicitly rounded
// FP64 operation (no FMA contraction).
#pragma once

namespace amfmm {

// ---- opening criterion (Sec. 2), shared by the walk and the learned selector ----
// per cell {Z_x, Z_y, Z_z, R_max}, one 32-byte load
__device__ __forceinline__ bool well_separated(const double4_32a a, const double4_32a b, double theta) {
  const double dx = __dsub_rn(a.x, b.x);
  const double dy = __dsub_rn(a.y, b.y);
  const double dz = __dsub_rn(a.z, b.z);
  const double d2 = __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
  const double th2 = __dmul_rn(theta, theta);
  const double s = __dadd_rn(a.w, b.w);
  return __dmul_rn(th2, d2) >= __dmul_rn(s, s);
}

// FP32 filter of the criterion.  On this GPU an FP64 operation costs about
// as much as 64 FP32 ones, so the walk first evaluates theta^2 d^2 - (R_A +
// R_B)^2 in FP32, from Z split into hi + lo floats (d carries FP32 relative
// accuracy even for close centres).  Each side of the comparison then has a
// relative error below 1e-6 against its exact value, and so does the FP64
// expression; when the two sides differ by more than 1e-5 of their sum, the
// FP32 sign is therefore the FP64 decision.  The lo parts carry an absolute
// error of about 2^-48 |Z| each; for centres closer than ~2^-20 |Z| that term
// outgrows the relative bound, so the tolerance adds 3e-21 max|Z|^2, which
// covers it (2 d e <= 1e-6 d^2 + 1e6 e^2).  Closer calls, and values outside
// the comfortable FP32 range, return -1 and are decided in FP64.
struct CellF {
  float4 h;  // Z hi (x, y, z), R_max rounded to FP32
  float4 l;  // Z - hi (x, y, z), bits of nchild | level << 8
};

__device__ __forceinline__ int separated_fast(const CellF &a, const CellF &b, float th2) {
  const float dx = (a.h.x - b.h.x) + (a.l.x - b.l.x);
  const float dy = (a.h.y - b.h.y) + (a.l.y - b.l.y);
  const float dz = (a.h.z - b.h.z) + (a.l.z - b.l.z);
  const float lhs = th2 * (dx * dx + dy * dy + dz * dz);
  const float sr = a.h.w + b.h.w;
  const float rhs = sr * sr;
  const float tot = lhs + rhs;
  if (!(tot > 1e-30f && tot < 1e30f)) return -1;
  const float m = fmaxf(fmaxf(fmaxf(fabsf(a.h.x), fabsf(a.h.y)), fabsf(a.h.z)),
                        fmaxf(fmaxf(fabsf(b.h.x), fabsf(b.h.y)), fabsf(b.h.z)));
  const float diff = lhs - rhs, tol = 1e-5f * tot + 3e-21f * m * m;
  if (diff > tol) return 1;
  if (diff < -tol) return 0;
  return -1;
}

// ---- records of the walk's frontier ----
// Up to eight pairs: {first varying cell, fixed cell, n | side << 4} stands for
// (v + a, fixed), a < n (side 1: (fixed, v + a)); the pairs of a cell's children
// f .. f + k - 1 with themselves, (f, f) .. (f+k-1, f+k-1), (f, f+1), (f, f+2) ..,
// from the q-th on, are {f, k, n | 32 | q << 8}.
__device__ __forceinline__ int4 split_record(int first, int n, int fixed, bool second) {
  return make_int4(first, fixed, n | (second ? 16 : 0), 0);
}
__device__ __forceinline__ int4 self_record(int first, int k, int q, int n) {
  return make_int4(first, k, n | 32 | (q << 8), 0);
}
__device__ __forceinline__ bool front_pair(int4 rec, int a, int2 &pr) {
  if (a >= (rec.z & 15)) return false;
  if (rec.z & 32) {
    int q = (rec.z >> 8) + a, i = 0;
    if (q < rec.y) {
      pr = make_int2(rec.x + q, rec.x + q);
    } else {
      q -= rec.y;
      while (q >= rec.y - 1 - i) q -= rec.y - 1 - i++;
      pr = make_int2(rec.x + i, rec.x + i + 1 + q);
    }
  } else {
    pr = rec.z & 16 ? make_int2(rec.y, rec.x + a) : make_int2(rec.x + a, rec.y);
  }
  return true;
}

}  // namespace amfmm
