"""The FP64 near field's steps for one target (csrc/p2p64.cu on csrc/fix64.cuh),
compiled for the host: batches of 32 sources, one window each, taken in classes of
mass; pairs that the integers leave are added in FP64 as the kernel does."""
import ctypes
import os
import subprocess

import numpy as np

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1706_06989_gb300", "csrc")

SOURCE = r"""
#include <algorithm>
#include <cmath>
#include <cstdlib>
#include "fix64.cuh"
namespace amfmm { namespace fix { float seed_error = 0; } }
using namespace amfmm::fix;
namespace {
void pair64(const double *t, const double *s, double m, double eps2, double f[3]) {
  const double d[3] = {t[0] - s[0], t[1] - s[1], t[2] - s[2]};
  const double d2 = std::fma(d[2], d[2], std::fma(d[1], d[1], d[0] * d[0]));
  const double ri = d2 == 0 ? 0 : 1 / std::sqrt(d2 + eps2), q = m * (ri * ri * ri);
  for (int c = 0; c < 3; ++c) f[c] += q * d[c];
}
}  // namespace
// own: the target's place among the sources, -1 if it is none.  how[j]: 0
// integers, 1 integers in a window of the pair's own, 2 FP64.
extern "C" void near_sum(int ns, const double *t, const double *s, const double *m, int own, double scale, double eps2,
                         float err, double *out, unsigned char *how) {
  seed_error = err;
  const bool soft = eps2 > 0;
  const int g0 = extent_exponent(scale) - 95;
  W96 pt[3], o[3], ref[3];
  uint32_t rmag = 0;
  for (int c = 0; c < 3; ++c) {
    pt[c] = fixed96(t[c], g0);
    ref[c] = fixed96(s[c], g0);
    o[c] = sub96(pt[c], ref[c]);
    rmag = std::max(rmag, top_mag(o[c]));
  }
  int unit = -100000, terms = 0;
  Acc a;
  acc_clear(a);
  out[0] = out[1] = out[2] = 0;
  auto flush = [&] {
    acc_carry(a, terms);
    for (int c = 0; c < 3; ++c)
      out[c] += std::ldexp(std::fma(static_cast<double>(a.a2[c]), 536870912.0, static_cast<double>(a.a1[c])),
                           a.Ua + 2 * kDig);
    acc_clear(a);
    terms = 0;
  };
  for (int j0 = 0; j0 < ns; j0 += 32) {
    const int n = std::min(32, ns - j0);
    W96 ps[32][3];
    uint64_t M[32];
    int em[32];
    uint32_t cmag = 0;
    for (int j = 0; j < n; ++j) {
      mantissa64(m[j0 + j], &M[j], &em[j]);
      for (int c = 0; c < 3; ++c) {
        ps[j][c] = fixed96(s[3 * (j0 + j) + c], g0);
        cmag = std::max(cmag, top_mag(sub96(ps[j][c], ref[c])));
      }
    }
    const int sh = window_shift(rmag, cmag), gd = g0 + sh;
    int32_t H[3], L[3], h[32][3], lo[32][3];
    bool rounded = false;
    for (int c = 0; c < 3; ++c) rounded |= digits(o[c], sh, &H[c], &L[c]);
    for (int j = 0; j < n; ++j)
      for (int c = 0; c < 3; ++c) rounded |= digits(sub96(ps[j][c], ref[c]), sh, &h[j][c], &lo[j][c]);
    const int32_t bound = soft || rounded ? kCloseRounded : kCloseExact;
    const int class_span = soft ? kSoftClassSpan : kClassSpan, unit_span = soft ? kSoftUnitSpan : kUnitSpan;
    Soft sw{};
    if (soft) sw = soft_window(eps2, gd);
    bool todo[32];
    for (int j = 0; j < n; ++j) todo[j] = true;
    for (;;) {
      const int none = -100000;
      int top = none, heavy = none;
      for (int j = 0; j < n; ++j)
        if (todo[j]) top = std::max(top, em[j]);
      if (top == none) break;
      // the heaviest source; a single heaviest body at the target's place is none
      int tops = 0, at = 0;
      for (int j = 0; j < n; ++j)
        if (todo[j] && em[j] == top) ++tops, at = j;
      heavy = top;
      bool here = true;
      for (int c = 0; c < 3; ++c) here = here && h[at][c] == H[c] && lo[at][c] == L[c];
      if (!soft && tops == 1 && here) {
        heavy = none;
        for (int j = 0; j < n; ++j)
          if (todo[j] && em[j] != top) heavy = std::max(heavy, em[j]);
      }
      const int u = soft ? unit_soft(gd, heavy, sw) : unit_guess(gd, heavy);
      if (heavy >= top - class_span && std::abs(u - unit) > unit_span) {
        flush();
        a.Ua = unit = u;
      }
      const int kb = k_base(a.Ua, gd) + 3 * sw.t;
      for (int j = 0; j < n; ++j) {
        if (!todo[j] || em[j] < top - class_span) continue;
        todo[j] = false;
        how[j0 + j] = 2;
        if (j0 + j == own) continue;
        int32_t dH[3], dL[3], qd[3];
        for (int c = 0; c < 3; ++c) dH[c] = H[c] - h[j][c], dL[c] = L[c] - lo[j][c];
        int64_t hi;
        uint32_t rem;
        square(dH, dL, &hi, &rem);
        const bool close = is_close(hi, bound);
        int shc = sh, s2;
        if (close) {
          shc = soft ? kNoDigits : close_digits(pt, ps[j], dH, dL);
          square(dH, dL, &hi, &rem);
        }
        if (shc != kNoDigits) {
          if (soft) soften(sw, &hi, &rem);
          const uint64_t w = inv_cube(hi, rem, &s2);
          const uint64_t q = times_mass(w, static_cast<uint32_t>(M[j] >> 32), static_cast<uint32_t>(M[j]));
          const int k = kb + 2 * (shc - sh) - em[j] - 3 * s2;
          if (static_cast<unsigned>(k) < kShiftEnd) {
            factor_digits(q, k, qd);
            acc_add(a, qd, dH, dL);
            ++terms;
            how[j0 + j] = close;
          }
        }
        if (how[j0 + j] == 2) pair64(t, s + 3 * (j0 + j), m[j0 + j], eps2, out);
      }
      acc_carry(a, terms);
      terms = 0;
    }
  }
  flush();
}
"""


def build(directory):
    """near_sum as a Python function: (target, sources, masses, own=place of the
    target among them) -> (sum of m (t - s) / (r^2 + eps^2)^(3/2), how[])."""
    src, so = os.path.join(directory, "near.cpp"), os.path.join(directory, "near.so")
    with open(src, "w") as f:
        f.write(SOURCE)
    subprocess.run(["g++", "-O2", "-std=gnu++17", "-shared", "-fPIC", "-I", CSRC, "-o", so, src], check=True)
    f = ctypes.CDLL(so).near_sum
    P, D = ctypes.c_void_p, ctypes.c_double
    f.argtypes = [ctypes.c_int, P, P, P, ctypes.c_int, D, D, ctypes.c_float, P, P]
    f.restype = None

    def near_sum(t, s, m, eps=0.0, own=-1, err=0.0, extent=None):
        t, s, m = (np.ascontiguousarray(v, dtype=np.float64) for v in (t, s, m))
        p = np.vstack([t[None], s])
        ext = (p.max(0) - p.min(0)).max() if extent is None else extent
        out, how = np.zeros(3), np.zeros(len(s), dtype=np.uint8)
        f(len(s), t.ctypes.data, s.ctypes.data, m.ctypes.data, own, 2.0 ** 21 / ext, eps * eps, err, out.ctypes.data,
          how.ctypes.data)
        return out, how

    return near_sum


def exact(t, s, m, eps=0.0):
    """The sum in extended precision, and the sum of its terms' magnitudes."""
    L = np.longdouble
    d = t.astype(L) - s.astype(L)
    r2 = (d * d).sum(1)
    e2 = r2 + L(eps * eps)
    q = np.where(r2 > 0, m.astype(L) / np.where(r2 > 0, e2 * np.sqrt(e2), 1), 0)
    term = q[:, None] * d
    return term.sum(0), float(np.sqrt((term ** 2).sum(1)).sum())
