"""The FP64 near field's fixed-point arithmetic (csrc/fix64.cuh), compiled for
the host: the sum over a batch of sources against extended precision, with the
hardware seed of 1/r replaced by one perturbed up to its error bound."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1706_06989_gb300", "csrc")

SOURCE = r"""
#include <algorithm>
#include <cstdlib>
#include "fix64.cuh"
namespace amfmm { namespace fix { float seed_error = 0; } }
using namespace amfmm::fix;
// The kernel's steps for one target: batches of 32 sources, one window each.
// Returns the number of sources left to FP64 (not summed).
extern "C" int near_sum(int ns, const double *t, const double *s, const double *m, double scale,
                        float err, double *out, unsigned char *taken) {
  seed_error = err;
  const int g0 = extent_exponent(scale) - 95;
  W96 pt[3], o[3], ref[3];
  uint32_t rmag = 0;
  for (int c = 0; c < 3; ++c) {
    pt[c] = fixed96(t[c], g0);
    ref[c] = fixed96(s[c], g0);
    o[c] = sub96(pt[c], ref[c]);
    rmag = std::max(rmag, top_mag(o[c]));
  }
  uint64_t M;
  int em, heavy = -5000, left = 0;
  for (int j = 0; j < ns; ++j) {
    mantissa64(m[j], &M, &em);
    heavy = std::max(heavy, em);
  }
  Acc a;
  acc_clear(a);
  int unit = -1000;
  out[0] = out[1] = out[2] = 0;
  auto flush = [&] {
    for (int c = 0; c < 3; ++c)
      out[c] += __builtin_ldexp(static_cast<double>(a.a2[c]) * 536870912.0 + static_cast<double>(a.a1[c]), a.Ua + 2 * kDig);
    acc_clear(a);
  };
  for (int j0 = 0; j0 < ns; j0 += 32) {
    const int n = std::min(32, ns - j0);
    W96 ps[32][3];
    uint32_t cmag = 0;
    for (int j = 0; j < n; ++j)
      for (int c = 0; c < 3; ++c) {
        ps[j][c] = fixed96(s[3 * (j0 + j) + c], g0);
        cmag = std::max(cmag, top_mag(sub96(ps[j][c], ref[c])));
      }
    const int sh = window_shift(rmag, cmag), gd = g0 + sh;
    if (std::abs(sh - unit) > kWinSpan) {
      flush();
      a.Ua = unit_guess(gd, heavy);
      unit = sh;
    }
    int32_t H[3], L[3];
    bool rounded = false;
    for (int c = 0; c < 3; ++c) rounded |= digits(o[c], sh, &H[c], &L[c]);
    int32_t h[32][3], lo[32][3];
    for (int j = 0; j < n; ++j)
      for (int c = 0; c < 3; ++c) rounded |= digits(sub96(ps[j][c], ref[c]), sh, &h[j][c], &lo[j][c]);
    int terms = 0;
    for (int j = 0; j < n; ++j) {
      int32_t dH[3], dL[3], qd[3];
      for (int c = 0; c < 3; ++c) dH[c] = H[c] - h[j][c], dL[c] = L[c] - lo[j][c];
      int64_t hi;
      uint32_t rem;
      square(dH, dL, &hi, &rem);
      int shc = sh, s2;
      if (is_close(hi, rounded ? kCloseRounded : kCloseExact)) {
        shc = close_digits(pt, ps[j], dH, dL);
        square(dH, dL, &hi, &rem);
      }
      taken[j0 + j] = 0;
      if (shc == kNoDigits) { ++left; continue; }
      const uint64_t w = inv_cube(hi, rem, &s2);
      mantissa64(m[j0 + j], &M, &em);
      const uint64_t q = times_mass(w, static_cast<uint32_t>(M >> 32), static_cast<uint32_t>(M));
      const int k = k_base(a.Ua, gd) + 2 * (shc - sh) - em - 3 * s2;
      if (static_cast<unsigned>(k) >= kShiftEnd) { ++left; continue; }
      taken[j0 + j] = 1;
      ++terms;
      factor_digits(q, k, qd);
      acc_add(a, qd, dH, dL);
    }
    acc_carry(a, terms);
  }
  flush();
  return left;
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("fix64")
    (d / "near.cpp").write_text(SOURCE)
    so = d / "near.so"
    subprocess.run(["g++", "-O2", "-std=gnu++17", "-shared", "-fPIC", "-I", CSRC, "-o", str(so), str(d / "near.cpp")],
                   check=True)
    f = ctypes.CDLL(str(so)).near_sum
    P = ctypes.c_void_p
    f.argtypes = [ctypes.c_int, P, P, P, ctypes.c_double, ctypes.c_float, P, P]
    return f


@pytest.mark.parametrize("kind", ["plain", "offset", "origin", "close", "masses", "grid"])
@pytest.mark.parametrize("log2_unit", [-90, 0, 90])
def test_sum_of_a_target_matches_extended_precision(lib, kind, log2_unit):
    """A term's factor is good to 2^-54 and a difference to one unit of 2^-57
    of its window, which is at most 2^7 of a pair's distance: each term is
    within 2^-49 of itself (sqrt(3) and both factors' share included)."""
    rng = np.random.default_rng(7)
    L = np.longdouble
    unit = 2.0 ** log2_unit
    for trial in range(200):
        ns = int(rng.integers(1, 130))
        size = 10.0 ** rng.uniform(-3, 0)
        centre = {"origin": 0.0, "offset": 1e3}.get(kind, 1.0) * rng.uniform(-1, 1, 3)
        t = centre + size * rng.uniform(-1, 1, 3)
        s = centre + size * rng.uniform(-1, 1, (ns, 3))
        m = rng.uniform(0.1, 1.0, ns)
        if kind == "close":
            s[::3] = t + size * 10.0 ** rng.uniform(-12, -1, (len(s[::3]), 1)) * rng.normal(size=(len(s[::3]), 3))
        if kind == "masses":
            m = 10.0 ** rng.uniform(-12, 12, ns)
        if kind == "grid":
            t, s = np.round(t * 64) / 64, np.round(s * 64) / 64
        t, s, m = t * unit, np.ascontiguousarray(s * unit), m * unit
        scale = 2.0 ** 21 / (4.0 * unit)
        out, taken = np.zeros(3), np.zeros(ns, dtype=np.uint8)
        p = lambda a: a.ctypes.data  # noqa: E731
        left = lib(ns, p(t), p(s), p(m), scale, float(rng.uniform(-2.4e-7, 2.4e-7)), p(out), p(taken))
        d = t.astype(L) - s.astype(L)
        r2 = (d * d).sum(1)
        use = taken.astype(bool) & (r2 > 0)
        assert left == ns - int(taken.sum())
        assert not np.any(taken.astype(bool) & (r2 == 0))
        term = (m.astype(L)[use] / (r2[use] * np.sqrt(r2[use])))[:, None] * d[use]
        err = np.sqrt(((out.astype(L) - term.sum(0)) ** 2).sum())
        assert err <= 2.0 ** -49 * np.sqrt((term ** 2).sum(1)).sum(), (kind, trial, ns)
