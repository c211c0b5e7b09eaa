"""Generates csrc/expansion_gen.cuh: straight-line CUDA for the field of a local
expansion of App. A at a body (orders P = 4 .. 8), in multi-index form (a, e are
exponent triples, e_k a unit one, a! the product of factorials):
  g_k = - sum_a L^(a+e_k) x^a / a!,  |a| <= P - 1

Run `python gen_expansion.py` to rewrite csrc/expansion_gen.cuh; the build
uses the committed header.
"""
from __future__ import annotations

import math
import os
from fractions import Fraction

ORDERS = (4, 5, 6, 7, 8)
HERE = os.path.dirname(os.path.abspath(__file__))
OUT = os.path.join(HERE, "csrc", "expansion_gen.cuh")


def multi(n):
    """Exponent triples of order n: a = n..0, then b = n-a..0."""
    return [(a, b, n - a - b) for a in range(n, -1, -1) for b in range(n - a, -1, -1)]


def all_multi(P):
    out = []
    for n in range(P + 1):
        out += multi(n)
    return out


def idx_table(P):
    return {m: i for i, m in enumerate(all_multi(P))}


def fact(t):
    return math.factorial(t[0]) * math.factorial(t[1]) * math.factorial(t[2])


def add(a, b):
    return (a[0] + b[0], a[1] + b[1], a[2] + b[2])


def emit_P(P: int) -> str:
    mi = all_multi(P)
    im = idx_table(P)
    L = []
    w = L.append
    w(f"// ---------------- order P = {P}: {len(mi)} moments, {len(mi) - 1} local coefficients ----------------")
    w(f"template <> struct BodyField<{P}> {{")
    w("  // g = -sum_a L^(a+e) x^a / a!")
    w("  __device__ static __forceinline__ void eval(const double *Lc, const double x[3], double g[3]) {")
    w(f"    double px[{P}], py[{P}], pz[{P}], w;")
    w("    px[0] = py[0] = pz[0] = 1.0;")
    w(f"#pragma unroll\n    for (int k = 1; k < {P}; ++k) {{ px[k] = px[k - 1] * x[0]; py[k] = py[k - 1] * x[1]; pz[k] = pz[k - 1] * x[2]; }}")
    w("    g[0] = g[1] = g[2] = 0.0;")
    for a in mi:
        if sum(a) > P - 1:
            continue
        cf = float(Fraction(1, fact(a)))
        mono = " * ".join(f"p{v}[{k}]" for v, k in zip("xyz", a) if k) or "1.0"
        w(f"    w = {cf!r} * ({mono});" if cf != 1.0 else f"    w = {mono};")
        L[-1] += " " + " ".join(f"g[{k}] -= Lc[{im[add(a, e)] - 1}] * w;"
                                for k, e in enumerate(((1, 0, 0), (0, 1, 0), (0, 0, 1))))
    w("  }")
    w("};")
    return "\n".join(L)


def render() -> str:
    parts = ["// expansion_gen.cuh -- GENERATED by gen_expansion.py; do not edit.",
             "// Field of a local expansion of order P at a body (see the generator's",
             "// docstring).  Included by expansion.cu.",
             "#pragma once",
             "",
             "template <int P> struct BodyField;",
             ""]
    for P in ORDERS:
        parts.append(emit_P(P))
        parts.append("")
    return "\n".join(parts) + "\n"


def main():
    with open(OUT, "w") as f:
        f.write(render())
    print(OUT)


if __name__ == "__main__":
    main()
