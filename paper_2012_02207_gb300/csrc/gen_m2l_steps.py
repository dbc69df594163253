"""Generate the swap and z-translation steps of the M2L by degrees (m2l.cu).

  SwapDeg<N, J, M>  the x<->z swap of degree N (Sec. 2.4) from its orders
                    j <= J to its orders m <= M, cosine and sine parts, zero
                    entries skipped. J < N after the z-translation, which
                    leaves F'_n^m = 0 for m > P - n; M < N before it, which
                    reads only those orders;
  ZTrans<P>         Fhat_n^m = sum_k (-1)^{k+m} tz(n,k,m) Mhat_k^m u^k v^n / rho
                    for n + k <= P, in place on the orders m <= min(n, P - n)
                    of every degree (mid_index).

Coefficients are literals in the code (immediates of the instructions); the
values come from gen_swap.py (exact rationals, rounded once to FP64) and are
rounded to FP32 here. Every rounding is written out, so the sums do not depend
on which products a compiler fuses: t0 + t1 + t2 + ... is fma(t0, product t1),
then one fma per term; a coefficient of +-1 gives a sum without a product, and
a negative first product is the rounded one. These are the roundings that the
straight-line steps of gen_m2l.py compile to, and both kernels give the same bits.

Run:  python gen_m2l_steps.py 10 12 14 > m2l_steps.inc
"""
from __future__ import annotations

import os
import struct
import sys

sys.path.insert(0, os.path.dirname(os.path.abspath(__file__)))
import gen_swap  # noqa: E402


def f32(v: float) -> float:
    return struct.unpack("f", struct.pack("f", v))[0]


def lit(v: float) -> str:
    return float.hex(f32(v)) + "f"


def value(c, e):
    """One term: the product c e (a plain operand for c = +-1)."""
    c = f32(c)
    return e if c == 1.0 else ("-%s" % e if c == -1.0 else "__fmul_rn(%s, %s)" % (lit(c), e))


def combination(terms):
    """c0 e0 + c1 e1 + ... as one expression."""
    def product(t):
        return abs(f32(t[0])) != 1.0

    if not terms:
        return "0.0f"
    if len(terms) == 1:
        return value(*terms[0])
    t0, t1 = terms[0], terms[1]
    if product(t0) and product(t1) and f32(t0[0]) < 0.0 < f32(t1[0]):
        acc = "__fmaf_rn(%s, %s, %s)" % (lit(t1[0]), t1[1], value(*t0))
    elif product(t0):
        acc = "__fmaf_rn(%s, %s, %s)" % (lit(t0[0]), t0[1], value(*t1))
    elif product(t1):
        acc = "__fmaf_rn(%s, %s, %s)" % (lit(t1[0]), t1[1], value(*t0))
    else:
        acc = "__f%s_rn(%s, %s)" % ("add" if f32(t1[0]) > 0 else "sub", value(*t0), t1[1])
    for t in terms[2:]:
        if product(t):
            acc = "__fmaf_rn(%s, %s, %s)" % (lit(t[0]), t[1], acc)
        else:
            acc = "__f%s_rn(%s, %s)" % ("add" if f32(t[0]) > 0 else "sub", acc, t[1])
    return acc


def mid_index(P, n, m, im):
    """Place of (n, m) in the vector between the rotations: degrees in order, orders m <= min(n, P - n)."""
    off = sum(2 * min(i, P - i) + 1 for i in range(n))
    return off + (0 if m == 0 else 2 * m - (0 if im else 1))


def main(orders, out=sys.stdout):
    pmax = max(orders)
    U = gen_swap.regular_polys(pmax)
    blocks = {n: gen_swap.hat_blocks(n, gen_swap.swap_blocks(U, n)) for n in range(pmax + 1)}
    tz = gen_swap.translation_coefficients(pmax)
    w = out.write
    w("// Generated by gen_m2l_steps.py; do not edit.\n")
    w("template <int N, int J, int M> struct SwapDeg;\n")
    w("template <int P> struct ZTrans;\n")
    combos = sorted({(n, j, m) for P in orders for n in range(1, P + 1)
                     for j, m in ((n, n), (n, min(n, P - n)), (min(n, P - n), n))})
    for n, J, M in combos:
        A, B = blocks[n]
        # x, y: 2n + 1 values as [Re 0, Re 1, Im 1, ...]
        w("template <> struct SwapDeg<%d, %d, %d> {\n" % (n, J, M))
        w("  static __device__ __forceinline__ void run(const float* x, float* y) {\n")
        for m in range(M + 1):
            terms = [(A[m][j], "x[%d]" % (2 * j - 1 if j else 0)) for j in range(J + 1)
                     if (j + m + n) % 2 == 0 and A[m][j] != 0.0]
            w("    y[%d] = %s;\n" % (2 * m - 1 if m else 0, combination(terms)))
            if m:
                terms = [(B[m - 1][j - 1], "x[%d]" % (2 * j)) for j in range(1, J + 1)
                         if (j + m + n) % 2 == 1 and B[m - 1][j - 1] != 0.0]
                w("    y[%d] = %s;\n" % (2 * m, combination(terms)))
        w("  }\n};\n")
    for P in orders:
        w("template <> struct ZTrans<%d> {\n" % P)
        w("  static __device__ __forceinline__ void run(float* s, float u, float v, float irho) {\n")
        for k in range(1, P + 1):
            w("    const float up%d = %s, vp%d = __fmul_rn(%s, v);\n" % (k, "u" if k == 1 else "__fmul_rn(up%d, u)" % (k - 1), k,
                                                              "irho" if k == 1 else "vp%d" % (k - 1)))
        for m in range(P // 2 + 1):
            w("    {\n")
            parts = ("r", "i") if m else ("r",)
            for k in range(m, P - m + 1):
                for q in parts:
                    at = mid_index(P, k, m, q == "i")
                    w("      const float %s%d = %s;\n" % (q, k, "s[%d]" % at if k == 0 else "__fmul_rn(up%d, s[%d])" % (k, at)))
            for n in range(m, P - m + 1):
                for q in parts:
                    terms = [((-1.0) ** (k + m) * tz[(n, k, m)], "%s%d" % (q, k)) for k in range(m, P - n + 1)]
                    if n == 0:  # (the last input of the monopole's sum is fused with its power of u)
                        head = combination(terms[:-1])
                        # (all orders here are even, so the last sign is +; 1/rho follows at the accumulation)
                        w("      s[0] = __fmaf_rn(up%d, s[%d], %s);\n" % (P, mid_index(P, P, 0, False), head))
                        continue
                    w("      s[%d] = __fmul_rn(vp%d, %s);\n" % (mid_index(P, n, m, q == "i"), n, combination(terms))
                      if n else "")
            w("    }\n")
        w("  }\n};\n")


if __name__ == "__main__":
    main([int(x) for x in sys.argv[1:]] or [10, 12, 14])
