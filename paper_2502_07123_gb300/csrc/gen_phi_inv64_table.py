"""Writes phi_inv64_table.h: the coefficients of the 64-bit fixed-point inverse
Normal (probit_q60 in exact64.cuh).

y(u) = -Phi^{-1}(u) on u = N 2^-33, N odd in [1, 2^32), is a quintic in each of
4096 parts: the 32 binary octaves of N (lz = leading zeros of N), each cut into
128 equal parts.  With M = N << lz the part is 128 lz + (M >> 24) - 128 and
s = 1 - (M mod 2^24) / 2^24 in (0, 1] its variable, the distance from the part's
upper end in part widths, so y and all its derivatives grow with s and every
coefficient is non-negative.  The quintic interpolates y at the six Chebyshev
nodes, computed with 50 digits and rounded from the top coefficient down; as
integers

    c0 2^60, c1 2^71, c2 2^79 (its low 19 bits hold c5), c3 2^55, c4 2^56, c5 2^57.

Error of the integer evaluation against y: below 2^-54, root mean square
2^-57.8 over uniform words (emulated in tests/test_phi_inv64_table.py).  Run from this directory:

    python gen_phi_inv64_table.py        # rewrites phi_inv64_table.h
"""
import os

import mpmath as mp

OCTAVES, SUB, DEG = 32, 128, 5
mp.mp.dps = 50


def probit(u):
    """-Phi^{-1}(u) for 0 < u <= 1/2 by Newton's method on the Normal tail."""
    x = mp.sqrt(2) * mp.erfinv(1 - 2 * u) if u > 1e-3 else mp.sqrt(-2 * mp.log(u))
    for _ in range(60):
        step = (mp.erfc(x / mp.sqrt(2)) / 2 - u) * mp.sqrt(2 * mp.pi) * mp.exp(x * x / 2)
        x += step
        if abs(step) < mp.mpf(10) ** -35:
            return x
    raise ArithmeticError(u)


def interpolant(ys, nodes):
    """Monomial coefficients of the polynomial through (nodes, ys): divided differences, expanded."""
    n = len(nodes)
    dd = list(ys)
    for j in range(1, n):
        for i in range(n - 1, j - 1, -1):
            dd[i] = (dd[i] - dd[i - 1]) / (nodes[i] - nodes[i - j])
    c = [mp.mpf(0)] * n
    for k in range(n - 1, -1, -1):
        c = [(c[i - 1] if i else 0) - nodes[k] * c[i] for i in range(n)]
        c[0] += dd[k]
    return c


def part(lz, m):
    """Integer coefficients of part (lz, m).  The highest is rounded first and the lower ones refitted to what it
    leaves, and so on down, so that the roundings of c5, c4 and c3 (whose units are the coarse ones) are taken up
    by the coefficients below them.  c4 and c3 carry the half unit that the kernel's truncated products lose."""
    lo = mp.mpf(2) ** (-2 - lz)
    f = lambda s: probit(lo * (1 + (m + 1 - s) / SUB)) if lz or m + 1 < SUB or s else mp.mpf(0)  # noqa: E731
    scale, fixed, q = (60, 71, 79, 55, 56, 57), [mp.mpf(0)] * (DEG + 1), [0] * (DEG + 1)
    ys = {}
    for k in range(DEG, -1, -1):
        nodes = [(1 + mp.cos(mp.pi * (2 * i + 1) / (2 * (k + 1)))) / 2 for i in range(k + 1)]
        for x in nodes:
            if x not in ys:
                ys[x] = f(x)
        c = interpolant([ys[x] - sum(fixed[j] * x ** j for j in range(k + 1, DEG + 1)) for x in nodes], nodes)
        half = mp.mpf(1) / 2 if k in (3, 4) else mp.mpf(0)
        q[k] = max(0, int(mp.nint(c[k] * mp.mpf(2) ** scale[k] + half)))
        if k == 2:                       # c5 2^57 in the low 19 bits
            q[2] = max(0, (q[2] - q[5] + (1 << 18)) >> 19 << 19) + q[5]
        fixed[k] = (q[k] - half) / mp.mpf(2) ** scale[k]
    assert q[0] < 1 << 64 and q[1] < 1 << 64 and q[2] < 1 << 64
    assert q[3] < 1 << 32 and q[4] < 1 << 32 and q[5] < 1 << 19
    return q


def main():
    from concurrent.futures import ProcessPoolExecutor
    with ProcessPoolExecutor() as ex:
        rows = list(ex.map(_octave, range(OCTAVES)))
    rows = [r for octave in rows for r in octave]
    lines = ["// Generated by gen_phi_inv64_table.py: the quintics of -Phi^{-1} by part 128 lz + (M >> 24) - 128;",
             "// k_phi64_a: c0 2^60, c1 2^71; k_phi64_b: c2 2^79 with c5 2^57 in its low 19 bits, c4 2^56 << 32 | c3 2^55.",
             "#pragma once",
             "#include <cuda_runtime.h>",
             "",
             "namespace mlmc {",
             "constexpr int PHI64_SUB = %d, PHI64_PARTS = %d;" % (SUB, len(rows)),
             "static __device__ const ulonglong2 k_phi64_a[PHI64_PARTS] = {"]
    pairs = [["{0x%xu, 0x%xu}" % (r[0], r[1]) for r in rows],
             ["{0x%xu, 0x%xu}" % (r[2], r[4] << 32 | r[3]) for r in rows]]
    lines += ["    %s, %s," % (pairs[0][i], pairs[0][i + 1]) for i in range(0, len(rows), 2)]
    lines += ["};", "static __device__ const ulonglong2 k_phi64_b[PHI64_PARTS] = {"]
    lines += ["    %s, %s," % (pairs[1][i], pairs[1][i + 1]) for i in range(0, len(rows), 2)]
    lines += ["};", "}  // namespace mlmc", ""]
    with open(os.path.join(os.path.dirname(os.path.abspath(__file__)), "phi_inv64_table.h"), "w") as f:
        f.write("\n".join(lines))


def _octave(lz):
    return [part(lz, m) for m in range(SUB)]


if __name__ == "__main__":
    main()
