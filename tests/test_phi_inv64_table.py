"""The FP64 exact path's inverse-Normal quintics (csrc/phi_inv64_table.h): the
integer evaluation the kernels perform (probit_q60 of exact64.cuh, emulated
here) stays within its error bound of -Phi^{-1} computed with 50 digits, and
the committed header is its generator's output (a sample of its parts)."""
import importlib.util
import os
import re

import numpy as np
import pytest

mp = pytest.importorskip("mpmath")
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2502_07123_gb300", "csrc")


@pytest.fixture(scope="module")
def gen():
    spec = importlib.util.spec_from_file_location("gen_phi_inv64_table", os.path.join(CSRC, "gen_phi_inv64_table.py"))
    mod = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(mod)
    return mod


@pytest.fixture(scope="module")
def table():
    txt = open(os.path.join(CSRC, "phi_inv64_table.h")).read()
    v = [int(x, 16) for x in re.findall(r"0x([0-9a-f]+)u", txt)]
    assert len(v) == 4 * 4096
    return [(v[2 * k], v[2 * k + 1], v[8192 + 2 * k], v[8193 + 2 * k]) for k in range(4096)]


def evaluate(J, table):
    """probit_q60 step by step (the assertions: no word overflows)."""
    N = 2 * J + 1
    lz = 32 - N.bit_length()
    M = N << lz
    t = 0x1000000 - (M & 0xFFFFFF)
    T = t << 7
    c0, c1, c2, c34 = table[128 * lz + (M >> 24) - 128]
    a4 = (c34 >> 32) + ((c2 & 0x7FFFF) * T >> 32)
    a3 = (c34 & 0xFFFFFFFF) + (a4 * T >> 32)
    a2 = c2 + a3 * t
    a1 = c1 + (a2 >> 32) * t + ((a2 & 0xFFFFFFFF) * t >> 32)
    assert a4 < 1 << 32 and a3 < 1 << 32 and a2 < 1 << 64 and a1 < 1 << 64
    return c0 + (((a1 >> 32) * t + ((a1 & 0xFFFFFFFF) * t >> 32)) >> 3)


@pytest.mark.parametrize("lz,m", [(0, 0), (0, 127), (1, 64), (3, 127), (4, 0), (17, 5), (31, 0), (31, 127)])
def test_header_is_the_generator_output(gen, table, lz, m):
    c0, c1, c2, c34 = table[128 * lz + m]
    q = gen.part(lz, m)
    assert (c0, c1, c2, c34 & 0xFFFFFFFF, c34 >> 32) == tuple(q[:5]) and c2 & 0x7FFFF == q[5]


def test_error_bound(gen, table):
    """Every octave of u, both ends of parts, the smallest and the largest words."""
    rng = np.random.default_rng(3)
    J = [0, 1, 2, 3, 99, 2**30 - 1, 2**30, 2**30 + 1, 2**31 - 2, 2**31 - 1]
    for lz in range(32):   # N = 2 J + 1 has 32 - lz bits
        lo, hi = (1 << (31 - lz)) // 2, (1 << (32 - lz)) // 2
        J += [int(x) for x in rng.integers(lo, max(lo + 1, hi), 40)]
    for k in rng.integers(0, 1024, 60):   # part edges of the eight upper octaves
        lz, m = divmod(int(k), 128)
        edge = (128 + m) << (23 - lz)     # J at the lower end of the part
        J += [edge - 1, edge]
    err = [mp.mpf(evaluate(j, table)) / 2**60 - gen.probit(mp.mpf(2 * j + 1) / 2**33) for j in J if 0 <= j < 2**31]
    assert max(abs(e) for e in err) <= mp.mpf(2) ** -54
    assert mp.sqrt(sum(e * e for e in err) / len(err)) <= mp.mpf(2) ** -56


def test_monotone(table):
    """y decreases over consecutive words, across part and octave edges too."""
    for j0 in (0, 2**12, 2**23 - 40, 2**30 - 40, 2**31 - 80):
        y = [evaluate(j, table) for j in range(j0, min(j0 + 80, 2**31))]
        assert all(a > b for a, b in zip(y, y[1:]))
