"""The 110-bit software floating point (csrc/qf.cuh, host side) against big integers: the bounds that its header states."""
import ctypes
import os
import random
import shutil
import subprocess
from fractions import Fraction

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2106_01445_gb300", "csrc")
NVCC = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"

SOURCE = r'''
#include "qf.cuh"
extern "C" void run(int op, int n, const qf *a, const qf *b, const qf *c, const qf *d, const qf *e, qf *r) {
    for (int i = 0; i < n; ++i) {
        switch (op) {
        case 0: r[i] = qf_mul<false>(a[i], b[i]); break;
        case 1: r[i] = qf_mul<true>(a[i], b[i]); break;
        case 2: r[i] = a[i] + b[i]; break;
        case 3: r[i] = a[i] - b[i]; break;
        case 4: r[i] = qf_dot2<false, false>(a[i], b[i], c[i], d[i]); break;
        case 5: r[i] = qf_dot2<false, true>(a[i], b[i], c[i], d[i]); break;
        case 6: r[i] = qf_dot2s(true, a[i], b[i], false, c[i], d[i]); break;
        case 7: r[i] = qf_fma<false>(e[i], a[i], b[i]); break;
        case 8: r[i] = qf_fma<true>(e[i], a[i], b[i]); break;
        case 9: r[i] = qf_fma<false, true>(e[i], a[i], b[i]); break;
        case 10: r[i] = qf_fms2(e[i], a[i], b[i], c[i], d[i]); break;
        case 11: r[i] = qf_half(a[i]); break;
        }
    }
}
extern "C" void dots(int n, int k, const qf *a, const qf *b, qf *r) {
    for (int i = 0; i < n; ++i)
        r[i] = qf_dot(0, 1, k, [&](int j) { return a + i * k + j; }, [&](int j) { return b + i * k + j; });
}
extern "C" void from(int n, const double *x, qf *r) {
    for (int i = 0; i < n; ++i) r[i] = qf_from_double(x[i]);
}
'''


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    if not os.path.exists(NVCC):
        pytest.skip("no nvcc")
    d = tmp_path_factory.mktemp("qf")
    (d / "qf_host.cu").write_text(SOURCE)
    subprocess.run([NVCC, "-std=c++17", "-O1", "-gencode", "arch=compute_103a,code=sm_103a", "-I", CSRC, "-shared",
                    "-Xcompiler", "-fPIC", "-o", str(d / "qf_host.so"), str(d / "qf_host.cu")], check=True, capture_output=True)
    return ctypes.CDLL(str(d / "qf_host.so"))


def pack(m, e):
    """m 2^-110 4^e, 2^109 <= |m| <= 2^111."""
    u = m & ((1 << 112) - 1)
    w = [(u >> (30 * k)) & 0x3fffffff for k in range(3)]
    return w + [((u >> 90) << 10 | (e + 512)) & 0xffffffff]


def value(w):
    m = w[0] | w[1] << 30 | w[2] << 60 | (w[3] >> 10) << 90
    if m >> 111:
        m -= 1 << 112
    assert m == 0 or 1 << 109 <= abs(m) <= 1 << 111
    return Fraction(m) * Fraction(4) ** ((w[3] & 1023) - 512) / (1 << 110)


def numbers(rng, n):
    out = []
    for _ in range(n):
        kind = rng.random()
        m = (1 << 109) + rng.getrandbits(109) if kind < 0.6 else rng.choice([1 << 109, (1 << 111) - 1, 1 << 110, (1 << 110) - 1])
        if kind < 0.3:
            m = min(2 * m, (1 << 111) - 1)
        m = rng.choice([-1, 1]) * m
        out.append(pack(m, rng.choice([0, 0, 0, 1, -1, 2, -3, 10, -20, 54, -55, 60])) if rng.random() > 0.03 else [0, 0, 0, 0])
    return np.array(out, dtype=np.uint32)


def call(f, *args):
    f(*[a.ctypes.data_as(ctypes.c_void_p) if isinstance(a, np.ndarray) else a for a in args])


# terms of the result as products of (sign, operand letters), and the bound against the largest of them
OPS = {0: ([(1, "ab")], 2.0 ** -109), 1: ([(-1, "ab")], 2.0 ** -109), 2: ([(1, "a"), (1, "b")], 2.0 ** -108),
       3: ([(1, "a"), (-1, "b")], 2.0 ** -108), 4: ([(1, "ab"), (1, "cd")], 2.0 ** -106), 5: ([(1, "ab"), (-1, "cd")], 2.0 ** -106),
       6: ([(-1, "ab"), (1, "cd")], 2.0 ** -106), 7: ([(1, "e"), (1, "ab")], 2.0 ** -106), 8: ([(1, "e"), (-1, "ab")], 2.0 ** -106),
       9: ([(-1, "e"), (1, "ab")], 2.0 ** -106), 10: ([(1, "e"), (-1, "ab"), (-1, "cd")], 2.0 ** -105), 11: ([(Fraction(1, 2), "a")], 2.0 ** -109)}


@pytest.mark.parametrize("op", sorted(OPS))
def test_operation(lib, op):
    rng = random.Random(op)
    n = 3000
    x = {k: numbers(rng, n) for k in "abcde"}
    if op in (4, 5, 6, 10):  # cancelling ones among them
        x["c"][::3], x["d"][::3] = x["a"][::3], x["b"][::3]
    if op == 3:
        x["b"][::3] = x["a"][::3]
    r = np.empty((n, 4), dtype=np.uint32)
    call(lib.run, op, n, *[x[k] for k in "abcde"], r)
    v = {k: [value([int(w) for w in row]) for row in x[k]] for k in "abcde"}
    terms, bound = OPS[op]
    for i in range(n):
        parts = []
        for s, letters in terms:
            t = Fraction(s)
            for k in letters:
                t *= v[k][i]
            parts.append(t)
        got = value([int(w) for w in r[i]])
        assert abs(got - sum(parts)) <= Fraction(bound) * max(abs(t) for t in parts), (op, i)


@pytest.mark.parametrize("k", [1, 2, 7, 40, 64])
def test_dot(lib, k):
    rng = random.Random(k)
    n = 200
    a, b = numbers(rng, n * k), numbers(rng, n * k)
    r = np.empty((n, 4), dtype=np.uint32)
    call(lib.dots, n, k, a, b, r)
    for i in range(n):
        t = [value([int(w) for w in a[i * k + j]]) * value([int(w) for w in b[i * k + j]]) for j in range(k)]
        assert abs(value([int(w) for w in r[i]]) - sum(t)) <= (k + 1) * Fraction(2) ** -107 * max(abs(x) for x in t)


def test_from_double(lib):
    x = np.array([0.0, -0.0, 1.0, -1.0, 1e-300, -3e300, 2.0 ** -1074, np.pi, 1 / 3, 2.0 ** 1023])
    r = np.empty((len(x), 4), dtype=np.uint32)
    call(lib.__getitem__("from"), len(x), x, r)
    for v, w in zip(x, r):
        w = [int(q) for q in w]
        if abs(v) < 2.0 ** -1022 and v:  # below the exponents' range
            assert value(w) in (0, Fraction(v))
        elif (w[3] & 1023) != 1023:
            assert value(w) == Fraction(v)
        else:
            assert abs(v) >= 2.0 ** 1022
    bad = np.array([np.nan, np.inf, -np.inf])
    call(lib.__getitem__("from"), 3, bad, r[:3])
    assert all((int(w[3]) & 1023) == 1023 for w in r[:3])
