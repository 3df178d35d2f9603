"""The fixed-point arithmetic of the Type-I terms and the accumulators (csrc/rs_numeric.cuh),
compiled as host C++ (no GPU), against exact integers: the rounding of the directed values, the pair
products and their sums, the scaling, the three-word sums and their conversion."""
import ctypes
import math
import os
import random
import shutil
import subprocess
from fractions import Fraction

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2508_01485_gb300", "csrc")
S_MAX = (24 * 2.0 ** 24) ** (1 / 3)                       # w <= L log2 L, L < 2^24
S_MIN = 0.0142                                            # two communities, one member of 2^24 - 1
M64 = (1 << 64) - 1


@pytest.fixture(scope="module")
def lib():
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no host C++ compiler")
    out = os.path.join(HERE, "_build", "libnumericpairs.so")
    os.makedirs(os.path.dirname(out), exist_ok=True)
    tmp = out + ".%d.tmp" % os.getpid()
    subprocess.check_call([cxx, "-O2", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, "-o", tmp,
                           os.path.join(HERE, "numeric_pairs_host.cpp")])
    os.replace(tmp, out)
    L = ctypes.CDLL(out)
    u64, P, I = ctypes.c_uint64, ctypes.c_void_p, ctypes.c_int
    L.sig.restype, L.sig.argtypes = u64, [ctypes.c_float, ctypes.c_float]
    L.pair.argtypes = [u64, u64, P]
    L.add96.argtypes = [P, P]
    L.limb_sum.argtypes = [P, I, P]
    L.scaled.argtypes = [u64, P, P]
    L.term192.argtypes = [u64, u64, P]
    L.add192.argtypes = [P, P, I, I]
    L.to_double.restype, L.to_double.argtypes = ctypes.c_double, [P]
    return L


def _words(v, n):
    return np.array([(v >> (64 * i)) & M64 for i in range(n)], np.uint64)


def _int(a):
    return sum(int(x) << (64 * i) for i, x in enumerate(a))


def _call(n, f, *args):
    out = np.zeros(n, np.uint64)
    f(*args, out.ctypes.data)
    return _int(out)


def _values(rng, lib, count):
    """Directed values in fixed point over their whole range, its ends first."""
    top = math.floor(S_MAX * 2.0 ** lib.sig_frac())
    yield from (top, math.ceil(S_MIN * 2.0 ** lib.sig_frac()), 1 << lib.sig_frac(), 1)
    for _ in range(count):
        yield int(2.0 ** rng.uniform(math.log2(S_MIN), math.log2(S_MAX)) * 2.0 ** lib.sig_frac())


def test_small_values_keep_their_bits(lib):
    """Rounding a directed value to fixed point costs at most 2^-47 of it at any size (half a unit
    in the last place at the smallest value), so a small weight is as good as a large one."""
    rng = random.Random(1)
    for i in range(20000):
        x = (S_MIN, S_MAX)[i] if i < 2 else 2.0 ** rng.uniform(math.log2(S_MIN), math.log2(S_MAX))
        hi = np.float32(x)
        lo = np.float32(x - float(hi))
        exact = Fraction(float(hi)) + Fraction(float(lo))
        got = Fraction(lib.sig(hi, lo), 1 << lib.sig_frac())
        assert abs(got - exact) <= exact / 2 ** 47, (x, float(abs(got - exact) / exact))
    assert lib.sig(0.0, 0.0) == 0


def test_pair_products_are_exact_ones_rounded_down(lib):
    rng = random.Random(2)
    shift = 2 * lib.sig_frac() - lib.term_frac()
    xs = list(_values(rng, lib, 400))
    assert 2 * max(xs) <= M64                            # a pair sum fits a word
    for x in xs[:4] + rng.sample(xs, 60):
        for a, b in [(x, x)] + [tuple(rng.choices(xs, k=2)) for _ in range(40)]:
            p = _call(2, lib.pair, x, a + b)
            assert p == x * (a + b) >> shift and p < 1 << 85
            # what is dropped is lost in the last bit of a double
            if min(x, a, b) > S_MIN * 2.0 ** lib.sig_frac():
                assert x * (a + b) - (p << shift) <= Fraction(x * (a + b), 2 ** 52)


def test_sums_of_pairs(lib):
    """1,024 of the largest pairs fit the running sums, 128 of them the carry-free words."""
    rng = random.Random(3)
    shift = 2 * lib.sig_frac() - lib.term_frac()
    top = math.floor(S_MAX * 2.0 ** lib.sig_frac())
    xs = list(_values(rng, lib, 1020))
    for factors in ([(top, 2 * top)] * 1024, [(x, x + rng.choice(xs)) for x in xs]):
        pairs = [x * y >> shift for x, y in factors]
        a = np.zeros(2, np.uint64)
        for p in pairs:
            w = _words(p, 2)
            lib.add96(a.ctypes.data, w.ctypes.data)
        assert _int(a) == sum(pairs) < 1 << 96
        xy = np.array(factors, np.uint64)
        for m in (1, 127, 128):
            assert _call(2, lib.limb_sum, xy.ctypes.data, m) == sum(pairs[:m])


def test_scaling_is_exact(lib):
    rng = random.Random(4)
    for s in _values(rng, lib, 300):
        for p in (0, 1, (1 << 96) - 1, rng.randrange(1 << 96), rng.randrange(1 << 80)):
            w = _words(p, 2)
            assert _call(3, lib.scaled, s, w.ctypes.data) == s * p << (lib.acc_frac() - lib.sig_frac() - lib.term_frac())
    for v in ((1 << 116) - 1, 1, rng.randrange(1 << 116)):
        assert _call(3, lib.term192, v & M64, v >> 64) == v << (lib.acc_frac() - lib.term_frac())


@pytest.mark.parametrize("atomic", [0, 1])
def test_three_word_sums(lib, atomic):
    """Sums and differences modulo 2^192, carries through full words included."""
    rng = random.Random(5)
    edge = [0, 1, M64, M64 << 64, (1 << 128) - 1, (1 << 192) - 1, 1 << 128, 1 << 64]
    for trial in range(300):
        want, a = 0, np.zeros(3, np.uint64)
        for _ in range(20):
            v = rng.choice(edge) if rng.random() < 0.5 else rng.randrange(1 << rng.choice([60, 130, 190]))
            neg = rng.random() < 0.4
            w = _words(v, 3)
            lib.add192(a.ctypes.data, w.ctypes.data, int(neg), atomic)
            want = (want + (-v if neg else v)) % (1 << 192)
            assert _int(a) == want


def test_conversion_rounds_to_nearest(lib):
    """The double nearest to a sum, ties to even, whichever word decides."""
    rng = random.Random(6)
    one = 1 << lib.acc_frac()
    sums = [1, one, one - 1, (1 << 191) + 1]
    for bits in list(range(54, 193)) + [rng.randrange(54, 193) for _ in range(2000)]:
        m = rng.randrange(1 << 52, 1 << 53)
        half = (2 * m + 1) << (bits - 54)                # halfway between two doubles
        sums += [half, half + 1, half - 1, rng.randrange(1 << (bits - 1), 1 << bits), m << (bits - 53)]
    for v in sums:
        w = _words(v, 3)
        assert lib.to_double(w.ctypes.data) == v / one, hex(v)      # (a quotient of ints is correctly rounded)
