"""The integer arithmetic of the FP64 kernels, compiled for the host: the sums of
csrc/reduce.cuh against exact rational sums."""
import ctypes
import math
import random
import subprocess
from fractions import Fraction

import numpy as np
import pytest

SOURCE = r"""
#include "reduce.cuh"
using namespace wl;
static unsigned long long bits(double v) { unsigned long long u; memcpy(&u, &v, 8); return u; }
// block_sum_of over n values
extern "C" double host_sum(const double* v, int n) {
    unsigned m = 0, l[3] = {0, 0, 0};
    for (int i = 0; i < n; i++) m = max(m, (unsigned)(bits(v[i]) >> 32));
    const int e = (int)(m >> 20);
    for (int i = 0; i < n; i++) {
        const unsigned long long t = sum_term((unsigned)(bits(v[i]) >> 32), (unsigned)bits(v[i]), e);
        l[0] += (unsigned)t & 0x1FFFFFu;
        l[1] += (unsigned)(t >> 21) & 0x1FFFFFu;
        l[2] += (unsigned)(t >> 42);
    }
    const unsigned long long s = sum_bits(l[2], l[1], l[0], e);
    double r;
    memcpy(&r, &s, 8);
    return r;
}
"""


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    from paper_0710_2442_gb300 import build
    d = tmp_path_factory.mktemp("fixed_point")
    src, lib = d / "host.cu", d / "host.so"
    src.write_text("#include <cstring>\n" + SOURCE)
    subprocess.run([build.nvcc(), *build.ARCH, "-O1", "-std=c++17", "--expt-relaxed-constexpr", "-Xcompiler", "-fPIC",
                    "-I", build.CSRC, "-shared", "-cudart", "static", str(src), "-o", str(lib)], check=True)
    h = ctypes.CDLL(str(lib))
    h.host_sum.restype = ctypes.c_double
    return h


def block_sum(host, v):
    a = np.asarray(v, dtype=np.float64)
    return host.host_sum(a.ctypes.data_as(ctypes.c_void_p), len(a))


@pytest.mark.parametrize("n", [1, 2, 3, 8, 64, 256, 2048])
def test_block_sum_error(host, n):
    """Half a unit in the last place of the sum, and 2^-62 of the largest term's scale (less than
    twice the term) for each term below 2^-9 of it; a term alone comes back as it is."""
    rng = random.Random(n)
    for spread in (0, 3, 12, 40):
        for _ in range(20 if n > 256 else 200):
            v = [rng.uniform(1.0, 2.0) * 2.0 ** -rng.uniform(0, spread) for _ in range(n)]
            if n > 2 and rng.random() < 0.3:
                v[rng.randrange(n)] = 0.0
            got, exact = Fraction(block_sum(host, v)), sum(map(Fraction, v))
            small = sum(1 for x in v if x < max(v) * 2.0 ** -8)
            assert abs(got - exact) <= Fraction(math.ulp(float(exact))) / 2 + small * Fraction(max(v)) / 2 ** 61
            if n == 1:
                assert got == exact


def test_block_sum_edges(host):
    assert block_sum(host, [2.0 ** 1023, 2.0 ** 1023]) == math.inf
    assert block_sum(host, [np.finfo(np.float64).max]) == np.finfo(np.float64).max
    assert block_sum(host, [np.finfo(np.float64).max] * 2048) == math.inf
    assert block_sum(host, [1.0, 2.0 ** -53]) == 1.0 and block_sum(host, [1.0 + 2.0 ** -52, 2.0 ** -53]) == 1.0 + 2.0 ** -51
    assert block_sum(host, [2.0 - 2.0 ** -52] * 2048) == 2048 * (2.0 - 2.0 ** -52)
    assert block_sum(host, [2.0 ** -895] * 3) == 3 * 2.0 ** -895  # exponent field 128, the smallest taken
    assert block_sum(host, [1.0, 5e-324, 0.0]) == 1.0
