"""The Montgomery products of Fq and Fr (`mp::mont_mul` in fp.cuh), compiled for the host and checked
against Python integers: a b 2^(-32 n) mod m for a < m and any b of n words (the operand that may
not be reduced), at the values where its carries run furthest (no GPU)."""
import ctypes
import os
import random
import shutil
import subprocess

import pytest

from tests import _pyref as ref

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2601_03031_gb300", "csrc")


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    gxx = shutil.which("g++")
    if not gxx:
        pytest.skip("g++ not available")
    so = str(tmp_path_factory.mktemp("emu_mul") / "libmul.so")
    subprocess.check_call([gxx, "-std=c++20", "-O1", "-shared", "-fPIC", f"-I{CSRC}", "-o", so,
                           os.path.join(HERE, "emu", "product.cpp")])
    L = ctypes.CDLL(so)
    L.emu_fq_mul.restype = L.emu_fr_mul.restype = None
    return L


@pytest.mark.parametrize("field", ["fq", "fr"])
def test_product_against_python(lib, field):
    m, n, fn = (ref.P, 12, lib.emu_fq_mul) if field == "fq" else (ref.R, 8, lib.emu_fr_mul)
    top = 1 << (32 * n)
    rnd = random.Random(29)
    ones = [(1 << (32 * k)) - 1 for k in range(1, n)]
    alt = sum(0xFFFFFFFF << (64 * k) for k in range(n // 2))
    avals = [0, 1, m - 1, m - 2, m >> 1, *ones, alt % m] + [rnd.randrange(m) for _ in range(30)]
    bvals = [0, 1, m - 1, m, m + 1, top - 1, top - m, alt, (alt << 32) % top, *ones] + \
            [rnd.randrange(top) for _ in range(30)]
    rinv = pow(top, -1, m)

    def words(x):
        return (ctypes.c_uint32 * n)(*[(x >> (32 * i)) & 0xFFFFFFFF for i in range(n)])

    out = (ctypes.c_uint32 * n)()
    for a in avals:
        for b in bvals:
            fn(words(a), words(b), out)
            assert sum(out[i] << (32 * i) for i in range(n)) == a * b * rinv % m, (hex(a), hex(b))
