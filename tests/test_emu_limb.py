"""The limb-lane engine (limb.cuh: Fq sums of products with one limb per lane; limb12.cuh: Fq12
operations on it), compiled for the host with every lane as a thread, against Python integers and the
oracle (no GPU)."""
import ctypes
import os
import random
import shutil
import subprocess

import pytest

import oracle as O
from tests import _pyref as ref

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2601_03031_gb300", "csrc")


@pytest.fixture(scope="module")
def emu(tmp_path_factory):
    gxx = shutil.which("g++")
    if not gxx:
        pytest.skip("g++ not available")
    so = str(tmp_path_factory.mktemp("emu_limb") / "liblimb.so")
    subprocess.check_call([gxx, "-std=c++20", "-O1", "-shared", "-fPIC", f"-I{CSRC}", "-o", so,
                           os.path.join(HERE, "emu", "limb.cpp")])
    L = ctypes.CDLL(so)
    for f in (L.emu_limb_dot3, L.emu_limb_final_exp, L.emu_limb_g1_mul, L.emu_limb_g2_mul_add, L.emu_limb_g1_mul_add, L.emu_limb_miller):
        f.restype = None
    return L


def test_sum_of_products_against_python(emu):
    """x0 y0 + x1 y1 + x2 y2 times 2^-390 mod p, at values with all limbs at their largest, zero and
    random ones."""
    P = ref.P
    rnd = random.Random(3)
    vals = [0, 1, P - 1, (1 << 380) - 1, (1 << 338) - 1, 1 << 338, P >> 1]
    cases = [[(a, b)] * 3 for a in vals for b in vals[1:4]]
    cases += [[(rnd.randrange(P), rnd.randrange(P)) for _ in range(3)] for _ in range(20)]
    out = (ctypes.c_uint32 * 12)()
    for c in cases:
        x, y = [(ctypes.c_uint32 * 36)(*[(t[i] >> (32 * j)) & 0xFFFFFFFF for t in c for j in range(12)])
                for i in (0, 1)]
        emu.emu_limb_dot3(x, y, out)
        want = sum(a * b for a, b in c) * pow(2, -390, P) % P
        assert sum(out[j] << (32 * j) for j in range(12)) == want, c


def test_final_exponentiation_against_oracle(emu):
    rnd = random.Random(8)
    for n in range(2):
        f = b"".join(rnd.randrange(ref.P).to_bytes(48, "big") for _ in range(12))
        if n:
            f = (1).to_bytes(48, "big") + bytes(528)
        out = ctypes.create_string_buffer(576)
        emu.emu_limb_final_exp(f, out)
        assert out.raw == O.final_exp(f)


def test_g1_scalar_mul_against_oracle(emu):
    """k P for edge and random k (digits that carry past bit 127 of a GLV half among them), and the
    identity."""
    rnd = random.Random(5)
    r, x2 = ref.R, 0xD201000000010000 ** 2
    ks = [0, 1, 2, 7, 8, 15, r - 1, x2, x2 - 1, x2 + 1, (x2 - 1) * (x2 + 1), r // 2] + [rnd.randrange(r) for _ in range(3)]
    P = O.g1_mul(O.g1_gen(), 12345)
    out = ctypes.create_string_buffer(96)
    for k in ks:
        for pt in (P, bytes(96)) if k == 7 else (P,):
            emu.emu_limb_g1_mul(pt, (ctypes.c_uint32 * 8)(*[((k % r) >> (32 * i)) & 0xFFFFFFFF for i in range(8)]), out)
            assert out.raw == O.g1_mul(pt, k % r), hex(k)


@pytest.mark.parametrize("pre", [0, 1])
def test_g2_scalar_mul_and_add_against_oracle(emu, pre):
    """k P + Q, directly and from tables of P's shifts, for edge and random k, with P = Q, P = -Q sums and identities among them."""
    rnd = random.Random(6)
    r, x = ref.R, 0xD201000000010000
    P = O.g2_mul(O.g2_gen(), 777)
    Q = O.g2_mul(O.g2_gen(), 4242)
    inf = bytes(192)
    cases = [(P, 0, Q), (P, 1, P), (P, r - 1, P), (P, 8, inf), (inf, 5, Q), (inf, 3, inf), (P, x, Q), (P, x - 1, Q),
             (P, x**3 + x**2 - 1, Q)] + [(P, rnd.randrange(r), Q) for _ in range(2)]
    out = ctypes.create_string_buffer(192)
    for p, k, q in cases:
        emu.emu_limb_g2_mul_add(pre, p, (ctypes.c_uint32 * 8)(*[(k >> (32 * i)) & 0xFFFFFFFF for i in range(8)]), q, out)
        assert out.raw == O.g2_add(O.g2_mul(p, k), q), hex(k)


@pytest.mark.parametrize("pre", [0, 1])
def test_g1_scalar_mul_and_add_against_oracle(emu, pre):
    rnd = random.Random(7)
    r = ref.R
    P, Q, inf = O.g1_mul(O.g1_gen(), 777), O.g1_mul(O.g1_gen(), 4242), bytes(96)
    x2 = 0xD201000000010000 ** 2
    cases = [(P, 0, Q), (P, 1, P), (P, r - 1, P), (P, 8, inf), (inf, 5, Q), (inf, 3, inf), (P, x2 - 1, Q),
             (P, (1 << 96) - 1, Q), (P, rnd.randrange(r), Q)]
    out = ctypes.create_string_buffer(96)
    for p, k, q in cases:
        emu.emu_limb_g1_mul_add(pre, p, (ctypes.c_uint32 * 8)(*[(k >> (32 * i)) & 0xFFFFFFFF for i in range(8)]), q, out)
        assert out.raw == O.g1_add(O.g1_mul(p, k), q), hex(k)


def test_miller_loop_against_oracle(emu):
    """The final exponentiation of the Miller value is the pairing (line scalings vanish under it); an
    identity on either side gives 1."""
    rnd = random.Random(9)
    out = ctypes.create_string_buffer(576)
    for _ in range(2):
        P, Q = O.g1_mul(O.g1_gen(), rnd.randrange(1, ref.R)), O.g2_mul(O.g2_gen(), rnd.randrange(1, ref.R))
        emu.emu_limb_miller(P, Q, out)
        assert O.final_exp(out.raw) == O.pairing(P, Q)
    one = (1).to_bytes(48, "big") + bytes(528)
    for p, q in ((bytes(96), Q), (P, bytes(192))):
        emu.emu_limb_miller(p, q, out)
        assert out.raw == one
