"""Blocks of the FP64-class product (csrc/crt_gemm.cu) against its scratch: what
every block lays out, counted here from the documented layout, fits, for any
shape and any scratch down to the least one; and its K splits against the words
of the reconstruction.  No device."""
import ctypes
import math
import random

import pytest

MODULI = 16


@pytest.fixture(scope="module")
def lib():
    from paper_1810_08142_gb300 import build
    return ctypes.CDLL(build.build())


def up(x, to):
    return (x + to - 1) // to * to


def block_need(m, n, k):
    """Residues (2 bytes) and exponents of both operands, one byte per modulus, row and padded column."""
    kp = up(k, 8)
    return sum(up(MODULI * r * kp * 2, 256) + up(4 * r, 256) for r in (m, n)) + MODULI * m * up(n, 16)


def blocks(lib, m, n, k, scratch, sms=152):
    f = getattr(lib, "_ZN6ladder15crt_gemm_blocksExxximRA3_x")
    f.restype = ctypes.c_bool
    f.argtypes = [ctypes.c_longlong] * 3 + [ctypes.c_int, ctypes.c_size_t, ctypes.POINTER(ctypes.c_longlong * 3)]
    out = (ctypes.c_longlong * 3)()
    return list(out) if f(m, n, k, sms, scratch, ctypes.byref(out)) else None


def check(lib, m, n, k, scratch):
    b = blocks(lib, m, n, k, scratch)
    assert b is not None, (m, n, k, scratch)
    for x, whole, step in zip(b, (m, n, k), (128, 16, 64)):
        assert 0 < x <= whole and (x == whole or x % step == 0)
    # the full blocks and the last ones of every direction
    tails = [(x, (whole - 1) % x + 1) for x, whole in zip(b, (m, n, k))]
    for mm in tails[0]:
        for nn in tails[1]:
            for kk in tails[2]:
                assert block_need(mm, nn, kk) <= scratch, (m, n, k, scratch, b)


# the (kc|ld) product of a dressed ladder, m = n = o v, in 1 GiB of scratch
@pytest.mark.parametrize("o,v,n", [(20, 406, 1380), (26, 319, 1276), (15, 447, 2155), (17, 417, 1950), (34, 259, 1036),
                                   (23, 362, 1267)])
def test_rows_halved_below_the_columns(lib, o, v, n):
    check(lib, o * v, o * v, n, 1 << 30)


def test_every_scratch_down_to_the_least(lib):
    rng = random.Random(1)
    least = block_need(128, 16, 8192)
    for _ in range(4000):
        m, n = sorted((int(2 ** rng.uniform(0, 17)), int(2 ** rng.uniform(0, 17))), reverse=True)
        check(lib, m, n, int(2 ** rng.uniform(0, 21)), int(least * 2 ** rng.uniform(0, 8)) + 256)
    assert blocks(lib, 128, 16, 8192, least - 256) is None


def test_long_contractions_run_in_even_blocks(lib):
    """At most 2^17 terms a block, which leaves 53 bits to the operands."""
    for k in (1 << 17, (1 << 17) + 1, 300000, 1 << 20, (1 << 30) - 1):
        kb = blocks(lib, 1, 1, k, 1 << 40)[2]
        assert kb <= 1 << 17 and -(-k // kb) == -(-k // (1 << 17)) and min(58, (123 - (kb - 1).bit_length()) // 2) >= 53


def test_splits_fit_the_reconstruction(lib):
    """Residues of all K splits are summed before the reconstruction, which adds (sum of three moduli's) x (M / the
    three) in 32-bit words held in 64 bits: no word may wrap at the most splits that any K and any GPU get."""
    f = getattr(lib, "_ZN6ladder14crt_gemm_bytesExxxi")
    f.restype, f.argtypes = ctypes.c_size_t, [ctypes.c_longlong] * 3 + [ctypes.c_int]
    operands = block_need(1, 1, 1 << 17) - MODULI * 16
    splits = (f(1, 1, 1 << 17, 1 << 20) - operands) // (MODULI * 16)
    assert (f(1, 1, 64, 1 << 20) - (block_need(1, 1, 64) - MODULI * 16)) // (MODULI * 16) == 1 < splits
    p = [256, 255, 253, 251, 247, 241, 239, 233, 229, 227, 223, 217, 211, 199, 197, 193]
    threes = [(0, 1, 2), (4, 5, 6), (8, 9, 10), (12, 13, 14), (3, 7, 11), (15,)]
    for word in range(4):
        total = 1 << 32  # carry
        for t in threes:
            q = math.prod(p[i] for i in t)
            most = splits * sum((q // p[i]) * (p[i] - 1) for i in t)
            assert most < 1 << 32
            total += most * ((math.prod(p) // q >> (32 * word)) & 0xffffffff)
        assert total < 1 << 64
