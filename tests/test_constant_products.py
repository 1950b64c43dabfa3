"""The products by twiddles of field.cuh (f_mul_const) modelled limb by limb in Python
integers (no GPU): the quotient from the columns 6 .. 14 alone, the low halves modulo 2^256
and the bound below 2N for operands below 4N; and the table's quotients found by reduction
from the Montgomery form.  The GPU transforms are compared with the oracle."""
import random

import pytest

from oracle import bn254 as bn

M32 = (1 << 32) - 1
R256 = 1 << 256
N = bn.R


def limbs(x):
    return [(x >> (32 * i)) & M32 for i in range(8)]


def table_quotient(w):
    """floor(w 2^256 / N) by eight reduction steps on the Montgomery form of w."""
    t, q = w * R256 % N, 0
    inv = (-pow(N, -1, 1 << 32)) & M32
    for i in range(8):
        qi = ((t >> (32 * i)) & M32) * inv & M32
        t += qi * N << (32 * i)
        q |= qi << (32 * i)
    assert t % R256 == 0
    return q


def mul_const(x, w, wq):
    q = sum(a * b << (32 * (i + j)) for i, b in enumerate(limbs(wq)) for j, a in enumerate(limbs(x)) if i + j >= 6) >> 256
    low = sum(a * b << (32 * (i + j)) for i, b in enumerate(limbs(w)) for j, a in enumerate(limbs(x)) if i + j <= 7)
    low += sum(a * b << (32 * (i + j)) for i, b in enumerate(limbs(q)) for j, a in enumerate(limbs(R256 - N)) if i + j <= 7)
    return low % R256


rng = random.Random(7)
WS = [0, 1, 2, N - 1, N - 2, N // 2, (1 << 224) - 1, 1 << 224] + [rng.randrange(N) for _ in range(40)]
XS = [0, 1, N - 1, N, 2 * N - 1, 2 * N, 4 * N - 1, (1 << 192) - 1, 1 << 192] + [rng.randrange(4 * N) for _ in range(40)]


@pytest.mark.parametrize("w", WS)
def test_quotient_and_product(w):
    wq = table_quotient(w)
    assert wq == w * R256 // N
    for x in XS:
        r = mul_const(x, w, wq)
        assert r < 2 * N and r % N == x * w % N
