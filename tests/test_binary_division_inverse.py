"""The inversion of field.cuh modelled in Python integers (no GPU): batches of 30 halvings of
a binary division on low words, the exact update of (f, g) on complements with its
corrections, and the update of (d, e) modulo N.  Row sums stay within 2^30, f and g within
[-N, N], d and e within 3N/2, every 64-bit term in range, and d ends as the inverse within the
batch limit.  On the GPU the same values go through the elementwise inverse."""
import random

import pytest

from oracle import bn254 as bn

M32, M256, M288 = (1 << 32) - 1, (1 << 256) - 1, (1 << 288) - 1
BATCH, LIMIT = 30, 30


def low_bits_batch(due, f, g):
    fa, fb, ga, gb, left = 1, 0, 0, 1, BATCH
    while True:
        z = min((g & -g).bit_length() - 1 if g else 32, left)
        g, fa, fb, left, due = g >> z, fa << z, fb << z, left - z, due + z
        if left == 0:
            return due, *((a, b) if a >= 0 else (-a, -b) for a, b in ((fa, fb), (ga, gb)))
        if due > 0:
            f, g, fa, fb, ga, gb, due = g, f, ga, gb, fa, fb, -due
        want = 1 - due
        bits = min(want, left, 5)
        w = -g * (3 * f ^ 2) & ((1 << bits) - 1)
        if bits == want and w >> (bits - 1):
            w -= 1 << bits
        g, ga, gb = (g + f * w) & M32, ga + fa * w, gb + fb * w
        assert g & ((1 << bits) - 1) == 0
        assert max(abs(fa) + abs(fb), abs(ga) + abs(gb)) <= 1 << BATCH


def combine(x, a, y, b):
    """(a x + b y) / 2^30 as field.cuh forms it from the 256-bit patterns of x and y."""
    s, m = -1 if b < 0 else 0, abs(b)
    X, Y = x & M256, (y & M256) ^ (s & M256)
    assert a >= 0 and all((X >> j & M32) * a + (Y >> j & M32) * m + m < 1 << 63 for j in range(0, 256, 32))
    high = (a & (-1 if x < 0 else 0)) + (m & ((-1 if y < 0 else 0) ^ s))
    t = (X * a + Y * m + (m & s) - (high << 256)) & M288
    t -= (t >> 287) << 288
    assert t == a * x + b * y and t % (1 << BATCH) == 0
    return t >> BATCH


def combine_mod(x, a, y, b, N):
    assert 0 <= 2 * x <= 3 * N and 0 <= 2 * y <= 3 * N and a >= 0
    t = a * x + abs(b) * (2 * N - y if b < 0 else y)
    t += (t * pow(-N, -1, 1 << 32) & M32) * N
    assert t & M32 == 0
    return t >> 32


def inverse(y, N):
    f, g, d, e, due = N, y, 0, (1 << 768) % N, 0
    for n in range(1, LIMIT + 1):
        due, rf, rg = low_bits_batch(due, f & M32, g & M32)
        f, g = combine(f, rf[0], g, rf[1]), combine(f, rg[0], g, rg[1])
        assert abs(f) <= N and abs(g) <= N
        d, e = combine_mod(d, rf[0], e, rf[1], N), combine_mod(d, rg[0], e, rg[1], N)
        if g == 0:
            break
    assert g == 0 and abs(f) == 1
    return f * d * (1 << (2 * n)) * pow(1 << 256, -1, N) % N, n


def test_inverse_modulo_32():
    assert all(f * (3 * f ^ 2) % 32 == 1 for f in range(1, 1 << 12, 2))


def values(N):
    rng = random.Random(7)
    vals = [1, 2, 3, N - 1, N - 2, (N - 1) // 2, (N + 1) // 2, (1 << 253) - 1, (1 << 30) - 1, 1 << 30, (1 << 32) + 1]
    vals += [1 << k for k in range(253)] + [(1 << k) - 1 for k in range(1, 253, 5)]
    vals += [rng.randrange(1, N) for _ in range(1500)] + [rng.randrange(1, 1 << rng.randrange(1, 253)) for _ in range(300)]
    # quotients +-1 after single halvings, as far as 253 bits decide them: the remainders that
    # shrink most slowly (ratio of neighbours rho = 2 / (2 rho' - q) modulo a power of two)
    for signs in ([1] * 130, [-1] * 130, [1, -1] * 65, [rng.choice((1, -1)) for _ in range(130)]):
        rho = 0
        for q in signs:
            rho = 2 * pow(2 * rho - q, -1, 1 << 260) % (1 << 260)
        vals.append(N * rho % (1 << 253))
    return vals


@pytest.mark.parametrize("N", [bn.P, bn.R], ids=["p", "r"])
def test_binary_division_inverse(N):
    worst = 0
    for y in values(N):
        x, batches = inverse(y, N)
        assert x * y % N == (1 << 512) % N
        worst = max(worst, batches)
    assert worst <= 28


@pytest.mark.gpu
@pytest.mark.parametrize("name,N", [("fp", bn.P), ("fr", bn.R)])
def test_device_inverse(name, N):
    import torch
    from tests import _util
    assert torch.cuda.is_available()
    nv = _util.native()
    back = pow(1 << 256, -1, N)  # the device inverts the Montgomery form y = a 2^256
    a = [y * back % N for y in values(N)]
    got = _util.u8_to_ints(getattr(nv, f"zkvc_{name}_inv")(_util.to_cuda(_util.ints_to_u8(a))).cpu().numpy())
    assert got == [pow(x, -1, N) for x in a]
