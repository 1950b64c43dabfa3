"""The divstep inversion of field.cuh modelled in Python integers (no GPU): batches of 30
steps on the low 32 bits, several steps per round, with the exact and modular updates on
signed 30-bit limbs.  Every matrix entry stays within 2^30, (d, e) within (-2N, N), every
64-bit accumulator in range, at most 25 batches are needed and d ends as the inverse."""
import random

import pytest

from oracle import bn254 as bn

M30, M32 = (1 << 30) - 1, (1 << 32) - 1


def s32(x):
    x &= M32
    return x - (1 << 32) if x >> 31 else x


def divsteps30(eta, f, g):
    u, v, q, r, i = 1, 0, 0, 1, 30
    while True:
        x = g | (M32 << i) & M32
        z = (x & -x).bit_length() - 1
        g, u, v, eta, i = g >> z, u << z & M32, v << z & M32, eta - z, i - z
        if i == 0:
            return eta, [s32(t) for t in (u, v, q, r)]
        if eta < 0:
            eta, f, g, u, q, v, r = -eta, g, -f & M32, q, -u & M32, r, -v & M32
        lim = min(eta + 1, i, 6)
        w = f * g * (f * f - 2) & M32 & ((1 << lim) - 1)
        g, q, r = (g + f * w) & M32, (q + u * w) & M32, (r + v * w) & M32
        assert g & ((1 << lim) - 1) == 0


def limbs30(x):
    out = [(x >> (30 * i)) & M30 for i in range(8)]
    return out + [x >> 240]


def accumulate(rows):
    """sum of coefficient times number, limb by limb with arithmetic shifts, over 2^30."""
    c, out = 0, []
    for i in range(9):
        for k, x in rows:
            assert -(1 << 31) <= k < 1 << 31
            c += k * x[i]
            assert -(1 << 63) <= c < 1 << 63
        if i == 0:
            assert c & M30 == 0
        else:
            out.append(c & M30)
        c >>= 30
    assert -(1 << 31) <= c < 1 << 31
    return sum(v << (30 * i) for i, v in enumerate(out)) + (c << 240)


def inverse(y, N):
    f, g, d, e, eta = N, y, 0, (1 << 512) % N, -1
    ninv = pow(N, -1, 1 << 30)
    for batch in range(1, 26):
        eta, (u, v, q, r) = divsteps30(eta, f & M32, g & M32)
        assert max(abs(u) + abs(v), abs(q) + abs(r)) <= 1 << 30
        new = []
        for a, b in ((u, v), (q, r)):
            m = (a if d < 0 else 0) + (b if e < 0 else 0)
            m -= (ninv * (a * (d & M30) + b * (e & M30)) + m) & M30
            new.append(accumulate([(a, limbs30(d)), (b, limbs30(e)), (m, limbs30(N))]))
        d, e = new
        assert -2 * N < d < N and -2 * N < e < N
        f, g = accumulate([(u, limbs30(f)), (v, limbs30(g))]), accumulate([(q, limbs30(f)), (r, limbs30(g))])
        if g == 0:
            break
    assert g == 0 and abs(f) == 1
    x = d + N if d < 0 else d
    x = -x if f < 0 else x
    return (x + N if x < 0 else x), batch


@pytest.mark.parametrize("N", [bn.P, bn.R])
def test_divstep_inverse(N):
    rng = random.Random(5)
    vals = [1, 2, 3, N - 1, N - 2, (N - 1) // 2, (1 << 253) - 1, (1 << 30) - 1, 1 << 30, 1 << 252]
    vals += [1 << k for k in range(0, 253, 7)] + [rng.randrange(1, N) for _ in range(1500)]
    vals += [rng.randrange(1, 1 << rng.randrange(1, 253)) for _ in range(300)]
    worst = 0
    for y in vals:
        x, batches = inverse(y, N)
        assert 0 <= x < N and x * y % N == (1 << 512) % N
        worst = max(worst, batches)
    assert worst <= 25
