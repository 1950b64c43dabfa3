"""The even/odd products of field.cuh modelled limb by limb in Python integers (no GPU):
no chain drops a carry and every result is below 2N before its one conditional subtraction,
for f_mul (first operand below 2N, any 256-bit second operand where the first is below N),
f_mul2 (operands up to N), the whole product and square with their reduction, and the lazy
Fp2 products' full-width sums.  The GPU tests compare the kernels with the oracle."""
import itertools
import random

import pytest

from oracle import bn254 as bn

M32 = (1 << 32) - 1
R = 1 << 256


def limbs(x, n=8):
    return [(x >> (32 * i)) & M32 for i in range(n)]


def value(t, w=0):
    return sum(v << (32 * (i + w)) for i, v in enumerate(t))


def chain(t, at, xs, y, n=None, carry_to=None):
    """t[at..] += xs[0] y, xs[1] y, .. on limb pairs; the carry goes to limb carry_to, else
    there must be none."""
    n = len(xs)
    s = value(t[at:at + 2 * n]) + sum((x * y) << (64 * i) for i, x in enumerate(xs))
    t[at:at + 2 * n] = limbs(s, 2 * n)
    c = s >> (64 * n)
    if carry_to is None:
        assert c == 0
    else:
        t[carry_to] += c
        assert t[carry_to] <= M32


def rows(pairs, N, e=None, o=None):
    """sum a b over the pairs (a, b), divided by 2^256 mod N row by row; or, without pairs,
    the reduction of e + 2^32 o."""
    ninv = (-pow(N, -1, 1 << 32)) & M32
    n = limbs(N)
    e, o, pend = (e or [0] * 8), (o or [0] * 8), 0
    for i in range(8):
        s = e[0] + pend  # chain_p2: pend enters the even limb, its carry the odd chain
        e[0] = s & M32
        oc = value(o) + (s >> 32)
        assert oc < R
        o = limbs(oc)
        for a, b in pairs:
            chain(o, 0, limbs(a)[1::2], limbs(b)[i])
            chain_even(e, o, limbs(a)[0::2], limbs(b)[i])
        q = (e[0] * ninv) & M32
        chain(o, 0, n[1::2], q)
        chain_even(e, o, n[0::2], q)
        assert e[0] == 0
        pend, e, o = e[1], o, e[2:] + [0, 0]
    out = value(e) + value(o, 1) + pend
    assert out < R
    return out


def chain_even(e, o, xs, y):
    s = value(e) + sum((x * y) << (64 * i) for i, x in enumerate(xs))
    e[:] = limbs(s)
    o[7] += s >> 256
    assert o[7] <= M32


def wide(a, b):
    """mul_wide's chains: (e[0..15], o[0..14])."""
    A, B = limbs(a), limbs(b)
    e, o = [0] * 17, [0] * 16
    for i in range(8):
        same, other = A[i % 2::2], A[1 - i % 2::2]
        if i % 2:
            chain(e, i + 1, same, B[i])
            chain(o, i - 1, other, B[i], carry_to=i + 7)
        elif i == 0:
            chain(e, 0, same, B[0])
            chain(o, 0, other, B[0])
        else:
            chain(e, i, same, B[i], carry_to=i + 8)
            chain(o, i, other, B[i])
    return e[:16], o[:15]


def wide_sqr(a):
    """sqr_wide's chains over the doubled limbs."""
    A = limbs(a)
    d = [0] + [((A[j] << 1) | (A[j - 1] >> 31)) & M32 for j in range(1, 8)]
    s = [(x << 1) & M32 for x in A]
    assert A[7] >> 31 == 0
    e, o = [0] * 16, [0] * 15
    chain(o, 0, [s[1], d[3], d[5], d[7]], A[0])
    chain(e, 2, [d[2], d[4], d[6]], A[0])
    for i in range(1, 7):
        odd, even = [s[i + 1]] + d[i + 3::2], d[i + 2::2]
        # rows of odd i hand the odd chain's carry on, rows of even i the even chain's
        chain(o, 2 * i, odd, A[i], carry_to=2 * i + 2 * len(odd) if i % 2 else None)
        if even:
            chain(e, 2 * i + 2, even, A[i], carry_to=None if i % 2 else 2 * i + 2 + 2 * len(even))
    chain(e, 0, A, 0)
    t = value(e) + sum((x * x) << (64 * i) for i, x in enumerate(A))
    assert t < 1 << 512
    return limbs(t, 16), o


def redc(e, o, N):
    top = value(e[8:16]) + value(o[7:15])
    assert top < R
    r = rows([], N, e[:8], o[:7] + [0]) + top
    assert r < 2 * N
    return r


def edge(N, rng, upto):
    near = [0, 1, 2, N - 1, N - 2, N >> 1, (1 << 253) - 1, M32, R - N, (1 << 224) - 1, ((1 << 254) - 1) ^ M32]
    vals = [v for v in near + [N, 2 * N - 1, 2 * N - 2, R - 1, R - 2] if v < upto]
    return vals + [rng.randrange(upto) for _ in range(20)]


@pytest.mark.parametrize("N", [bn.P, bn.R])
def test_products(N):
    rng = random.Random(11)
    ri = pow(R, -1, N)
    for amax, bmax in ((2 * N, 2 * N), (N, R)):  # the two operand ranges of f_mul
        for a, b in itertools.product(edge(N, rng, amax), edge(N, rng, bmax)):
            r = rows([(a, b)], N)
            assert r < 2 * N and (r - a * b * ri) % N == 0
    vals = edge(N, rng, N + 1)
    for a, b in itertools.product(vals, vals):
        c, d = rng.choice(vals), rng.choice(vals)
        r = rows([(a, b), (c, d)], N)
        assert r < 2 * N and (r - (a * b + c * d) * ri) % N == 0


@pytest.mark.parametrize("N", [bn.P, bn.R])
def test_wide_products_squares_and_reduction(N):
    rng = random.Random(12)
    vals = edge(N, rng, N + 1)
    for a, b in itertools.product(vals, vals):
        e, o = wide(a, b)
        assert value(e) + value(o, 1) == a * b
    for a, b in itertools.product(edge(N, rng, 2 * N), repeat=2):  # Karatsuba's unreduced sums
        e, o = wide(a, b)
        assert value(e) + value(o, 1) == a * b
    for a in vals + [rng.randrange(N) for _ in range(300)]:
        e, o = wide_sqr(a)
        assert value(e) + value(o, 1) == a * a
        assert (redc(e, o, N) - a * a * pow(R, -1, N)) % N == 0


def test_fp2_lazy_sums():
    """re = a0 b0 - a1 b1 (+ c0 d0 - c1 d1), made positive by N R, and im stay below N R, the
    range of the reduction; the sign is limb 15's top bit."""
    N, rng = bn.P, random.Random(13)
    vals = edge(N, rng, N + 1)
    for _ in range(4000):
        a0, a1, b0, b1, c0, c1, d0, d1 = (rng.choice(vals) for _ in range(8))
        im = (a0 + a1) * (b0 + b1) - a0 * b0 - a1 * b1 + (c0 + c1) * (d0 + d1) - c0 * d0 - c1 * d1
        assert 0 <= im < N * R
        re = a0 * b0 - a1 * b1 + c0 * d0 - c1 * d1
        assert (re % (1 << 512)) >> 511 == (1 if re < 0 else 0)
        re += N * R if re < 0 else 0
        assert 0 <= re < N * R
        t = limbs(re, 16)
        r = rows([], N, t[:8], [0] * 8) + value(t[8:])
        assert r < 2 * N and (r - re * pow(R, -1, N)) % N == 0
