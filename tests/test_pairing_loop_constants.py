"""What the GPU Miller loop's subgroup test and reductions rely on (no GPU needed)."""
from math import gcd

from oracle import bn254 as bn

U, P, R = bn.U, bn.P, bn.R
T = 6 * U * U + 1  # trace of Frobenius


def _naf(n):
    out = []
    while n:
        z = 2 - (n & 3) if n & 1 else 0
        out.append(z)
        n = (n - z) >> 1
    return out


def test_subgroup_equation():
    """[6u+2]Q + pi(Q) - pi^2(Q) + pi^3(Q) = O on the twist holds exactly for [r]Q = O.  With
    pi^2 - t pi + p = 0 the left side is (a pi + b)Q; its norm is a multiple of r whose
    cofactor is prime to the twist's order r (2p - r), so the equation forces [r]Q = O; and pi
    acts on the points of order r as p mod r, which is a root of X^3 - X^2 + X + 6u + 2."""
    assert P + 1 - T == R
    a, b = (T * T - P) - T + 1, -T * P + P + 6 * U + 2
    norm = b * b + a * b * T + a * a * P
    assert norm % R == 0 and gcd(norm // R, R * (2 * P - R)) == 1
    lam = P % R
    assert (lam ** 3 - lam ** 2 + lam + 6 * U + 2) % R == 0 and (lam * lam - T * lam + P) % R == 0
    # the twist's order: [r (2p - r)] kills a point outside the subgroup, [r] and [2p - r] do not
    x = (1, 0)
    while True:
        y = _sqrt(bn.f2_add(bn.f2_mul(bn.f2_mul(x, x), x), bn.B2))
        if y is not None:
            Q = (x, y)
            if bn.g2_mul_noshortcut(Q, R) is not None:
                break
        x = (x[0] + 1, 0)
    S = bn.g2_mul_noshortcut(Q, R)
    assert bn.g2_mul_noshortcut(S, 2 * P - R) is None


def _sqrt(a):
    """a square root in Fp2 or None (p = 3 mod 4, complex method)."""
    n = (a[0] * a[0] + a[1] * a[1]) % P
    s = pow(n, (P + 1) // 4, P)
    if s * s % P != n:
        return None
    for h in ((a[0] + s) * pow(2, -1, P) % P, (a[0] - s) * pow(2, -1, P) % P):
        c = pow(h, (P + 1) // 4, P)
        if c and c * c % P == h:
            r = (c, a[1] * pow(2 * c, -1, P) % P)
            if bn.f2_mul(r, r) == (a[0] % P, a[1] % P):
                return r
    return None


def test_signed_digits():
    """6u + 2 in 66 signed digits, 22 of them nonzero; u in 63, 24 nonzero; no prefix of the
    loop scalar is 0 or +-1 modulo r when Q is added, and the closing multiples differ."""
    for n, length, weight in ((6 * U + 2, 66, 22), (U, 63, 24)):
        d = _naf(n)
        assert len(d) == length and sum(1 for z in d if z) == weight and sum(z << i for i, z in enumerate(d)) == n
    k = 1
    for z in reversed(_naf(6 * U + 2)[:-1]):
        k *= 2
        if z:
            assert k % R not in (0, 1, R - 1)
            k += z
    assert k == 6 * U + 2
    lam = P % R
    assert k % R not in (lam, R - lam) and (k + lam) % R not in (lam * lam % R, -lam * lam % R)


def test_quotient_estimate():
    """f_mod9: for t < 64 p the quotient from t / 2^240 and 2^32 / 12389 is exact or one short."""
    import random
    rng = random.Random(3)
    for _ in range(20000):
        t = rng.choice([rng.randrange(64 * P), rng.randrange(64) * P + rng.randrange(-3, 4)])
        if 0 <= t < 64 * P:
            q = ((t >> 240) * 346675) >> 32
            assert t >> 240 < 1 << 20 and 0 <= t - q * P < 2 * P
