"""GPU verification on statements built from known discrete logs (a verifying key of chosen
exponents, C solved from the pairing equation), which isolate what honest proofs cannot:

* B's subgroup alone: with A at infinity the equation holds for every B, so the verdict is the
  subgroup test's -- B of order r and at infinity, B outside the subgroup, of each small order
  that the twist has, and a point of order r plus one of those;
* the merged sum of the public inputs through the pairwise affine rounds with a base array per
  output: keys whose points repeat, cancel or lie at infinity, inputs that put every term into
  a few buckets."""
import random

import numpy as np
import pytest

from oracle import bn254 as bn
from tests import _util
from tests.test_gpu_verify import _twist_point_off_subgroup

pytestmark = pytest.mark.gpu

COFACTOR = 2 * bn.P - bn.R  # of the order-r subgroup on the twist
SMALL = (10069, 5864401, 1875725156269)


@pytest.fixture(scope="module")
def nv():
    import torch
    assert torch.cuda.is_available()
    return _util.native()


class Key:
    """A verifying key with alpha, beta, gamma, delta and the IC points' logs known."""

    def __init__(self, nv, rng, shape, ic):
        self.al, self.be, self.ga, self.de = (rng.randrange(1, bn.R) for _ in range(4))
        self.ic = ic
        pts = {k: bn.g1_bytes(bn.g1_mul(bn.G1_GEN, k) if k else None) for k in set(ic)}
        g2 = [bn.g2_bytes(bn.g2_mul(bn.G2_GEN, k)) for k in (self.be, self.ga, self.de)]
        self.vk = nv.zkvc_vk_import(*shape, bn.g1_bytes(bn.g1_mul(bn.G1_GEN, self.al)), *g2, b"".join(pts[k] for k in ic))

    def c_log(self, X, Y, ab):
        """C's log for an e(A, B) of exponent ab."""
        values = np.concatenate([X.ravel().astype(np.int64), Y.ravel().astype(np.int64)])
        logs = np.array(self.ic[1:], dtype=object)
        s = self.ic[0] + int(sum(logs * values.astype(object)))
        return (ab - self.al * self.be - s * self.ga) * pow(self.de, -1, bn.R) % bn.R


def test_subgroup_decides_when_a_is_infinity(nv):
    rng = random.Random(71)
    X, Y = np.array([[-7]], dtype=np.int8), np.array([[123456]], dtype=np.int32)
    key = Key(nv, rng, (1, 1, 1), [rng.randrange(1, bn.R) for _ in range(3)])
    C = bn.g1_bytes(bn.g1_mul(bn.G1_GEN, key.c_log(X, Y, 0)))
    off = _twist_point_off_subgroup()
    inside = bn.g2_mul(bn.G2_GEN, rng.randrange(1, bn.R))
    cases = [(None, True), (bn.G2_GEN, True), (inside, True), (off, False),
             (bn.g2_mul_noshortcut(off, bn.R), False)]  # the last: the cofactor's part alone
    for q in SMALL:
        assert COFACTOR % q == 0
        part = bn.g2_mul_noshortcut(off, bn.R * COFACTOR // q)
        assert part is not None and bn.g2_on_curve(part) and bn.g2_mul_noshortcut(part, q) is None
        cases += [(part, False), (bn.g2_add(part, inside), False)]
    proofs = [bytes(64) + bn.g2_bytes(B) + C for B, _ in cases]
    m = len(cases)
    got = nv.zkvc_verify_batch([key.vk] * m, [X] * m, [Y] * m, proofs)
    assert got == [ok for _, ok in cases]
    assert got == [nv.zkvc_verify(key.vk, X, Y, p) for p in proofs]
    # a C that is off by one point fails whatever B is
    wrong = bn.g1_bytes(bn.g1_mul(bn.G1_GEN, key.c_log(X, Y, 0) + 1))
    assert nv.zkvc_verify_batch([key.vk] * m, [X] * m, [Y] * m, [p[:192] + wrong for p in proofs]) == [False] * m


def test_merged_sum_special_terms(nv):
    """256 statements of 20,480 terms each (5.2 M terms, 40 per bucket on average: two rounds)."""
    rng = random.Random(72)
    shape = (64, 64, 64)
    n = 2 * 64 * 64
    k = [rng.randrange(1, bn.R) for _ in range(8)]
    patterns = [k, [k[0]], [k[0], bn.R - k[0]], [k[0], 0, bn.R - k[0], k[1], 0]]
    keys = [Key(nv, rng, shape, [rng.randrange(1, bn.R)] + [p[i % len(p)] for i in range(n)]) for p in patterns]
    g = np.random.default_rng(72)

    def inputs(kind):
        X = g.integers(-128, 128, (64, 64), dtype=np.int8)
        Y = g.integers(-(1 << 31), 1 << 31, (64, 64), dtype=np.int64).astype(np.int32)
        if kind == 1:
            X[:], Y[:] = 1, 0x01010101
        if kind == 2:
            X[:], Y[:] = -128, -(1 << 31)
        if kind == 3:
            X[:], Y[:] = 0, 0
            X[5, 5], Y[63, 63] = 127, (1 << 31) - 1
        return X, Y

    a, b = rng.randrange(1, bn.R), rng.randrange(1, bn.R)
    AB = bn.g1_bytes(bn.g1_mul(bn.G1_GEN, a)) + bn.g2_bytes(bn.g2_mul(bn.G2_GEN, b))
    vks, Xs, Ys, proofs, expect = [], [], [], [], []
    for i in range(16):
        key = keys[i % 4]
        X, Y = inputs(i // 4)
        good = AB + bn.g1_bytes(bn.g1_mul(bn.G1_GEN, key.c_log(X, Y, a * b)))
        for j in range(16):
            ok = j % 3 != 1
            Xj = X if ok else X.copy()
            if not ok:  # an input whose point is not at infinity
                Xj[0, 3 * (j % 5)] ^= 1 << (j % 7)
            vks.append(key.vk)
            Xs.append(Xj)
            Ys.append(Y)
            proofs.append(good)
            expect.append(ok or key.ic[1 + 3 * (j % 5)] == 0)
    assert nv.zkvc_verify_batch(vks, Xs, Ys, proofs) == expect
