"""Sums whose upper windows are empty (small scalars, points at infinity): the same values as
the oracle, and no doublings of nothing -- such a call's time stays well below that of a sum
of full scalars, whose doublings bound it."""
import random
import time

import pytest
import torch

from oracle import bn254 as bn
from tests import _util

pytestmark = pytest.mark.gpu


def _median_s(f):
    for _ in range(3):
        f()
    out = []
    for _ in range(15):
        t = time.perf_counter()
        f()
        out.append(time.perf_counter() - t)
    return sorted(out)[7]


@pytest.mark.parametrize("n", [1, 16, 300])
@pytest.mark.parametrize("group", [1, 2])
def test_empty_windows(group, n):
    assert torch.cuda.is_available()
    nv = _util.native()
    rng = random.Random(group * 1000 + n)
    gen, mul, enc, rows, msm = ((bn.G1_GEN, bn.g1_mul, bn.g1_bytes, _util.g1_rows, nv.zkvc_msm_g1) if group == 1 else
                                (bn.G2_GEN, bn.g2_mul, bn.g2_bytes, _util.g2_rows, nv.zkvc_msm_g2))
    logs = [rng.randrange(1, bn.R) for _ in range(n)]
    P = _util.to_cuda(rows([mul(gen, k) for k in logs]))
    none = torch.zeros_like(P)
    ws = torch.empty(nv.zkvc_msm_workspace_bytes(n, group), dtype=torch.uint8, device="cuda")

    def scalars(bits):
        v = [rng.randrange(1, 1 << bits) % bn.R for _ in range(n)]
        return v, _util.to_cuda(_util.ints_to_u8(v))

    full, full_d = scalars(253)
    for bits in (1, 2, 8, 16, 40, 127, 130, 253):
        v, d = (full, full_d) if bits == 253 else scalars(max(bits, 2) if bits > 1 else 1)
        total = sum(a * b for a, b in zip(logs, v)) % bn.R
        assert msm(P, d, ws) == enc(mul(gen, total)), bits
    assert msm(none, full_d, ws) == bytes(64 * group)
    t_full, t_none = _median_s(lambda: msm(P, full_d, ws)), _median_s(lambda: msm(none, full_d, ws))
    assert t_none < 0.5 * t_full, (t_none, t_full)


@pytest.mark.parametrize("group,n", [(1, (1 << 20) + 3), (2, (1 << 18) + 3)])
def test_infinity_makes_no_terms(group, n):
    """Points at infinity beside a few others, in sums large enough for the affine rounds: the
    oracle's value, in less than half the time of a sum of as many other points."""
    assert torch.cuda.is_available()
    nv = _util.native()
    rng = random.Random(group)
    gen, mul, enc, rows, msm = ((bn.G1_GEN, bn.g1_mul, bn.g1_bytes, _util.g1_rows, nv.zkvc_msm_g1) if group == 1 else
                                (bn.G2_GEN, bn.g2_mul, bn.g2_bytes, _util.g2_rows, nv.zkvc_msm_g2))
    logs = [rng.randrange(1, bn.R) for _ in range(5)]
    at = [0, 1, n // 3, n - 2, n - 1]
    v = [rng.randrange(1, bn.R) for _ in range(5)]
    g = torch.Generator(device="cuda").manual_seed(group)
    s = torch.randint(0, 256, (n, 32), dtype=torch.uint8, device="cuda", generator=g)
    s[at] = _util.to_cuda(_util.ints_to_u8(v))
    few = _util.to_cuda(rows([mul(gen, k) for k in logs]))
    P = torch.zeros((n, 64 * group), dtype=torch.uint8, device="cuda")
    P[at] = few
    full = few[torch.arange(n, device="cuda") % 5].contiguous()
    ws = torch.empty(nv.zkvc_msm_workspace_bytes(n, group), dtype=torch.uint8, device="cuda")
    assert msm(P, s, ws) == enc(mul(gen, sum(a * b for a, b in zip(logs, v)) % bn.R))
    assert _median_s(lambda: msm(P, s, ws)) < 0.5 * _median_s(lambda: msm(full, s, ws))
