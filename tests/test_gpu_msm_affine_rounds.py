"""Large MSMs go through the pairwise affine rounds (from 2^22 bucket terms): every case of
an affine addition -- distinct points, doublings, cancellations, infinity on either side --
over whole buckets, against the oracle's [sum s_i k_i]G for points of known discrete logs."""
import ctypes
import math
import random

import pytest
import torch

from oracle import bn254 as bn

pytestmark = pytest.mark.gpu

N = (1 << 18) + 77  # 16 windows' terms per point: just above the rounds' threshold


def _points(group, logs):
    gen, mul, enc = (bn.G1_GEN, bn.g1_mul, bn.g1_bytes) if group == 1 else (bn.G2_GEN, bn.g2_mul, bn.g2_bytes)
    width = 64 * group
    rows = [enc(mul(gen, k % bn.R)) if k % bn.R else bytes(width) for k in logs]
    return torch.tensor(list(b"".join(rows)), dtype=torch.uint8).view(len(logs), width).cuda(), mul, enc, gen


def _case(name, rng):
    """(discrete logs of the distinct points, scalars of the distinct classes): point i is
    point i mod len(logs), scalar i is scalar i mod len(scalars)."""
    k = [rng.randrange(1, bn.R) for _ in range(16)]
    full = [rng.randrange(bn.R) for _ in range(251)]
    return {
        "random": (k, full),
        "one point, one scalar": ([k[0]], [full[0]]),          # doublings all the way up
        "one point, many scalars": ([k[0]], full),
        "point and negative": ([k[0], -k[0]], [full[0]]),       # every bucket cancels
        "negatives in thirds": ([k[0], -k[0], k[1]], full[:7]),
        "infinity among them": ([k[0], 0, k[1], 0, 0], full),
        "only infinity": ([0], full),
        "small scalars": (k, [0, 1, 2, bn.R - 1]),             # a few buckets take every term
    }[name]


@pytest.mark.parametrize("name", ["random", "one point, one scalar", "one point, many scalars", "point and negative",
                                  "negatives in thirds", "infinity among them", "only infinity", "small scalars"])
@pytest.mark.parametrize("group", [1, 2])
def test_affine_rounds(group, name):
    from paper_2504_12217_gb300 import native as nv
    rng = random.Random(31)
    logs, scalars = _case(name, rng)
    P, mul, enc, gen = _points(group, logs)
    s = torch.tensor(list(b"".join(v.to_bytes(32, "little") for v in scalars)), dtype=torch.uint8).view(-1, 32).cuda()
    i = torch.arange(N, device="cuda")
    points, sc = P[i % len(logs)].contiguous(), s[i % len(scalars)].contiguous()
    total = 0
    for a in range(len(logs)):
        for b in range(len(scalars)):
            total += _count(N, a, len(logs), b, len(scalars)) * logs[a] * scalars[b]
    total %= bn.R
    expect = enc(mul(gen, total)) if total else bytes(64 * group)
    got = nv.zkvc_msm_g1(points, sc) if group == 1 else nv.zkvc_msm_g2(points, sc)
    assert got == expect


def _count(n, a, la, b, lb):
    """indices i < n with i = a (mod la) and i = b (mod lb)"""
    period = math.lcm(la, lb)
    for i in range(a, period, la):
        if i % lb == b:
            return (n - 1 - i) // period + 1 if i < n else 0
    return 0


@pytest.mark.parametrize("group", [1, 2])
def test_short_workspace(group):
    """A workspace that holds the run only without the affine rounds gives the same sum; one
    that does not hold that either is refused."""
    from paper_2504_12217_gb300 import native as nv
    rng = random.Random(32)
    logs, scalars = _case("random", rng)
    P, _, _, _ = _points(group, logs)
    s = torch.tensor(list(b"".join(v.to_bytes(32, "little") for v in scalars)), dtype=torch.uint8).view(-1, 32).cuda()
    i = torch.arange(N, device="cuda")
    points, sc = P[i % len(logs)].contiguous(), s[i % len(scalars)].contiguous()
    full = nv.zkvc_msm_workspace_bytes(N, group)
    ws = torch.empty(full, dtype=torch.uint8, device="cuda")
    call = nv.lib().zkvc_msm_g1 if group == 1 else nv.lib().zkvc_msm_g2
    out = [(ctypes.c_uint8 * (64 * group))() for _ in range(3)]
    rc = [call(nv._dev_ptr(points), nv._dev_ptr(sc), N, nv._dev_ptr(ws), size, o, nv._stream())
          for size, o in zip((full, full // 2, full // 16), out)]
    assert rc == [nv.ZKVC_OK, nv.ZKVC_OK, nv.ZKVC_EINVAL]
    assert bytes(out[0]) == bytes(out[1]) and any(out[0])
