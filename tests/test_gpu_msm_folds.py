"""The folds of an MSM's partial sums with a thread per bucket and the tree's slots listed per
block (runs of more than 16,384 serial folds): buckets of every size side by side, against
the oracle's [sum s_i k_i]G for points of known discrete logs."""
import random

import pytest
import torch

from oracle import bn254 as bn

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scalars", ["random", "half equal", "few"])
@pytest.mark.parametrize("n", [30011, 65536])
@pytest.mark.parametrize("group", [1, 2])
def test_folds(group, n, scalars):
    from paper_2504_12217_gb300 import native as nv
    gen, mul, enc = (bn.G1_GEN, bn.g1_mul, bn.g1_bytes) if group == 1 else (bn.G2_GEN, bn.g2_mul, bn.g2_bytes)
    rng = random.Random(n + group)
    logs = [rng.randrange(1, bn.R) for _ in range(7)]
    s = [rng.randrange(bn.R) for _ in range(n)]
    if scalars == "half equal":  # one bucket per window holds half of the terms
        s[::2] = [s[0]] * len(s[::2])
    elif scalars == "few":       # a few hundred buckets of one to several hundred partial sums
        s = [s[min(rng.randrange(1, 200), rng.randrange(1, 200))] for _ in range(n)]
    P = torch.tensor(list(b"".join(enc(mul(gen, k)) for k in logs)), dtype=torch.uint8).view(len(logs), -1).cuda()
    points = P[torch.arange(n, device="cuda") % len(logs)].contiguous()
    sc = torch.frombuffer(bytearray(b"".join(v.to_bytes(32, "little") for v in s)), dtype=torch.uint8).view(-1, 32).cuda()
    total = sum(v * logs[i % len(logs)] for i, v in enumerate(s)) % bn.R
    got = nv.zkvc_msm_g1(points, sc) if group == 1 else nv.zkvc_msm_g2(points, sc)
    assert got == enc(mul(gen, total))
