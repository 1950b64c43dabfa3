"""The pairwise affine rounds where several follow one another: infinities that a round's
cancellations leave are the next round's operands, doublings double intermediate sums, the
rounds' two buffers trade places, and more than one slab of terms is run."""
import random

import pytest
import torch

from oracle import bn254 as bn
from tests.test_gpu_msm_affine_rounds import _case, _count, _points

pytestmark = pytest.mark.gpu

THREE = (1 << 20) + 77  # 64 terms per bucket on average: three rounds
SLABS = (1 << 21) + 5   # 2^25 terms and a few more: two slabs, four rounds


def _check(group, name, n):
    from paper_2504_12217_gb300 import native as nv
    logs, scalars = _case(name, random.Random(33))
    P, mul, enc, gen = _points(group, logs)
    s = torch.tensor(list(b"".join(v.to_bytes(32, "little") for v in scalars)), dtype=torch.uint8).view(-1, 32).cuda()
    i = torch.arange(n, device="cuda")
    total = sum(_count(n, a, len(logs), b, len(scalars)) * logs[a] * scalars[b]
                for a in range(len(logs)) for b in range(len(scalars))) % bn.R
    expect = enc(mul(gen, total)) if total else bytes(64 * group)
    points, sc = P[i % len(logs)].contiguous(), s[i % len(scalars)].contiguous()
    assert (nv.zkvc_msm_g1 if group == 1 else nv.zkvc_msm_g2)(points, sc) == expect


@pytest.mark.parametrize("name", ["random", "one point, one scalar", "one point, many scalars", "point and negative",
                                  "negatives in thirds", "infinity among them", "only infinity", "small scalars"])
@pytest.mark.parametrize("group", [1, 2])
def test_three_rounds(group, name):
    _check(group, name, THREE)


@pytest.mark.parametrize("name", ["random", "one point, one scalar", "point and negative", "only infinity"])
def test_two_slabs(name):
    _check(1, name, SLABS)
