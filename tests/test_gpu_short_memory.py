"""A call that allocates its own scratch on a device with little memory left: where the MSM
run's larger form (pairwise affine rounds) does not fit, it runs in the smaller one."""
import pytest
import torch

from paper_2504_12217_gb300 import inputs
from tests import _util

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def nv():
    assert torch.cuda.is_available()
    return _util.native()


def _leave(free):
    """Holds all device memory but `free` bytes."""
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return torch.empty(torch.cuda.mem_get_info()[0] - free, dtype=torch.uint8, device="cuda")


def test_verify_batch(nv):
    """600 proofs of [49,320]x[320,512]: a merged sum of 70 M terms, 3.4 GB with the rounds'
    points and 1.6 GB without, in 2.4 GB."""
    a, n, b = inputs.SHAPE_CFG2
    inst = inputs.instance(inputs.SEED_CFG[2], (a, n, b))
    pk, vk = nv.zkvc_setup(a, n, b, inputs.to_bytes32(inst["toxic"]))
    proof, Y = nv.zkvc_prove(pk, torch.from_numpy(inst["X"]).cuda(), torch.from_numpy(inst["W"]).cuda(),
                             inputs.to_bytes32(inst["rs"]))
    Yh = Y.cpu().numpy()
    bad = Yh.copy()
    bad[3, 5] += 1
    m = 600
    Ys = [bad if i % 7 == 3 else Yh for i in range(m)]
    args = ([vk] * m, [inst["X"]] * m, Ys, [proof] * m)
    expect = [i % 7 != 3 for i in range(m)]
    assert nv.zkvc_verify_batch(*args) == expect
    hold = _leave(2400 << 20)
    try:
        got = nv.zkvc_verify_batch(*args)
    finally:
        del hold
        torch.cuda.empty_cache()
    assert got == expect

