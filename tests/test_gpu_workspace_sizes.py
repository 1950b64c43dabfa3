"""Workspaces smaller than the *_workspace_bytes answers, but as large as the runs' smaller
form needs (no pairwise affine rounds, chunks of 16 terms), are accepted and give the same
bytes: callers keep the sizes that earlier builds asked for."""

import ctypes

import pytest
import torch

from paper_2504_12217_gb300 import inputs
from tests import _util

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def nv():
    assert torch.cuda.is_available()
    return _util.native()


def _scalars(seed, n):
    g = torch.Generator(device="cuda").manual_seed(seed)
    k = torch.randint(0, 256, (n, 32), dtype=torch.uint8, device="cuda", generator=g)
    k[:, 31] &= 0x1F
    return k


def _ws(n):
    return torch.empty(n, dtype=torch.uint8, device="cuda")


MSM = [(1, 1, 84928), (1, 7, 93376), (1, 100, 233664), (1, 1000, 1194432), (1, 2000, 2224576),
       (1, 262221, 144158400), (1, 3000001, 1107914944), (2, 1, 151168), (2, 7, 163456), (2, 100, 374912), (2, 1000, 1873536),
       (2, 2000, 3486592), (2, 262221, 220363904), (2, 1048576, 597881728)]


@pytest.mark.parametrize("group,n,size", MSM)
def test_msm_former_size(nv, group, n, size):
    mul, msm = ((nv.zkvc_g1_generator_mul, nv.zkvc_msm_g1) if group == 1 else
                (nv.zkvc_g2_generator_mul, nv.zkvc_msm_g2))
    P, s = mul(_scalars(n, n)), _scalars(n + 1, n)
    assert size < nv.zkvc_msm_workspace_bytes(n, group)
    call = nv.lib().zkvc_msm_g1 if group == 1 else nv.lib().zkvc_msm_g2  # (the binding replaces short workspaces)
    out, ws = (ctypes.c_uint8 * (64 * group))(), _ws(size)
    assert call(nv._dev_ptr(P), nv._dev_ptr(s), n, nv._dev_ptr(ws), size, out, nv._stream()) == nv.ZKVC_OK
    assert bytes(out) == msm(P, s)


PROVE = [((1, 1, 1), 10712320, 5431296), ((4, 16, 8), 10865920, 5540352), ((5, 7, 3), 10782208, 5479680),
         ((49, 320, 512), 59400960, 39049472), ((63, 333, 517), 64838144, 39825152),
         ((197, 768, 768), 281837056, 199092480)]


@pytest.mark.parametrize("shape,fold,chain", PROVE)
def test_prove_former_size(nv, shape, fold, chain):
    seed = 4100 + sum(shape)
    pk, _ = nv.zkvc_setup(*shape, inputs.to_bytes32(inputs.setup_values(seed)))
    X, W = (torch.from_numpy(m).cuda() for m in inputs.matrices(seed, *shape))
    rs = inputs.to_bytes32(inputs.prover_values(seed))
    for mode, size in ((nv.ZKVC_PROVE_FOLD, fold), (nv.ZKVC_PROVE_CHAIN, chain)):
        assert size < nv.zkvc_prove_workspace_bytes_mode(pk, mode)
        expect, Y0 = nv.zkvc_prove_mode(pk, mode, X, W, rs)
        ws, Y, proof = _ws(size), torch.empty_like(Y0), ctypes.create_string_buffer(256)
        for _ in range(3):  # direct, captured, replayed
            rc = nv.lib().zkvc_prove_mode(pk.handle, mode, nv._dev_ptr(X), nv._dev_ptr(W), rs, nv._dev_ptr(Y),
                                          nv._dev_ptr(ws), size, proof, nv._stream())
            assert rc == nv.ZKVC_OK
            assert proof.raw == expect and torch.equal(Y, Y0)


CIRCUIT = [("crpc", (4, 16, 8), 21338368), ("crpc_psq", (20, 30, 20), 22326784),
           ("crpc_psq_gelu", (4, 16, 8), 21409536), ("psq", (4, 16, 8), 21776640), ("vanilla", (20, 30, 20), 29816320)]


@pytest.mark.parametrize("circuit,shape,size", CIRCUIT)
def test_circuit_former_size(nv, circuit, shape, size):
    seed = 4200 + sum(shape)
    pk, _ = nv.zkvc_setup_circuit(*shape, circuit, "xy", inputs.to_bytes32(inputs.setup_values(seed)))
    X, W = (torch.from_numpy(m).cuda() for m in inputs.matrices(seed, *shape))
    rs = inputs.to_bytes32(inputs.prover_values(seed))
    assert size < nv.zkvc_prove_workspace_bytes(pk)
    expect, Y = nv.zkvc_prove(pk, X, W, rs)
    ws, proof = _ws(size), ctypes.create_string_buffer(256)
    assert nv.lib().zkvc_prove(pk.handle, nv._dev_ptr(X), nv._dev_ptr(W), rs, nv._dev_ptr(Y), nv._dev_ptr(ws), size,
                               proof, nv._stream()) == nv.ZKVC_OK
    assert proof.raw == expect


def test_server_footprints(nv):
    """What the server needs for a request at the least: the smaller workspace, X, W and Y."""
    def up(x):
        return (x + 255) // 256 * 256
    for (a, n, b), fold, chain in PROVE:
        pk, _ = nv.zkvc_setup(a, n, b, inputs.to_bytes32(inputs.setup_values(7)))
        rest = up(a * n) + up(n * b) + up(4 * a * b)
        assert nv.zkvc_server_request_bytes(pk, nv.ZKVC_PROVE_FOLD) <= fold + rest
        assert nv.zkvc_server_request_bytes(pk, nv.ZKVC_PROVE_CHAIN) <= chain + rest
