"""The proof server's memory admission for keys whose large MSM runs can use more memory than
a request's footprint: a budget of k footprints has k requests in flight, and the larger form
is taken where it leaves room for the other workers' requests."""
import pytest
import torch

from paper_2504_12217_gb300 import inputs
from tests import _util

pytestmark = pytest.mark.gpu

SHAPE, SLOTS = (100, 1280, 1408), 6


@pytest.fixture(scope="module")
def case():
    assert torch.cuda.is_available()
    nv = _util.native()
    pk, _ = nv.zkvc_setup(*SHAPE, inputs.to_bytes32(inputs.setup_values(78)))
    X, W = inputs.matrices(78, *SHAPE)
    rs = inputs.to_bytes32(inputs.prover_values(78))
    expect, _ = nv.zkvc_prove(pk, torch.from_numpy(X).cuda(), torch.from_numpy(W).cuda(), rs)
    return nv, pk, X, W, rs, expect


def _peak(case, policy, budget, count=24):
    nv, pk, X, W, rs, expect = case
    srv = nv.Server([pk], slots=SLOTS, mem_budget=budget, policy=policy)
    tickets = [srv.submit(0, X, W, rs) for _ in range(count)]
    for t in tickets:
        status, proof, _, _ = srv.wait(t, 0)
        assert status == nv.ZKVC_OK and proof == expect
    peak = srv.stats()["peak_bytes"]
    srv.close()
    return peak


@pytest.mark.parametrize("policy", ["fold", "chain"])
def test_footprints_in_flight(case, policy):
    nv, pk = case[:2]
    mode, policy = {"fold": (nv.ZKVC_PROVE_FOLD, nv.ZKVC_SERVER_FOLD),
                    "chain": (nv.ZKVC_PROVE_CHAIN, nv.ZKVC_SERVER_CHAIN)}[policy]
    least = nv.zkvc_server_request_bytes(pk, mode)
    a, n, b = SHAPE
    full = nv.zkvc_prove_workspace_bytes_mode(pk, mode) + a * n + n * b + 4 * a * b
    assert least % 256 == 0 and a * n % 256 == 0 and n * b % 256 == 0 and a * b % 64 == 0
    assert 2 * least < full < SLOTS * least  # the first request could take what two others need
    assert _peak(case, policy, SLOTS * least) == SLOTS * least
    # room for one larger form beside the other workers' footprints
    assert _peak(case, policy, full + (SLOTS - 1) * least) == full + (SLOTS - 1) * least
