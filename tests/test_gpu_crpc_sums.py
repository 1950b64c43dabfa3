"""The prover's CRPC sums (small integers times field elements, summed as whole numbers by
blocks of 256 threads over four rows at a time) against the oracle's closed-form proof: sums
longer than a block, row counts that leave every remainder of four, and the extreme entries
of both signs.  Proof bytes are exact."""
import numpy as np
import pytest

from oracle import crpc, groth16 as og
from paper_2504_12217_gb300 import inputs
from tests import _util

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(257, 5, 1), (1, 6, 300), (300, 3, 257), (255, 4, 256)])
@pytest.mark.parametrize("fill", ["random", "extreme"])
def test_proof_bytes(shape, fill):
    import torch
    nv = _util.native()
    a, n, b = shape
    inst = inputs.instance(4000 + a * 7 + n, shape)
    X, W = inst["X"], inst["W"]
    if fill == "extreme":
        rng = np.random.default_rng(a + n + b)
        X = rng.choice(np.array([-128, 127, 0], dtype=np.int8), size=(a, n))
        W = rng.choice(np.array([-128, 127, 0], dtype=np.int8), size=(n, b))
    pk, _ = nv.zkvc_setup(a, n, b, inputs.to_bytes32(inst["toxic"]))
    proof, _ = nv.zkvc_prove(pk, torch.from_numpy(X).cuda(), torch.from_numpy(W).cuda(), inputs.to_bytes32(inst["rs"]))
    cf, _ = og.closed_form_proof(crpc.Shape(a, n, b), inst["toxic"], X.astype(int).tolist(), W.astype(int).tolist(),
                                 *inst["rs"])
    assert proof == og.proof_bytes(cf)
