"""The measured cases: what a program that uses this library has it do.

Three layers of the public API, each from its smallest calls to its largest:

* proofs -- one per call (`zkvc_prove`, `zkvc_prove_mode`), many per call (`Batch.prove`),
  and over the generic circuits (`zkvc_setup_circuit`);
* the kernel layer -- `zkvc_msm_g1`, `zkvc_msm_g2`, `zkvc_ntt`;
* verification of proofs on the GPU (`zkvc_verify_batch`).

Shapes are [tokens, dim] x [dim, out] products of the Transformer layers that the
benchmark and the tests use; keys, plans and workspaces are made in `prepare` and kept, as
a program that proves more than once keeps them.
"""
import random

import numpy as np
import torch

from paper_2504_12217_gb300 import inputs
from paper_2504_12217_gb300 import native as nv

_MODES = {"fold": nv.ZKVC_PROVE_FOLD, "chain": nv.ZKVC_PROVE_CHAIN}
_KINDS = {"forward": nv.ZKVC_NTT_FORWARD, "inverse": nv.ZKVC_NTT_INVERSE,
          "coset_forward": nv.ZKVC_NTT_COSET_FORWARD, "coset_inverse": nv.ZKVC_NTT_COSET_INVERSE}
_R = 21888242871839275222246405745257275088548364400416034343698204186575808495617


def listed():
    return [
        # the smallest proof of the test suite: launches and serial chains only
        {"name": "prove_4x16x8", "op": "prove", "a": 4, "n": 16, "b": 8, "mode": "default"},
        # the benchmark's proof, in the mode that its autotuner and the server choose
        {"name": "prove_49x320x512_chain", "op": "prove", "a": 49, "n": 320, "b": 512, "mode": "chain"},
        # the same in the mode of a key that nobody tuned, at a ragged shape
        {"name": "prove_63x333x517", "op": "prove", "a": 63, "n": 333, "b": 517, "mode": "default"},
        # the largest layer of the batched workload (an MLP expansion of 197 tokens)
        {"name": "prove_197x768x3072_chain", "op": "prove", "a": 197, "n": 768, "b": 3072, "mode": "chain"},
        # the batched workload: 64 proofs of mixed layer shapes in one captured sequence
        {"name": "batch_64mix", "op": "batch", "count": 64, "mix": 1},
        # an ablation circuit on the generic engine (one row per product)
        {"name": "circuit_vanilla_49x64x128", "op": "circuit", "a": 49, "n": 64, "b": 128, "circuit": "vanilla",
         "public": "xy"},
        # multi-scalar multiplications of a caller's own points: a small commitment, the
        # sweep's first size, a large odd one, and the other group
        {"name": "msm_g1_1000", "op": "msm", "group": 1, "points": 1000},
        {"name": "msm_g1_65536", "op": "msm", "group": 1, "points": 65536},
        {"name": "msm_g1_3000001", "op": "msm", "group": 1, "points": 3000001},
        {"name": "msm_g2_65536", "op": "msm", "group": 2, "points": 65536},
        # one large polynomial evaluated on the domain and back from its coset
        {"name": "ntt_2e22_coset_inverse", "op": "ntt", "log_n": 22, "kind": "coset_inverse"},
        # a verifier's queue: proofs of one layer, checked together
        {"name": "verify_32", "op": "verify", "a": 49, "n": 320, "b": 512, "count": 32},
    ]


def _log_int(rng, lo, hi):
    """An integer of [lo, hi], spread over its logarithm (odd values as likely as even)."""
    return max(lo, min(hi, int(round(lo * (hi / lo) ** rng.random()))))


def draw(rng):
    op = rng.choice(["prove", "prove", "msm", "msm", "ntt", "circuit", "batch", "verify"])
    if op == "prove":
        return {"op": op, "a": _log_int(rng, 1, 197), "n": _log_int(rng, 2, 768), "b": _log_int(rng, 1, 3072),
                "mode": rng.choice(["default", "fold", "chain"])}
    if op == "msm":
        group = rng.choice([1, 1, 2])
        return {"op": op, "group": group, "points": _log_int(rng, 1, 3000001 if group == 1 else 300001)}
    if op == "ntt":
        return {"op": op, "log_n": rng.randint(1, 22), "kind": rng.choice(sorted(_KINDS))}
    if op == "circuit":
        return {"op": op, "a": _log_int(rng, 1, 49), "n": _log_int(rng, 1, 64), "b": _log_int(rng, 1, 128),
                "circuit": rng.choice(sorted(nv.CIRCUIT_NAMES)), "public": rng.choice(sorted(nv.PUBLIC_NAMES))}
    if op == "batch":
        return {"op": op, "count": _log_int(rng, 1, 64), "mix": rng.randint(2, 1 << 20)}
    return {"op": op, "a": _log_int(rng, 1, 64), "n": _log_int(rng, 2, 320), "b": _log_int(rng, 1, 512),
            "count": _log_int(rng, 12, 32)}


def _gen(seed, device="cuda"):
    return torch.Generator(device=device).manual_seed(seed)


def _int8(g, rows, cols):
    """Quantised activations and weights: int8, uniform."""
    return torch.randint(-128, 128, (rows, cols), dtype=torch.int8, device="cuda", generator=g)


def _scalars(g, n):
    """Uniform field elements of 253 bits, canonical little-endian."""
    k = torch.randint(0, 256, (n, 32), dtype=torch.uint8, device="cuda", generator=g)
    k[:, 31] &= 0x1F
    return k


def _toxic(seed):
    return inputs.to_bytes32(inputs.setup_values(seed))


def _rs(seed):
    return inputs.to_bytes32(inputs.prover_values(seed))


def _proof_array(proof):
    return np.frombuffer(proof, dtype=np.uint8)


def _batch_shapes(case):
    return inputs.batch_shapes(inputs.SEED_CFG[4] if case["mix"] == 1 else case["mix"], case["count"])


def prepare(case, seed):
    op = case["op"]
    g = _gen(seed)
    if op in ("prove", "circuit"):
        a, n, b = case["a"], case["n"], case["b"]
        if op == "prove":
            pk, _ = nv.zkvc_setup(a, n, b, _toxic(seed))
            mode = _MODES.get(case["mode"])
        else:
            pk, _ = nv.zkvc_setup_circuit(a, n, b, case["circuit"], case["public"], _toxic(seed))
            mode = None
        need = nv.zkvc_prove_workspace_bytes(pk) if mode is None else nv.zkvc_prove_workspace_bytes_mode(pk, mode)
        return {"op": op, "pk": pk, "mode": mode, "X": _int8(g, a, n), "W": _int8(g, n, b), "rs": _rs(seed),
                "Y": torch.empty((a, b), dtype=torch.int32, device="cuda"),
                "ws": torch.empty(need, dtype=torch.uint8, device="cuda")}
    if op == "batch":
        shapes = _batch_shapes(case)
        keys = {}
        for i, sh in enumerate(shapes):  # equal shapes share a key, as the layers of a model do
            if sh not in keys:
                keys[sh] = nv.zkvc_setup(*sh, _toxic(seed + i))[0]
        pks = [keys[sh] for sh in shapes]
        ends = np.cumsum([a * b for a, _, b in shapes]).tolist()
        Y = torch.empty(ends[-1], dtype=torch.int32, device="cuda")
        return {"op": op, "batch": nv.Batch(pks), "X": [_int8(g, a, n) for a, n, _ in shapes],
                "W": [_int8(g, n, b) for _, n, b in shapes], "rs": [_rs(seed + i) for i in range(len(shapes))],
                "Y": Y, "Ys": [Y[e - a * b:e].view(a, b) for e, (a, _, b) in zip(ends, shapes)]}
    if op == "msm":
        n, group = case["points"], case["group"]
        mul = nv.zkvc_g1_generator_mul if group == 1 else nv.zkvc_g2_generator_mul
        return {"op": op, "group": group, "P": mul(_scalars(g, n)), "s": _scalars(g, n),
                "ws": torch.empty(nv.zkvc_msm_workspace_bytes(n, group), dtype=torch.uint8, device="cuda")}
    if op == "ntt":
        return {"op": op, "x": _scalars(g, 1 << case["log_n"]), "kind": _KINDS[case["kind"]]}
    a, n, b = case["a"], case["n"], case["b"]
    pk, vk = nv.zkvc_setup(a, n, b, _toxic(seed))
    Xs, Ys, proofs, rng = [], [], [], random.Random(seed)
    for i in range(case["count"]):
        X, W = _int8(g, a, n), _int8(g, n, b)
        proof, Y = nv.zkvc_prove(pk, X, W, _rs(seed + i))
        if rng.random() < 0.25:  # claims that do not hold are among them, as a verifier meets
            Y[0, 0] += 1
        Xs.append(X.cpu().numpy())
        Ys.append(Y.cpu().numpy())
        proofs.append(proof)
    return {"op": op, "vks": [vk] * case["count"], "Xs": Xs, "Ys": Ys, "proofs": proofs}


def run(state):
    op = state["op"]
    if op in ("prove", "circuit"):
        if state["mode"] is None:
            proof, Y = nv.zkvc_prove(state["pk"], state["X"], state["W"], state["rs"], Y=state["Y"],
                                     workspace=state["ws"])
        else:
            proof, Y = nv.zkvc_prove_mode(state["pk"], state["mode"], state["X"], state["W"], state["rs"],
                                          Y=state["Y"], workspace=state["ws"])
        return {"proof": _proof_array(proof), "Y": Y}
    if op == "batch":
        proofs, _ = state["batch"].prove(state["X"], state["W"], state["rs"], state["Ys"])
        return {"proofs": _proof_array(b"".join(proofs)), "Y": state["Y"]}  # Y holds every instance's product
    if op == "msm":
        msm = nv.zkvc_msm_g1 if state["group"] == 1 else nv.zkvc_msm_g2
        return _proof_array(msm(state["P"], state["s"], state["ws"]))
    if op == "ntt":  # the transform is in place; the caller keeps its coefficients
        return nv.zkvc_ntt(state["x"].clone(), state["kind"])
    return np.array(nv.zkvc_verify_batch(state["vks"], state["Xs"], state["Ys"], state["proofs"]), dtype=np.int32)


# ------------------------------------------------------------------ the work of one pass
# One modular product of 256 bits: 8 x 8 limb products and as many for the reduction, each
# a 32 x 32 -> 64-bit multiply-add (two operations).
_PRODUCT = 2 * 128
_G2 = 3  # base-field products per product of the quadratic extension


def _msm_products(terms):
    """An addition of two affine points: 6 products, its inversion shared."""
    return 6 * terms


def _variable_terms(n):
    c = max(4, min(16, (2 * n - 1).bit_length() - 3))
    return 2 * n * -(-128 // c)


def _domain(rows):
    return 1 << max(1, (rows - 1).bit_length())


def _proof_work(a, n, b):
    N = _domain(n + 1 + a * n + a * b)
    products = 7 * (N // 2) * (N.bit_length() - 1)                      # quotient: 7 transforms
    products += _msm_products(16 * N + a * n + 4 * a * b + 4 * 32 * n)  # H, X, Y and row terms
    products += _G2 * _msm_products(32 * n)
    products += a * n + n * b + a * b                                   # CRPC evaluations
    return {"bytes": a * n + n * b + 4 * a * b + 64 * (16 * N + a * n + 4 * a * b + 64 * n) + 128 * 32 * n,
            "flops": _PRODUCT * products + 2 * a * n * b}


def _circuit_work(case):
    a, n, b = case["a"], case["n"], case["b"]
    public = 1 if case["public"] == "none" else 1 + a * n + a * b
    aux = {"crpc_psq": n, "crpc": n, "psq": a * n * b, "vanilla": a * n * b, "crpc_psq_softmax": n + 72 * a * b,
           "crpc_psq_gelu": n + 2 * a * b}[case["circuit"]]
    N = _domain(aux + public)
    terms = 16 * (N + aux) + 2 * a * n + 2 * n * b + 2 * a * b
    return {"bytes": a * n + n * b + 4 * a * b + 64 * terms,
            "flops": _PRODUCT * (7 * (N // 2) * (N.bit_length() - 1) + _msm_products(terms))}


def work(case):
    op = case["op"]
    if op == "prove":
        return _proof_work(case["a"], case["n"], case["b"])
    if op == "batch":
        each = [_proof_work(*sh) for sh in _batch_shapes(case)]
        return {k: sum(w[k] for w in each) for k in ("bytes", "flops")}
    if op == "circuit":
        return _circuit_work(case)
    if op == "msm":
        n, wide = case["points"], case["group"]
        products = _msm_products(_variable_terms(n)) * (1 if wide == 1 else _G2)
        return {"bytes": n * (64 * wide + 32) + 64 * wide, "flops": _PRODUCT * products}
    if op == "ntt":
        N = 1 << case["log_n"]
        return {"bytes": 64 * N, "flops": _PRODUCT * (N // 2) * case["log_n"]}
    # four Miller loops of 64 doublings and 37 additions (about 60 products each) and one
    # final exponentiation (about 9,000 products) per proof, and the public inputs' sum
    a, n, b, m = case["a"], case["n"], case["b"], case["count"]
    products = m * (4 * 101 * 60 + 9000 + _msm_products(a * n + 2 * a * b))
    return {"bytes": m * (256 + a * n + 4 * a * b) + 64 * (a * n + a * b), "flops": _PRODUCT * products}


# ------------------------------------------------------------------ exact values
def _product(X, W):
    return X.cpu().numpy().astype(np.int64) @ W.cpu().numpy().astype(np.int64)


def _exact_ntt(log_n, kind, values):
    """The transform in Python integers (natural order in and out)."""
    N = 1 << log_n
    w = pow(pow(5, (_R - 1) >> 28, _R), 1 << (28 - log_n), _R)
    inverse = kind in ("inverse", "coset_inverse")
    if inverse:
        w = pow(w, -1, _R)
    x = list(values)
    if kind == "coset_forward":
        s = 1
        for i in range(N):
            x[i] = x[i] * s % _R
            s = s * 5 % _R
    roots = [1] * max(1, N // 2)
    for i in range(1, N // 2):
        roots[i] = roots[i - 1] * w % _R
    half, step = N // 2, 1  # decimation in frequency: natural in, bit-reversed out
    while half:
        for lo in range(0, N, 2 * half):
            for j in range(half):
                u, v = x[lo + j], x[lo + j + half]
                x[lo + j] = (u + v) % _R
                x[lo + j + half] = (u - v) * roots[j * step] % _R
        half //= 2
        step *= 2
    out = [0] * N
    for i in range(N):
        out[int(format(i, f"0{log_n}b")[::-1], 2)] = x[i]
    if inverse:
        s, g = pow(N, -1, _R), pow(5, -1, _R) if kind == "coset_inverse" else 1
        for i in range(N):
            out[i] = out[i] * s % _R
            s = s * g % _R
    return out


def exact(case, seed):
    """Y as numpy's 64-bit product, transforms as Python integers; a proof, a sum of points
    and a verdict have no value that plain numpy or torch computes."""
    op = case["op"]
    g = _gen(seed)
    if op in ("prove", "circuit"):
        X, W = _int8(g, case["a"], case["n"]), _int8(g, case["n"], case["b"])
        return {"proof": None, "Y": _product(X, W)}
    if op == "batch":
        shapes = _batch_shapes(case)
        if sum(a * n * b for a, n, b in shapes) > 1 << 31:
            return None
        Xs = [_int8(g, a, n) for a, n, _ in shapes]
        Ws = [_int8(g, n, b) for _, n, b in shapes]
        return {"proofs": None, "Y": np.concatenate([_product(X, W).ravel() for X, W in zip(Xs, Ws)])}
    if op == "ntt" and case["log_n"] <= 18:
        raw = _scalars(g, 1 << case["log_n"]).cpu().numpy()
        out = _exact_ntt(case["log_n"], case["kind"], [int.from_bytes(r.tobytes(), "little") for r in raw])
        return np.frombuffer(b"".join(v.to_bytes(32, "little") for v in out), dtype=np.uint8).reshape(-1, 32).copy()
    return None
