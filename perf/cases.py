"""Performance cases of the library: what its users have it do, over the sizes they do it at.

A case is a dict of plain values. Kinds:

  prepare   chunk inverse + W/U (`chunk_prepare`), bf16 or fp32, every chunk size, dense [B,H,T,d] tensors
  layer     the whole chunk-wise layer as model code calls it (`gated_delta_layer`: token-major tensors, raw log-gates, raw
            key / query projections), with or without a state carried in
  packed    the same on sequences of different lengths laid end to end (`cu_seqlens`), as a serving batch arrives
  int8      the INT8 entry point (`chunk_prepare_int8`), chunks of 64 or 128 tokens
  int16     the INT16 entry point (`chunk_prepare_int16`)

`run` calls the public binding and lets it allocate its outputs, as a caller without an output pool does.
"""
from __future__ import annotations

import math
import random

import torch

from paper_2606_06034_b200 import binding as gdn
from paper_2606_06034_b200 import inputs as gen

D = 128


def _prepare(name, B, H_k, H_v, T, C, dtype="bf16", adversarial="none", d=D):
    return {"name": name, "kind": "prepare", "B": B, "H_k": H_k, "H_v": H_v, "T": T, "C": C, "dtype": dtype,
            "adversarial": adversarial, "d": d}


def _layer(name, B, H_k, H_v, T, carry):
    return {"name": name, "kind": "layer", "B": B, "H_k": H_k, "H_v": H_v, "T": T, "C": 64, "carry": carry, "d": D}


def _packed(name, H_k, H_v, T, n_seq, pattern):
    return {"name": name, "kind": "packed", "B": 1, "H_k": H_k, "H_v": H_v, "T": T, "C": 64, "n_seq": n_seq, "pattern": pattern,
            "d": D}


def _integer(name, kind, B, H_k, H_v, T, C=64):
    return {"name": name, "kind": kind, "B": B, "H_k": H_k, "H_v": H_v, "T": T, "C": C, "d": D}


def listed():
    return [
        # one short fp32 call: the reference precision on a handful of chunks, where a launch's latency is all there is
        _prepare("fp32_tiny", 1, 2, 2, 256, 64, "fp32"),
        # fp32 over a layer of an ordinary prompt: offline checks of a model's quality against the low-precision paths
        _prepare("fp32_layer", 1, 16, 16, 4096, 64, "fp32"),
        # the chunk-size sweep: a training-sized batch at the chunk sizes models are run with
        _prepare("bf16_c32", 4, 16, 16, 4096, 32),
        _prepare("bf16_c64", 4, 16, 16, 4096, 64),
        _prepare("bf16_c128", 4, 16, 16, 4096, 128),
        # the largest: eight long documents, half of the heads with the strongly correlated keys and open gates on which the
        # series grows most
        _prepare("bf16_stress", 8, 32, 32, 65536, 64, "bf16", "odd"),
        # one more chunk of a running conversation: a layer call on 64 new tokens with the state so far
        _layer("layer_one_chunk", 1, 16, 32, 64, True),
        # prefill of one long prompt
        _layer("layer_prefill", 1, 16, 32, 32768, False),
        # prefill of a batch of equal prompts (or the forward pass of a training batch)
        _layer("layer_batch", 8, 32, 32, 4096, False),
        # a serving batch: prompts of very different lengths packed end to end, none of them a multiple of the chunk
        _packed("layer_packed", 16, 32, 16411, 61, 7),
        # the low-bit variants on a long prompt
        _integer("int8_prefill", "int8", 1, 16, 32, 32768),
        _integer("int16_prefill", "int16", 1, 16, 32, 32768),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["prepare", "prepare", "fp32", "layer", "layer", "packed", "packed", "int8", "int16"])
    H_k = rng.choice([1, 2, 3, 4, 6, 8, 12, 16, 24, 32])
    H_v = H_k * rng.choice([1, 1, 2, 4])
    if kind == "fp32":
        C = rng.choice([16, 24, 32, 48, 64, 64, 64, 128])
        B = rng.choice([1, 1, 2, 3])
        tokens = _log_int(rng, 256, 65536)  # of all heads together
        T = C * max(1, tokens // (B * H_v * C))
        return _prepare("", B, H_k, H_v, T, C, "fp32", "none", rng.choice([64, 96, 128, 128]))
    if kind == "prepare":
        C = rng.choice([16, 32, 64, 64, 128])
        B = rng.choice([1, 1, 2, 4, 5, 8])
        tokens = _log_int(rng, 4096, 8 << 20)
        T = C * max(1, tokens // (B * H_v * C))
        return _prepare("", B, H_k, H_v, T, C, "bf16", rng.choice(["none", "odd"]))
    if kind == "layer":
        B = rng.choice([1, 1, 1, 2, 4, 8, 12])
        tokens = _log_int(rng, 2048, 1 << 20)
        T = 64 * max(1, tokens // (B * H_v * 64))
        return _layer("", B, H_k, H_v, T, rng.random() < 0.5)
    if kind == "packed":
        T = _log_int(rng, 8, 32768)
        n_seq = min(T, _log_int(rng, 1, 256))
        return _packed("", H_k, H_v, T, n_seq, rng.randrange(1 << 16))
    B = rng.choice([1, 1, 2, 4])
    C = rng.choice([64, 64, 128]) if kind == "int8" else 64
    tokens = _log_int(rng, 4096, 1 << 20)
    T = C * max(1, tokens // (B * H_v * C))
    return _integer("", kind, B, H_k, H_v, T, C)


def _boundaries(case):
    """Sequence boundaries of a packed case: lengths log-normal around their mean (a few long prompts, many short ones)."""
    r = random.Random(case["pattern"])
    w = [r.lognormvariate(0.0, 1.0) for _ in range(case["n_seq"])]
    spare = case["T"] - case["n_seq"]  # every sequence has at least one token
    total, acc, cu = sum(w), 0.0, [0]
    for i, x in enumerate(w):
        acc += x
        cu.append(i + 1 + int(spare * acc / total))
    cu[-1] = case["T"]
    return cu


def prepare(case, seed):
    dev = "cuda"
    kind = case["kind"]
    if kind in ("prepare", "int8", "int16"):
        d = case["d"]
        inp = gen.make_inputs(case["B"], case["H_k"], case["H_v"], case["T"], case["C"], d, d, seed=seed, device=dev,
                              dtype=torch.float32 if case.get("dtype") == "fp32" else torch.bfloat16,
                              adversarial_heads=case.get("adversarial", "none"))
        if kind == "prepare":
            return {"case": case, "K": inp.K, "V": inp.V, "beta": inp.beta, "g": inp.g}
        return {"case": case, "q": gen.make_int8_inputs(inp) if kind == "int8" else gen.make_int16_inputs(inp)}
    # layer and packed: what the projections of a model hand over, token-major
    g = torch.Generator(device=dev)
    g.manual_seed(seed)
    lead = (case["B"], case["T"]) if kind == "layer" else (case["T"],)
    H_k, H_v = case["H_k"], case["H_v"]

    def randn(*shape):
        return torch.randn(*shape, generator=g, device=dev, dtype=torch.float32)

    st = {"case": case, "Q": randn(*lead, H_k, D).bfloat16(), "K": randn(*lead, H_k, D).bfloat16(),
          "V": randn(*lead, H_v, D).bfloat16(), "beta": torch.sigmoid(randn(*lead, H_v)),
          "g": -torch.nn.functional.softplus(randn(*lead, H_v)), "S": None}
    if kind == "packed":
        st["cu"] = _boundaries(case)
    elif case["carry"]:
        st["S"] = 0.3 * randn(case["B"], H_v, D, D)
    return st


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "prepare":
        return gdn.chunk_prepare(state["K"], state["V"], state["beta"], state["g"], case["C"])
    if kind == "layer":
        return gdn.gated_delta_layer(state["Q"], state["K"], state["V"], state["beta"], state["g"], S_in=state["S"])
    if kind == "packed":
        return gdn.gated_delta_layer(state["Q"], state["K"], state["V"], state["beta"], state["g"], cu_seqlens=state["cu"])
    if kind == "int8":
        return gdn.chunk_prepare_int8(state["q"])
    return gdn.chunk_prepare_int16(state["q"])


def work(case):
    """Every input read once, every output written once; multiply-adds on the triangles the scheme needs (Gram matrix, exact
    inverse, W and U; for the layer the products with the state and the masked attention of a chunk)."""
    B, H_k, H_v, T, C, d = (case[k] for k in ("B", "H_k", "H_v", "T", "C", "d"))
    kind = case["kind"]
    keys, vals = B * H_k * T, B * H_v * T  # token rows
    flops = keys * C * d + vals * (C * C / 3 + 2 * C * d)
    if kind == "prepare":
        e = 4 if case["dtype"] == "fp32" else 2
        return {"bytes": e * d * (keys + 3 * vals) + e * C * vals + 8 * vals, "flops": flops}
    if kind in ("int8", "int16"):
        e = 1 if kind == "int8" else 2
        exps = 4 * (keys + (7 if C == 128 else 4) * vals) / C
        return {"bytes": e * d * (keys + 3 * vals) + e * C * vals + 6 * vals + exps, "flops": flops}
    n_state = case["n_seq"] if kind == "packed" else B
    states = 4 * d * d * H_v * n_state * (2 if case.get("carry") else 1)
    return {"bytes": 2 * d * (2 * keys + 2 * vals) + 8 * vals + states,
            "flops": flops + keys * C * d + vals * (6 * d * d + C * d)}


def tolerance(case):
    kind = case["kind"]
    if kind in ("int8", "int16"):
        return "exact"  # whole numbers: a pure function of the integer inputs
    # four times the measured distance from the same quantities evaluated in fp64: 2.6e-8 (fp32; the diagonal of T, exact,
    # carries most of the norm of W and U), 1.7e-3 (bf16 W and U: one rounding of the result), 2.35e-3 (layer: W and U pass
    # through bf16 on their way to the output)
    if kind == "prepare":
        return {"rel": 1.2e-7 if case["dtype"] == "fp32" else 7e-3}
    return {"rel": 9.5e-3}


def _inverse(A, C):
    """The scheme's inverse of I + A in fp64 (A strictly lower triangular, [..., C, C]): band-masked Neumann sum of order N, then
    T0 (I + E + ... + E^S); 128 tokens as two 64-blocks and the block formula for the lower-left one."""
    if C == 128:
        T = torch.zeros_like(A)
        T11, T22 = _inverse(A[..., :64, :64], 64), _inverse(A[..., 64:, 64:], 64)
        T[..., :64, :64], T[..., 64:, 64:] = T11, T22
        T[..., 64:, :64] = -T22 @ A[..., 64:, :64] @ T11
        return T
    N = min(3, C - 1)
    S = {16: 3, 32: 4, 64: 8}.get(C, max(0, (C + 3) // 4 - 1))
    eye = torch.eye(C, dtype=A.dtype, device=A.device)
    P, T0 = -A, eye - A
    for _ in range(N - 1):
        P = P @ -A
        T0 = T0 + P
    T0 = T0.tril().triu(-N)
    E = eye - (eye + A) @ T0
    X = eye.expand_as(E)
    for _ in range(S):  # Horner: I + E (I + E (...))
        X = eye + E @ X
    return T0 @ X


def _chunks(K, V, beta, g, C, gated=False):
    """W, U and the inverse of chunks K, V [..., C, d], beta and cumulative g [..., C], all fp64."""
    decay = (g[..., :, None] - g[..., None, :]).tril(-1).exp().tril(-1)
    T = _inverse(beta[..., :, None] * decay * (K @ K.transpose(-1, -2)), C)
    w = beta * g.exp() if gated else beta
    return T @ (w[..., None] * K), T @ (beta[..., None] * V), T


def _exact_prepare(case, st):
    B, H_k, H_v, T, C, d = (case[k] for k in ("B", "H_k", "H_v", "T", "C", "d"))
    n, r = T // C, H_v // H_k

    def empty(*shape):
        return torch.empty(*shape, dtype=torch.float64, device="cuda")

    W, U, Ti = empty(B, H_v, n, C, d), empty(B, H_v, n, C, d), empty(B, H_v, n, C, C)
    for b in range(B):
        for h in range(H_v):
            W[b, h], U[b, h], Ti[b, h] = _chunks(*(x.double().view(n, C, -1) for x in (st["K"][b, h // r], st["V"][b, h])),
                                                 *(x.double().view(n, C) for x in (st["beta"][b, h], st["g"][b, h])), C)
    return W.view(B, H_v, T, d), U.view(B, H_v, T, d), Ti


def _unit(x):
    x = x.double()
    return x / x.norm(dim=-1, keepdim=True).clamp_min(1e-300)


def _exact_layer(case, st):
    H_k, H_v, C = case["H_k"], case["H_v"], case["C"]
    dense = case["kind"] == "layer"
    Q, K, V, beta, g = (st[k].flatten(0, 1) if dense else st[k] for k in ("Q", "K", "V", "beta", "g"))  # [tokens, H, ...]
    cu = [b * case["T"] for b in range(case["B"] + 1)] if dense else st["cu"]
    n_seq = len(cu) - 1
    S = torch.zeros(n_seq, H_v, D, D, dtype=torch.float64, device="cuda") if st["S"] is None else st["S"].double()
    O = torch.empty(V.shape, dtype=torch.float64, device="cuda")
    key = torch.arange(H_v, device="cuda") // (H_v // H_k)
    row = torch.arange(C, device="cuda")
    causal = torch.ones(C, C, dtype=torch.bool, device="cuda").tril()
    longest = max(cu[s + 1] - cu[s] for s in range(n_seq))
    for t0 in range(0, longest, C):  # the next chunk of every sequence that has one: [sequences, H_v, C, ...]
        alive = [s for s in range(n_seq) if cu[s] + t0 < cu[s + 1]]
        first = torch.tensor([cu[s] + t0 for s in alive], device="cuda")
        size = torch.tensor([min(C, cu[s + 1] - cu[s] - t0) for s in alive], device="cuda")
        real = row < size[:, None]
        at = torch.where(real, first[:, None] + row, first[:, None])
        # rows past a sequence's end write nothing: no key, no value, no further decay
        q, k = (torch.where(real[..., None, None], _unit(x[at]), 0.0)[:, :, key].transpose(1, 2) for x in (Q, K))
        v = torch.where(real[..., None, None], V[at].double(), 0.0).transpose(1, 2)
        b, gc = (torch.where(real[..., None], x[at].double(), 0.0).transpose(1, 2) for x in (beta, g))
        gc = gc.cumsum(-1)
        W, U, _ = _chunks(k, v, b, gc, C, gated=True)
        s0 = S[alive]
        u = U - W @ s0.transpose(-1, -2)
        P = (q @ k.transpose(-1, -2)) * torch.where(causal, gc[..., :, None] - gc[..., None, :], -torch.inf).exp()
        o = D ** -0.5 * (gc.exp()[..., None] * (q @ s0.transpose(-1, -2)) + P @ u)
        O[at[real]] = o.transpose(1, 2)[real]
        end = gc[..., -1:]
        S[alive] = end.exp()[..., None] * s0 + (u * (end - gc).exp()[..., None]).transpose(-1, -2) @ k
    return O.view(st["V"].shape), S


def exact(case, seed):
    """What `run` returns for these inputs, from the definitions in fp64 (the integer kinds are whole numbers already)."""
    if case["kind"] in ("int8", "int16"):
        return None
    st = prepare(case, seed)
    return _exact_prepare(case, st) if case["kind"] == "prepare" else _exact_layer(case, st)
