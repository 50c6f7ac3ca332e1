"""What is timed when the speed of this library is compared between two versions of it.

A case is one pass through the public calls of ``paper_2006_16236_b200`` as a program makes them: a training step
(forward and backward), an encoder's forward pass, a prompt continued from a state, one token of a generation loop.
``listed()`` has the named ones, ``draw()`` gives others of the same ranges.  Sizes are those of the repository's
workloads, benchmark rows and tests; inputs are i.i.d. normal like theirs, drawn on the GPU from the seed.
"""
from __future__ import annotations

import math

import torch

import paper_2006_16236_b200 as la

DTYPES = {"bf16": torch.bfloat16, "f32": torch.float32}


def listed():
    return [
        # ---- generation ----------------------------------------------------------------------------------------
        # one token for one sequence: eight states, a call whose cost is latency and host work
        {"name": "decode_one_stream", "kind": "step", "B": 1, "H": 8, "D": 64, "M": 64, "dtype": "bf16", "prepared": False},
        # one token for 256 sequences at once, the loop of a server whose buffers stay where they are
        {"name": "decode_256_streams", "kind": "step", "B": 256, "H": 8, "D": 64, "M": 64, "dtype": "bf16", "prepared": True},
        # the same token with the projections of the attention sublayer around it
        {"name": "decode_layer_256_streams", "kind": "layer", "B": 256, "H": 8, "D": 64},
        # a prompt that arrives in pieces: one piece of one sequence, continued from the state of the piece before
        {"name": "prefill_piece", "kind": "prefill", "B": 1, "H": 8, "N": 2048, "D": 64, "M": 64, "dtype": "bf16"},
        # ---- causal training -----------------------------------------------------------------------------------
        # 28 x 28 pixel sequences in large batches: short, not a whole number of 128-position chunks
        {"name": "train_pixels_784", "kind": "causal", "B": 128, "H": 8, "N": 784, "D": 32, "M": 32, "dtype": "bf16"},
        # 32 x 32 x 3 pixel sequences
        {"name": "train_image_3072", "kind": "causal", "B": 16, "H": 8, "N": 3072, "D": 32, "M": 32, "dtype": "bf16"},
        # the long-sequence point of the sequence-length benchmark
        {"name": "train_long_16384", "kind": "causal", "B": 8, "H": 8, "N": 16384, "D": 64, "M": 64, "dtype": "bf16"},
        # the smallest problem that is trained in fp32 (a check of a model before it is scaled up): latency
        {"name": "train_fp32_256", "kind": "causal", "B": 1, "H": 2, "N": 256, "D": 32, "M": 32, "dtype": "f32"},
        # the N = 4096 point of the sequence-length benchmark trained in fp32
        {"name": "train_fp32_4096", "kind": "causal", "B": 32, "H": 8, "N": 4096, "D": 64, "M": 64, "dtype": "f32"},
        # another kernel: queries and keys through 128 random Fourier features, gradients back through both steps
        {"name": "train_fourier_1000", "kind": "fourier", "B": 8, "H": 8, "N": 1000, "D": 64, "C": 128, "M": 64},
        # ---- bidirectional encoder -----------------------------------------------------------------------------
        # a training step of a speech encoder on utterances of different lengths, padded to the longest
        {"name": "train_encoder_ragged_4096", "kind": "encoder", "B": 8, "H": 8, "N": 4096, "D": 64, "M": 64, "dtype": "bf16",
         "ragged": True},
        # one utterance encoded: the forward pass alone
        {"name": "encode_one_1000", "kind": "encode", "B": 1, "H": 8, "N": 1000, "D": 64, "M": 64, "dtype": "bf16",
         "ragged": False},
    ]


def _log_int(rng, lo, hi):
    """A whole number between lo and hi, spread evenly over the logarithm: every size is possible, odd ones too."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _batch(rng, most):
    """(B, H) with B * H at most `most`."""
    H = rng.choice([2, 4, 8, 8, 12, 16])
    H = min(H, most)
    return _log_int(rng, 1, max(1, most // H)), H


def draw(rng):
    """Another case of the ranges that the listed ones stand for; none moves more than train_fp32_4096 or
    multiplies more."""
    kind = rng.choice(["step", "layer", "prefill", "causal", "causal", "causal", "causal_f32", "causal_f32", "fourier",
                       "encoder", "encode"])
    if kind == "step":          # 1 to 2048 sequences with 8 heads
        B = _log_int(rng, 1, 2048)
        D = rng.choice([32, 64, 64])
        return {"kind": "step", "B": B, "H": 8, "D": D, "M": D, "dtype": rng.choice(["bf16", "bf16", "f32"]),
                "prepared": rng.random() < 0.5}
    if kind == "layer":
        return {"kind": "layer", "B": _log_int(rng, 1, 1024), "H": rng.choice([4, 8, 12]), "D": 64}
    if kind == "prefill":
        D = rng.choice([32, 64, 64])
        N = _log_int(rng, 128, 16384)
        B = _log_int(rng, 1, max(1, min(16, 65536 // N)))
        return {"kind": "prefill", "B": B, "H": 8, "N": N, "D": D, "M": D, "dtype": "bf16"}
    if kind == "causal":
        D = rng.choice([32, 64])
        N = _log_int(rng, 256, 65536)
        B, H = _batch(rng, max(2, (1 << 20) // N))
        return {"kind": "causal", "B": B, "H": H, "N": N, "D": D, "M": D, "dtype": "bf16"}
    if kind == "causal_f32":    # any head size that is a multiple of eight
        D = rng.choice([32, 64, 64, 8 * rng.randint(2, 12)])
        M = rng.choice([D, D, 8 * rng.randint(2, 8)])
        N = _log_int(rng, 64, 4096)
        B, H = _batch(rng, max(2, (1 << 20) * 64 * 64 // (N * max(D * M, 4096))))
        return {"kind": "causal", "B": min(B, 32), "H": min(H, 8), "N": N, "D": D, "M": M, "dtype": "f32"}
    if kind == "fourier":
        N = _log_int(rng, 128, 4096)
        return {"kind": "fourier", "B": _log_int(rng, 1, max(1, 16384 // N)), "H": 8, "N": N, "D": rng.choice([32, 64]),
                "C": 128, "M": 64}
    if kind == "encoder":
        D = rng.choice([32, 64, 64])
        N = _log_int(rng, 256, 8192)
        dtype = rng.choice(["bf16", "bf16", "f32"])
        return {"kind": "encoder", "B": _log_int(rng, 1, max(1, min(64, 32768 // N))), "H": 8, "N": N, "D": D, "M": D,
                "dtype": dtype, "ragged": rng.random() < 0.5}
    D = rng.choice([32, 64, 64])
    N = _log_int(rng, 64, 8192)
    return {"kind": "encode", "B": _log_int(rng, 1, max(1, min(64, 32768 // N))), "H": 8, "N": N, "D": D, "M": D, "dtype": "bf16",
            "ragged": rng.random() < 0.5}


def _lengths(case, g):
    """Half to the whole of N, evenly spread over the batch, in an order of the seed's."""
    B, N = case["B"], case["N"]
    if not case.get("ragged"):
        return None
    spread = torch.tensor([N - (N // 2) * b // B for b in range(B)], dtype=torch.int32, device="cuda")
    return spread[torch.randperm(B, generator=g, device="cuda")].contiguous()


def prepare(case, seed):
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    kind, B, H, D = case["kind"], case["B"], case["H"], case["D"]
    M = case.get("M", D)
    dtype = DTYPES[case.get("dtype", "bf16")]

    def normal(*shape, scale=1.0, dtype=dtype):
        return (torch.randn(shape, generator=g, device="cuda") * scale).to(dtype)

    def state():
        """What some hundred positions of unit-normal keys and values leave behind."""
        S = normal(B, H, D, M, scale=15.0, dtype=torch.float32)
        Z = normal(B, H, D, scale=10.0, dtype=torch.float32) + 120.0
        return S, Z

    s = {"kind": kind}
    if kind == "step":
        s["q"], s["k"], s["v"] = normal(B, H, D), normal(B, H, D), normal(B, H, M)
        s["S"], s["Z"] = state()
        if case["prepared"]:
            s["call"] = la.prepare_recurrent_step(s["q"], s["k"], s["v"], s["S"], s["Z"])
    elif kind == "layer":
        F = H * D
        s["x"] = normal(B, F)
        s["Wqkv"], s["Wo"] = normal(3 * F, F, scale=F ** -0.5), normal(F, F, scale=F ** -0.5)
        s["S"], s["Z"] = state()
    elif kind == "prefill":
        N = case["N"]
        s["Q"], s["K"], s["V"] = normal(B, H, N, D), normal(B, H, N, D), normal(B, H, N, M)
        s["S"], s["Z"] = state()
    elif kind == "fourier":
        N = case["N"]
        s["Q"], s["K"] = normal(B, H, N, D, scale=0.05), normal(B, H, N, D, scale=0.05)
        s["V"], s["G"] = normal(B, H, N, M), normal(B, H, N, M)
        s["W"] = normal(case["C"] // 2, D)
    else:
        N = case["N"]
        scale = 0.125 if kind in ("encoder", "encode") else 1.0
        s["Q"], s["K"], s["V"] = (normal(B, H, N, c, scale=scale) for c in (D, D, M))
        if kind != "encode":
            s["G"] = normal(B, H, N, M)
        s["lengths"] = _lengths(case, g)
    return s


def run(s):
    kind = s["kind"]
    if kind == "step":
        out = s["call"]() if "call" in s else la.la_recurrent_step(s["q"], s["k"], s["v"], s["S"], s["Z"])
        return out, s["S"], s["Z"]
    if kind == "layer":
        return la.la_decode_layer_step(s["x"], s["Wqkv"], s["Wo"], s["S"], s["Z"]), s["S"], s["Z"]
    Q, K, V = s["Q"], s["K"], s["V"]
    if kind == "prefill":
        S, Z = torch.empty_like(s["S"]), torch.empty_like(s["Z"])
        return la.la_causal_forward(Q, K, V, S_in=s["S"], Z_in=s["Z"], S_out=S, Z_out=Z), S, Z
    if kind == "causal":
        saved = la.saved_buffer(Q, V)
        O = la.la_causal_forward(Q, K, V, saved=saved)
        return (O, *la.la_causal_backward(Q, K, V, s["G"], saved=saved))
    if kind == "fourier":
        fQ, fK = la.la_feature_map_rff(Q, s["W"]), la.la_feature_map_rff(K, s["W"])
        O = la.la_causal_forward(fQ, fK, V, phi="identity")
        dfQ, dfK, dV = la.la_causal_backward(fQ, fK, V, s["G"], phi="identity")
        return (O, la.la_feature_map_rff_backward(Q, s["W"], dfQ), la.la_feature_map_rff_backward(K, s["W"], dfK), dV)
    if kind == "encoder":
        saved = la.linear_saved_buffer(Q, V)
        O = la.la_linear_attention(Q, K, V, lengths=s["lengths"], saved=saved)
        return (O, *la.la_linear_attention_backward(Q, K, V, s["G"], lengths=s["lengths"], saved=saved))
    return la.la_linear_attention(Q, K, V, lengths=s["lengths"])


def work(case):
    """Every input read once and every output written once (of a padded batch: the real positions of the inputs,
    all of the outputs); multiply-adds of the linear recurrence, two operations each."""
    kind, B, H, D = case["kind"], case["B"], case["H"], case["D"]
    M = case.get("M", D)
    e = 4 if case.get("dtype") == "f32" else 2
    state = B * H * D * (M + 1) * 4
    if kind == "step":
        return {"bytes": 2 * state + B * H * (2 * D + 2 * M) * e, "flops": 4 * B * H * D * M}
    if kind == "layer":
        F = H * D
        return {"bytes": 2 * state + 4 * F * F * e + 2 * B * F * e, "flops": 8 * B * F * F + 4 * B * H * D * M}
    rows = B * H * case["N"]
    if kind == "prefill":
        return {"bytes": 2 * state + rows * (2 * D + 2 * M) * e, "flops": 4 * rows * D * M}
    if kind == "fourier":
        C = case["C"]
        return {"bytes": rows * (4 * D + 4 * M) * e, "flops": rows * (14 * C * M + 2 * 2 * D * C)}
    real = rows
    if case.get("ragged"):
        real = H * sum(case["N"] - (case["N"] // 2) * b // B for b in range(B))
    if kind == "encode":
        return {"bytes": (real * (2 * D + M) + rows * M) * e, "flops": 4 * real * D * M}
    return {"bytes": (real * (2 * D + 2 * M) + rows * (2 * D + 2 * M)) * e,
            "flops": (14 if kind == "causal" else 12) * real * D * M}


def tolerance(case):
    """About four times the error measured on a B200 against the same formulas in 64 bits (2-norm, and the largest
    element over max(rms, |value|)).  bf16 training: gradients come from products of bf16 features, 4.8e-3 and 0.3 were
    seen (the last bit of a small gradient next to large ones); forward passes and decode steps end in one bf16
    rounding, 1.7e-3 to 2.3e-3 and 3.9e-3 to 1.2e-2.  fp32: 7.6e-7 and 2.5e-5 in the causal form, 3e-6 and 2.7e-5 in the
    bidirectional one, whose near-uniform weights cancel in dQ."""
    kind, f32 = case["kind"], case.get("dtype") == "f32"
    if kind == "step":
        return {"rel": 1e-6, "max": 1e-5} if f32 else {"rel": 7e-3, "max": 1.6e-2}
    if kind == "layer":
        return {"rel": 8e-3, "max": 2e-2}
    if kind in ("prefill", "encode"):
        return {"rel": 1e-2, "max": 5e-2}
    if kind == "fourier":
        return {"rel": 1.1e-2, "max": 0.35}
    if kind == "encoder":
        return {"rel": 1.2e-5, "max": 1.2e-4} if f32 else {"rel": 1.2e-2, "max": 6e-2}
    return {"rel": 4e-6, "max": 1e-4} if f32 else {"rel": 2e-2, "max": 0.9}


def _phi(x):
    return torch.where(x > 0, x + 1, torch.exp(torch.clamp(x, max=0.0)))


def _slope(x):
    return torch.where(x > 0, torch.ones_like(x), torch.exp(torch.clamp(x, max=0.0)))


def _ones(V):
    """The values with a column of ones: its sums are the normaliser."""
    return torch.cat([V, torch.ones_like(V[..., :1])], -1)


def _upstream(nd, G):
    """Gradient of the numerator and of the normaliser from that of the output."""
    dn, O = nd[..., -1:], nd[..., :-1] / nd[..., -1:]
    return torch.cat([G, -(G * O).sum(-1, keepdim=True)], -1) / dn


def _causal(q, k, V, G=None, St=None, T=128):
    """O, the final [S | Z] and, with G, the gradients of q, k (features) and V, chunk by chunk."""
    Vt, N = _ones(V), q.shape[2]
    St = torch.zeros_like(q[:, :, 0, :, None] * Vt[:, :, 0, None, :]) if St is None else St.clone()
    nd, gq, gk, gV, Gt = torch.empty_like(Vt), torch.empty_like(q), torch.empty_like(k), torch.empty_like(Vt), None
    if G is not None:
        Gt = torch.empty_like(Vt)
    cuts = [slice(i, min(i + T, N)) for i in range(0, N, T)]
    for c in cuts:
        qc, kc, vc = q[:, :, c], k[:, :, c], Vt[:, :, c]
        nd[:, :, c] = (qc @ kc.mT).tril() @ vc + qc @ St
        if G is not None:
            Gt[:, :, c] = _upstream(nd[:, :, c], G[:, :, c])
            gq[:, :, c] = (Gt[:, :, c] @ vc.mT).tril() @ kc + Gt[:, :, c] @ St.mT
        St += kc.mT @ vc
    O = nd[..., :-1] / nd[..., -1:]
    if G is None:
        return O, St
    R = torch.zeros_like(St)
    for c in reversed(cuts):
        qc, kc, vc, gc = q[:, :, c], k[:, :, c], Vt[:, :, c], Gt[:, :, c]
        gk[:, :, c] = (gc @ vc.mT).tril().mT @ qc + vc @ R.mT
        gV[:, :, c] = (qc @ kc.mT).tril().mT @ gc + kc @ R
        R += qc.mT @ gc
    return O, gq, gk, gV[..., :-1]


def exact(case, seed):
    """What run() returns, in 64 bits from the formulas of the method."""
    s = {n: t.double() if torch.is_tensor(t) and t.is_floating_point() else t for n, t in prepare(case, seed).items()}
    kind = case["kind"]
    if kind in ("step", "layer"):
        B, H, D = case["B"], case["H"], case["D"]
        if kind == "layer":
            q, k, v = (s["x"] @ s["Wqkv"].mT).view(B, 3, H, D).unbind(1)
        else:
            q, k, v = s["q"], s["k"], s["v"]
        q, k = _phi(q), _phi(k)
        S, Z = s["S"] + k[..., :, None] * v[..., None, :], s["Z"] + k
        out = (q[..., None, :] @ S)[..., 0, :] / (q * Z).sum(-1, keepdim=True)
        if kind == "layer":
            out = out.reshape(B, H * D) @ s["Wo"].mT + s["x"]
        return out, S, Z
    Q, K, V = s["Q"], s["K"], s["V"]
    if kind == "prefill":
        O, St = _causal(_phi(Q), _phi(K), V, St=torch.cat([s["S"], s["Z"][..., None]], -1))
        return O, St[..., :-1], St[..., -1]
    if kind == "causal":
        O, gq, gk, gV = _causal(_phi(Q), _phi(K), V, s["G"])
        return O, gq * _slope(Q), gk * _slope(K), gV
    if kind == "fourier":
        W, a = s["W"], s["W"].shape[0] ** -0.5             # sqrt(2 / C): C / 2 frequencies
        zq, zk = Q @ W.mT, K @ W.mT
        fq, fk = (a * torch.cat([z.cos(), z.sin()], -1) for z in (zq, zk))
        O, gq, gk, gV = _causal(fq, fk, V, s["G"])
        half = W.shape[0]
        dQ, dK = (a * (z.cos() * g[..., half:] - z.sin() * g[..., :half]) @ W for z, g in ((zq, gq), (zk, gk)))
        return O, dQ, dK, gV
    q, k, Vt = _phi(Q), _phi(K), _ones(V)
    real = torch.ones_like(q[..., :1])
    if s["lengths"] is not None:        # padded positions: no part in any sum, zeros in every output
        real = (torch.arange(Q.shape[2], device="cuda") < s["lengths"][:, None]).to(q.dtype)[:, None, :, None].expand_as(real)
    k = k * real
    St = k.mT @ (Vt * real)
    nd = q @ St
    O = nd[..., :-1] / nd[..., -1:] * real
    if kind == "encode":
        return O
    Gt = _upstream(nd, s["G"]) * real
    R = (q * real).mT @ Gt
    return O, Gt @ St.mT * _slope(Q), Vt @ R.mT * _slope(K) * real, (k @ R)[..., :-1]
