"""bf16 kernels whose warps take sixteen positions at a time, at the edges of their chunks, against the fp64 oracle under the bf16 gates:
causal, D = M = 32, a warp per piece of a sequence (whole and in pieces, ragged, from a state, with and without a saved buffer), and
non-causal, D = M = 32 and 64 (whole and split, ragged, with and without kept sums)."""
import os
import re

import numpy as np
import pytest
import torch

import oracle
import paper_2006_16236_b200 as la
from paper_2006_16236_b200.inputs import draw_qkvg
from parity import assert_close

DEV, BF, D = "cuda:0", torch.bfloat16, 32


@pytest.fixture(autouse=True)
def _automatic_plans():
    yield
    la.la_plan_override()


@pytest.mark.gpu
@pytest.mark.parametrize("pieces", [-1, 1, 2, 5])
@pytest.mark.parametrize("B,H,N", [(38, 8, 1), (38, 8, 15), (38, 8, 17), (38, 8, 63), (38, 8, 64), (38, 8, 65), (38, 8, 100), (38, 8, 128), (38, 8, 200),
                                   (56, 8, 200), (150, 8, 40), (1, 2, 2100), (2, 1, 2049 + 64)])
def test_pieces_lengths_and_states(B, H, N, pieces):
    Q, K, V, G = draw_qkvg(B, H, N, D, D, 7 + N, BF, 1.0)
    g = torch.Generator().manual_seed(N)
    S0, Z0 = torch.randn((B, H, D, D), generator=g) * 3.0, torch.rand((B, H, D), generator=g) * 4.0 + 1.0
    dSN, dZN = torch.randn((B, H, D, D), generator=g) * 0.05, torch.randn((B, H, D), generator=g) * 0.05
    lengths = [max(N - (7 * b) % (N + 1), 0) for b in range(B)]
    lengths[0] = N
    la.la_plan_override(pieces)
    dev = [t.to(DEV) for t in (Q, K, V, G)]
    st = {"S_in": S0.to(DEV), "Z_in": Z0.to(DEV)}
    ln = torch.tensor(lengths, dtype=torch.int32, device=DEV)
    for phi in ("elu1", "identity"):
        if phi == "identity":                           # features: positive, as the weights of a kernel are
            Q, K = (Q.float().abs() + 0.1).to(BF), (K.float().abs() + 0.1).to(BF)
            dev[:2] = Q.to(DEV), K.to(DEV)
        S, Z, den = torch.empty_like(st["S_in"]), torch.empty_like(st["Z_in"]), torch.empty(B, H, N, device=DEV)
        dS, dZ = torch.empty_like(S), torch.empty_like(Z)
        saved = la.saved_buffer(dev[0], dev[2], phi=phi)
        O = la.la_causal_forward(*dev[:3], phi=phi, lengths=ln, den=den, S_out=S, Z_out=Z, saved=saved, **st)
        kw = {"phi": phi, "lengths": ln, "dS_out": dSN.to(DEV), "dZ_out": dZN.to(DEV), **st}
        grads = la.la_causal_backward(*dev, saved=saved, dS_in=dS, dZ_in=dZ, **kw)
        again = la.la_causal_backward(*dev, **kw)       # the kept sums are those that it would make itself
        la.la_last_device_status()
        assert all(torch.equal(a, b) for a, b in zip(grads, again))
        for b in {0, min(1, B - 1), B - 1}:
            n, h = lengths[b], b % H
            assert not O[b, :, n:].any() and not den[b, :, n:].any() and not any(x[b, :, n:].any() for x in grads)
            sl = (slice(b, b + 1), slice(h, h + 1))
            s0, z0 = S0[sl].double().numpy(), Z0[sl].double().numpy()
            if n == 0:
                assert torch.equal(S[sl].cpu(), S0[sl]) and torch.equal(Z[sl].cpu(), Z0[sl])
                continue
            q, k, v, u = (t[sl][:, :, :n].double().numpy() for t in (Q, K, V, G))
            Or, denr, Sr, Zr = oracle.causal_from_state(q, k, v, s0, z0, phi=phi)
            for nm, x, ref in (("O", O[sl][:, :, :n], Or), ("den", den[sl][:, :, :n], denr), ("S_out", S[sl], Sr), ("Z_out", Z[sl], Zr)):
                assert_close(x, ref, BF, nm)
            refs = oracle.causal_backward_from_state(q, k, v, s0, z0, u, dSN[sl].double().numpy(), dZN[sl].double().numpy(), phi=phi)
            for nm, x, ref in zip(("dQ", "dK", "dV", "dS_in", "dZ_in"), [x[sl][:, :, :n] for x in grads] + [dS[sl], dZ[sl]], refs):
                assert_close(x, ref, BF, nm, grad=True)


@pytest.mark.gpu
def test_the_normaliser_divides_to_the_last_bit():
    """Features a, b along one axis and values chosen so that (a v0 + b v1) / (a + b) lies halfway between two bf16 numbers: all sums are
    exact, so the output is that of one correctly rounded fp32 reciprocal, a product and the rounding to bf16, to the bit.  (A
    reciprocal that is one fp32 bit off leaves the middle and may round the other way.)"""
    rng, heads = np.random.default_rng(0), 512
    a, b, v0, v1 = (np.zeros(s, np.float32) for s in ((heads,), (heads,), (heads, D), (heads, D)))
    n0, n1 = np.meshgrid(np.arange(129, 256, 2), np.arange(128, 256))           # v0 = n0 / 256, v1 = n1 / 128
    for h in range(heads):
        found = np.zeros(0, np.int64)
        while len(found) < D:
            a[h], b[h] = 2 * rng.integers(64) + 1, 2 * rng.integers(1, 256)
            total = (a[h] * n0 + 2 * b[h] * n1).astype(np.int64).ravel()
            r, rest = np.divmod(total, int(a[h] + b[h]))
            found = np.nonzero((rest == 0) & (r % 2 == 1) & (r > 256) & (r < 512))[0]       # an odd number of 1/256, between 1 and 2
        at = rng.permutation(found)[:D]
        v0[h], v1[h] = n0.ravel()[at] / 256, n1.ravel()[at] / 128
    Q, K, V = (torch.zeros(1, heads, 2, D) for _ in range(3))
    Q[..., 0], K[0, :, 0, 0], K[0, :, 1, 0], V[0, :, 0], V[0, :, 1] = 1.0, *map(torch.from_numpy, (a, b, v0, v1))
    Qd, Kd, Vd = (t.to(DEV, BF) for t in (Q, K, V))
    assert all(torch.equal(x.cpu().float(), t) for x, t in zip((Qd, Kd, Vd), (Q, K, V)))
    O = la.la_causal_forward(Qd, Kd, Vd, phi="identity", eps=0.0)
    inv = np.float32(1.0) / (a + b)
    want = torch.from_numpy((a[:, None] * v0 + b[:, None] * v1) * inv[:, None]).to(BF)
    assert torch.equal(O[0, :, 1].cpu(), want)


@pytest.mark.gpu
@pytest.mark.parametrize("pieces,N", [(2, 128), (2, 512), (5, 512)])
@pytest.mark.parametrize("phi", ["elu1", "identity"])
def test_sums_of_pieces_are_those_of_the_sweep(phi, pieces, N):
    """The gradient of the initial state is the sum of phi(q) / dn G over all positions: what the reverse sweep adds up itself where a
    sequence is one piece, and what records of the pieces hold where it is several.  Both round phi(q) / dn to bf16 once, so that they
    differ by the order of fp32 additions, and by the few operands that an fp32 bit of dn takes over a rounding boundary: 2^-24 of
    2^-8, one in 2^16, each off by 2^-8 of itself, 2^-16 of the whole.  Rounded twice they are 2^-9 apart."""
    B, H = 38, 8
    Q, K, V, G = draw_qkvg(B, H, N, D, D, 3, BF, 1.0)
    if phi == "identity":
        Q, K = (Q.float().abs() + 0.1).to(BF), (K.float().abs() + 0.1).to(BF)
    dev = [t.to(DEV) for t in (Q, K, V, G)]
    S0, Z0, got = torch.ones(B, H, D, D, device=DEV), torch.full((B, H, D), 3.0, device=DEV), []
    for n in (1, pieces):
        la.la_plan_override(n)
        dS, dZ = torch.empty_like(S0), torch.empty_like(Z0)
        la.la_causal_backward(*dev, phi=phi, S_in=S0, Z_in=Z0, dS_in=dS, dZ_in=dZ)
        got.append(dS)
    assert float((got[1] - got[0]).norm() / got[0].norm()) < 2.0 ** -14


@pytest.mark.gpu
@pytest.mark.parametrize("pieces", [1, 2])
def test_dq_of_near_uniform_weights(pieces):
    """With queries and keys close to zero dQ is a small difference of large sums.  Against 64 bits, what the rounding of the features
    alone leaves (rows 16 to 63, whose scores and sums are treated so that nothing else matters) is what every row up to 191 has;
    with the sums rounded to bf16 it is a third more."""
    B, H, N = 38, 8, 256
    Q, K, V, G = draw_qkvg(B, H, N, D, D, 5, BF, 0.125)
    la.la_plan_override(pieces)
    dQ = la.la_causal_backward(*(t.to(DEV) for t in (Q, K, V, G)))[0][:4].double().cpu().numpy()
    want = oracle.linear_attention_backward(*(t[:4].double().numpy() for t in (Q, K, V, G)), causal=True)[0]
    off = lambda lo, hi: np.linalg.norm((dQ - want)[:, :, lo:hi]) / np.linalg.norm(want[:, :, lo:hi])
    assert off(64, 192) < 1.1 * off(16, 64)


@pytest.mark.gpu
@pytest.mark.parametrize("splits", [-1, 1, 3])
@pytest.mark.parametrize("W", [32, 64])
@pytest.mark.parametrize("N", [1, 15, 17, 256, 257, 500, 900])
def test_noncausal_chunks_and_splits(N, W, splits):
    B, H = 5, 8
    Q, K, V, G = draw_qkvg(B, H, N, W, W, 11 + N, BF, 0.5)
    lengths = [N, 0, (N + 1) // 2, max(N - 1, 1), min(N, 16)]
    la.la_plan_override(-1, -1, splits)
    for phi in ("elu1", "identity"):
        if phi == "identity":
            Q, K = (Q.float().abs() + 0.1).to(BF), (K.float().abs() + 0.1).to(BF)
        dev = [t.to(DEV) for t in (Q, K, V, G)]
        for ln in (None, torch.tensor(lengths, dtype=torch.int32, device=DEV)):
            saved = la.linear_saved_buffer(dev[0], dev[2], phi=phi)
            den, KV, Zs = torch.empty(B, H, N, device=DEV), torch.empty(B, H, W, W, device=DEV), torch.empty(B, H, W, device=DEV)
            # (a clustered forward pass is another kernel's matter: with forced splits it is this one)
            O = la.la_linear_attention(*dev[:3], phi=phi, lengths=ln, saved=saved, den=den, KV=KV, Zs=Zs)
            grads = la.la_linear_attention_backward(*dev, phi=phi, lengths=ln, saved=saved)
            again = la.la_linear_attention_backward(*dev, phi=phi, lengths=ln)
            la.la_last_device_status()
            assert all(torch.equal(a, b) for a, b in zip(grads, again))
            for b in range(B):
                n, h = N if ln is None else lengths[b], b
                assert not O[b, :, n:].any() and not den[b, :, n:].any() and not any(x[b, :, n:].any() for x in grads)
                if n == 0:
                    assert not KV[b].any() and not Zs[b].any()
                    continue
                sl = (slice(b, b + 1), slice(h, h + 1), slice(0, n))
                q, k, v, u = (t[sl].double().numpy() for t in (Q, K, V, G))
                Or, denr = oracle.linear_attention(q, k, v, causal=False, phi=phi)[:2]
                fk = oracle.feature_map(k) if phi == "elu1" else k
                for nm, x, ref in (("O", O[sl], Or), ("den", den[sl], denr), ("KV", KV[b, h], np.einsum("nd,nm->dm", fk[0, 0], v[0, 0])),
                                   ("Zs", Zs[b, h][None], fk[0, 0].sum(0)[None])):
                    assert_close(x, ref, BF, nm)
                if n == 1:
                    continue                            # dQ and dK are analytically zero
                for nm, x, ref in zip(("dQ", "dK", "dV"), grads, oracle.linear_attention_backward(q, k, v, u, causal=False, phi=phi)):
                    assert_close(x[sl], ref, BF, nm, grad=True)


@pytest.mark.gpu
def test_kept_sums_of_another_plan_are_refused():
    if os.environ.get("LA_DEBUG"):
        pytest.skip("in checked mode the call itself reads the status and raises; this test reads it afterwards")
    dev = [t.to(DEV) for t in draw_qkvg(2, 4, 2200, D, D, 3, BF, 1.0)]
    la.la_plan_override(3)
    saved = torch.zeros(1 << 20, dtype=torch.uint8, device=DEV)
    la.la_causal_forward(*dev[:3], saved=saved)
    la.la_plan_override(4)
    dQ, dK, dV = (torch.full_like(dev[0], 7.0) for _ in range(3))
    la.la_causal_backward(*dev, saved=saved, dQ=dQ, dK=dK, dV=dV)
    with pytest.raises(la.LaError) as e:
        la.la_last_device_status()
    assert e.value.status == -1 and "plan" in str(e.value)
    assert torch.all(dQ == 7.0) and torch.all(dK == 7.0) and torch.all(dV == 7.0)


@pytest.mark.gpu
def test_steps_enqueued_behind_each_other():
    """Forward and backward passes of small grids start as programmatic dependents of each other; inputs change in between."""
    data = [[t.to(DEV) for t in draw_qkvg(1, 2, 2100, D, D, 20 + i, BF, 1.0)] for i in range(6)]
    step = lambda x, s: (la.la_causal_forward(*x[:3], saved=s), *la.la_causal_backward(*x, saved=s))
    want = []
    for x in data:
        want.append(step(x, la.saved_buffer(x[0], x[2])))
        torch.cuda.synchronize()
    buf, saved, got = [torch.empty_like(t) for t in data[0]], la.saved_buffer(data[0][0], data[0][2]), []
    for x in data:
        for a, b in zip(buf, x):
            a.copy_(b)
        got.append(step(buf, saved))
    torch.cuda.synchronize()
    assert all(torch.equal(a, b) for w, g in zip(want, got) for a, b in zip(w, g))


def test_workspace_and_saved_sizes():
    """Sequences in pieces need room for their sums, and keep them for a training step; whole ones, and forward passes that are one kernel,
    nothing."""
    p = lambda *s: la.make_problem(*s, 32, 32, la.LA_BF16)
    size = lambda q, op: la.la_workspace_bytes(q, op)
    assert size(p(8, 8, 3072), la.LA_OP_CAUSAL_FORWARD) > 0 and size(p(8, 8, 3072), la.LA_OP_CAUSAL_SAVED) > 0
    assert size(p(16, 8, 3072), la.LA_OP_CAUSAL_FORWARD) == 0 and size(p(16, 8, 3072), la.LA_OP_CAUSAL_SAVED) > 0
    assert size(p(128, 8, 784), la.LA_OP_CAUSAL_SAVED) == 0 and size(p(60, 8, 784), la.LA_OP_CAUSAL_SAVED) > 0


@pytest.mark.gpu
@pytest.mark.parametrize("BH,N,tcgen05", [(128, 512, True), (112, 1000, True), (100, 1000, False), (148, 300, True), (149, 512, False), (90, 512, True),
                                          (76, 1024, False)], ids=str)
@pytest.mark.parametrize("phi", ["elu1", "identity"])
def test_forward_passes_that_keep_no_sums(BH, N, tcgen05, phi):
    """A wave of one tcgen05 CTA per sequence takes them; training steps, which keep sums, stay on warps.  Both to the same gates, from a
    state; the identity map with lengths."""
    B, H = BH, 1
    Q, K, V, _ = draw_qkvg(B, H, N, D, D, 3, BF, 1.0, with_grad=False)
    if phi == "identity":
        Q, K = (Q.float().abs() + 0.1).to(BF), (K.float().abs() + 0.1).to(BF)
    g = torch.Generator().manual_seed(1)
    S0, Z0 = torch.randn((B, H, D, D), generator=g) * 3.0, torch.rand((B, H, D), generator=g) * 4.0 + 1.0
    dev, st = [t.to(DEV) for t in (Q, K, V)], {"S_in": S0.to(DEV), "Z_in": Z0.to(DEV)}
    lengths = [N] * B if phi == "elu1" else [(N - 37 * b) % (N + 1) for b in range(B)]
    ln = None if phi == "elu1" else torch.tensor(lengths, dtype=torch.int32, device=DEV)
    for saved in (None, la.saved_buffer(dev[0], dev[2], phi=phi)):
        S, Z, den = torch.empty_like(st["S_in"]), torch.empty_like(st["Z_in"]), torch.empty(B, H, N, device=DEV)
        la.la_profile_enable(True)
        O = la.la_causal_forward(*dev, phi=phi, lengths=ln, den=den, S_out=S, Z_out=Z, saved=saved, **st)
        la.la_last_device_status()
        names = set(la.la_profile_read())
        la.la_profile_enable(False)
        assert ("causal_fwd_kernel" in names) == (tcgen05 and saved is None) and ("causal_mma_forward_kernel" in names) != ("causal_fwd_kernel" in names)
        for b in (0, 1, B - 1):
            n = lengths[b]
            q, k, v = (t[b:b + 1, :, :n].double().numpy() for t in (Q, K, V))
            ref = oracle.causal_from_state(q, k, v, S0[b:b + 1].double().numpy(), Z0[b:b + 1].double().numpy(), phi=phi)
            assert not O[b, :, n:].any() and not den[b, :, n:].any()
            for nm, x, r in (("O", O[b:b + 1, :, :n], ref[0]), ("den", den[b:b + 1, :, :n], ref[1]), ("S_out", S[b:b + 1], ref[2]), ("Z_out", Z[b:b + 1], ref[3])):
                assert_close(x, r, BF, nm)


@pytest.mark.parametrize("BHN,pieces", [((50, 8, 2048), 8), ((444, 1, 512), 4), ((592, 1, 784), 2), ((500, 1, 100), 1), ((560, 1, 128), 1), ((180, 1, 192), 3),
                                        ((900, 1, 784), 1), ((128, 1, 3072), 8), ((4, 1, 4096), 32)], ids=str)
def test_numbers_of_pieces(BHN, pieces):
    """What was measured best, or within 3 % of it: just past a full wave of warps, two chunks, many sequences, few."""
    p = la.make_problem(*BHN, 32, 32, la.LA_BF16)
    kept = la.la_workspace_bytes(p, la.LA_OP_CAUSAL_SAVED)
    assert (kept - 16 if kept else 0) == BHN[0] * BHN[1] * (pieces - 1) * 32 * 33 * 4


def test_no_read_only_loads():
    """As the other kernels that may start as programmatic dependents."""
    for name in ("la_warp.cuh", "la_causal_warp.cuh", "la_linear_warp.cuh"):
        code = re.sub(r"//[^\n]*", "", open(os.path.join(os.path.dirname(la.__file__), "csrc", name)).read())
        assert not re.findall(r"__ldg\s*\(|ld\.global\.nc|const \w+\s*\*\s*__restrict__", code)
