"""Calls at fp32 accuracy on the warp-level tensor instructions: shapes at the edges of their tiles (chunks of
64 positions, strips of 16, columns padded to 32, 64 or 128), with the sequence whole and cut into pieces, from a state,
ragged, and without the optional workspace, against the fp64 oracle.

Tolerance (2-norm of the difference over the 2-norm of the result): an operand keeps 24 bits (2^-24), the tensor cores
truncate a running sum once per 16 terms (2^-23 of it, at most 8 blocks per sum), and the chunks' sums are added in
fp32: 16 * 2^-23 = 2e-6 bounds fp32 outputs whose terms do not cancel; gradients are differences of terms up to a few
times their size, so 8e-6.  bf16 outputs end in one rounding: 2^-8."""
import numpy as np
import pytest
import torch

import oracle
import paper_2006_16236_b200 as la
from paper_2006_16236_b200.inputs import draw_qkvg
from parity import assert_close

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.fixture(autouse=True)
def _automatic_plans():
    yield
    la.la_plan_override()


def _close(x, ref, tol, what):
    x, ref = x.double().cpu().numpy(), np.asarray(ref)
    scale = np.linalg.norm(ref)
    assert np.linalg.norm(x - ref) <= tol * scale + 1e-30, (what, np.linalg.norm(x - ref) / scale)


@pytest.mark.parametrize("pieces", [-1, 1, 3])
@pytest.mark.parametrize("N", [2, 16, 63, 64, 65, 200])
@pytest.mark.parametrize("dims", [(8, 8), (32, 32), (40, 24), (64, 64), (72, 64), (128, 64)], ids=str)
def test_tiles(dims, N, pieces):
    D, M = dims
    for dtype, phi in ((torch.float32, "elu1"), (torch.float32, "identity"), (torch.bfloat16, "identity"), (torch.bfloat16, "elu1")):
        if dtype == torch.bfloat16 and D == M and D in (32, 64):
            continue                                    # another kernel's problem
        Q, K, V, G = draw_qkvg(1, 2, N, D, M, 3 + N, dtype, 1.0)
        if phi == "identity":                           # features: positive, as the weights of a kernel are
            Q, K = Q.abs() + 0.1, K.abs() + 0.1
        la.la_plan_override(pieces)
        dev = [t.to(DEV) for t in (Q, K, V, G)]
        eps = 0.5 if N % 2 else 0.0
        O = la.la_causal_forward(*dev[:3], phi=phi, eps=eps)
        grads = la.la_causal_backward(*dev, phi=phi, eps=eps)
        la.la_last_device_status()
        q, k, v, g = (t.double().numpy() for t in (Q, K, V, G))
        f32 = dtype == torch.float32
        _close(O, oracle.linear_attention(q, k, v, causal=True, phi=phi, eps=eps)[0], 2e-6 if f32 else 2 ** -8, "O")
        for nm, x, ref in zip(("dQ", "dK", "dV"), grads, oracle.linear_attention_backward(q, k, v, g, causal=True, phi=phi, eps=eps)):
            _close(x, ref, 8e-6 if f32 else 2 ** -8, nm)


@pytest.mark.parametrize("pieces", [1, 2, 4])
def test_state_lengths_and_no_workspace(pieces):
    B, H, N, D, M = 3, 2, 150, 48, 40
    lengths = [150, 0, 70]
    Q, K, V, _ = draw_qkvg(B, H, N, D, M, 5, torch.float32, 1.0)
    la.la_plan_override(pieces)
    q, k, v = (t.to(DEV) for t in (Q, K, V))
    S0 = torch.rand(B, H, D, M, device=DEV)
    Z0 = torch.rand(B, H, D, device=DEV) + 1
    S, Z = torch.empty_like(S0), torch.empty_like(Z0)
    ln = torch.tensor(lengths, dtype=torch.int32, device=DEV)
    empty = torch.empty(0, dtype=torch.uint8, device=DEV)       # no room for records: one piece, the same sums
    for ws in (None, empty):
        O = la.la_causal_forward(q, k, v, S_in=S0, Z_in=Z0, S_out=S, Z_out=Z, lengths=ln, ws=ws)
        la.la_last_device_status()
        fk, fq = oracle.feature_map(K.double().numpy()), oracle.feature_map(Q.double().numpy())
        for b, n in enumerate(lengths):
            assert not O[b, :, n:].any()
            St = S0[b].double().cpu().numpy() + np.einsum("hnd,hnm->hdm", fk[b, :, :n], V[b, :, :n].double().numpy())
            Zt = Z0[b].double().cpu().numpy() + fk[b, :, :n].sum(1)
            _close(S[b], St, 2e-6, "S_out")
            _close(Z[b], Zt, 2e-6, "Z_out")
            if n:
                w = np.tril(np.einsum("hnd,hjd->hnj", fq[b, :, :n], fk[b, :, :n]))
                num = w @ V[b, :, :n].double().numpy() + fq[b, :, :n] @ S0[b].double().cpu().numpy()
                den = w.sum(-1) + np.einsum("hnd,hd->hn", fq[b, :, :n], Z0[b].double().cpu().numpy())
                _close(O[b, :, :n], num / den[..., None], 2e-6, "O")


@pytest.mark.parametrize("pieces", [-1, 2])
@pytest.mark.parametrize("N", [1, 64, 130, 1024])
def test_many_short_bf16_sequences(N, pieces):
    """bf16, D = M = 32, at least 444 sequences of at most 1024 positions, whole and ragged, held to the bf16 gates."""
    B, H, D = 56, 8, 32
    if N == 1024 and pieces > 0:
        pytest.skip("covered by the shorter ones")
    Q, K, V, G = draw_qkvg(B, H, N, D, D, 3 + N, torch.bfloat16, 1.0)
    la.la_plan_override(pieces)
    dev = [t.to(DEV) for t in (Q, K, V, G)]
    lengths = [N - (5 * b) % N for b in range(B)]
    for ln in (None, torch.tensor(lengths, dtype=torch.int32, device=DEV)):
        den = torch.empty(B, H, N, device=DEV)
        O = la.la_causal_forward(*dev[:3], den=den, lengths=ln)
        grads = la.la_causal_backward(*dev, lengths=ln)
        la.la_last_device_status()
        for b in (0, 1, 17, B - 1):
            n = N if ln is None else lengths[b]
            sl = (slice(b, b + 1), slice(0, H, 7), slice(0, n))
            q, k, v, g = (t[sl].double().numpy() for t in (Q, K, V, G))
            Or, denr = oracle.linear_attention(q, k, v, causal=True)[:2]
            assert_close(O[sl], Or, torch.bfloat16, "O")
            assert_close(den[sl], denr, torch.bfloat16, "den")
            for nm, x, ref in zip(("dQ", "dK", "dV"), grads, oracle.linear_attention_backward(q, k, v, g, causal=True)):
                assert_close(x[sl], ref, torch.bfloat16, nm, grad=True)
                assert not x[b, :, n:].any()
            assert not O[b, :, n:].any()


@pytest.mark.parametrize("pieces", [1, 3])
@pytest.mark.parametrize("N", [1, 63, 65, 200])
@pytest.mark.parametrize("B,dtype,phi,D,M", [(28, torch.float32, "elu1", 64, 64), (28, torch.bfloat16, "identity", 128, 64),
                                             (56, torch.bfloat16, "elu1", 32, 32),
                                             (20, torch.float32, "elu1", 64, 64), (20, torch.bfloat16, "identity", 128, 64)])
def test_one_warp_per_strip(B, dtype, phi, D, M, N, pieces):
    """The kernels of full grids (at least 222 CTAs; the third also of many short sequences; the last two, in one piece, the kernels
    with two warps per strip of 149 to 221 CTAs, which neither smaller grids nor full ones take): short last chunks, whole and
    cut into pieces, ragged, from a state and with state gradients, against the oracle on sampled heads.  Tolerances as above,
    8e-6 also for the fp32 state gradients; single planes are held to the bf16 gates."""
    H, eps = 8, 0.5 if N % 2 else 0.0
    Q, K, V, G = draw_qkvg(B, H, N, D, M, 7 + N, dtype, 1.0)
    if phi == "identity":
        Q, K = Q.abs() + 0.1, K.abs() + 0.1
    g = torch.Generator().manual_seed(N)
    S0, Z0 = torch.randn((B, H, D, M), generator=g), torch.rand((B, H, D), generator=g) * 4 + 1
    dS, dZ = torch.randn((B, H, D, M), generator=g) * 0.05, torch.randn((B, H, D), generator=g) * 0.05
    lengths = [N - (7 * b) % (N + 1) for b in range(B)]
    dev = [t.to(DEV) for t in (Q, K, V, G)]
    S0d, Z0d, dSd, dZd = (t.to(DEV) for t in (S0, Z0, dS, dZ))
    la.la_plan_override(pieces)

    def check(x, ref, what, state=False):
        if D == 32:
            assert_close(x, ref, dtype, what, grad=True)
        else:
            tight = dtype == torch.float32 or state
            _close(x, ref, (8e-6 if what[0] == "d" else 2e-6) if tight else 2 ** -8, what)

    for ln in (None, torch.tensor(lengths, dtype=torch.int32, device=DEV)):
        S1, Z1, dS0, dZ0 = (torch.empty_like(t) for t in (S0d, Z0d, S0d, Z0d))
        kw = {"phi": phi, "eps": eps, "lengths": ln, "S_in": S0d, "Z_in": Z0d}
        O = la.la_causal_forward(*dev[:3], S_out=S1, Z_out=Z1, **kw)
        grads = la.la_causal_backward(*dev, dS_out=dSd, dZ_out=dZd, dS_in=dS0, dZ_in=dZ0, **kw)
        la.la_last_device_status()
        for b in (0, 1, 10, B - 1):
            n = N if ln is None else lengths[b]
            assert not O[b, :, n:].any() and not any(x[b, :, n:].any() for x in grads)
            hs = (slice(b, b + 1), slice(0, H, 7))
            sl = (*hs, slice(0, n))
            q, k, v, gg = (t[sl].double().numpy() for t in (Q, K, V, G))
            st = [t[hs].double().numpy() for t in (S0, Z0, dS, dZ)]
            Or, _, Sr, Zr = oracle.causal_from_state(q, k, v, st[0], st[1], phi, eps)
            rq, rk, rv, rS, rZ = oracle.causal_backward_from_state(q, k, v, st[0], st[1], gg, st[2], st[3], phi, eps)
            check(S1[hs], Sr, "S_out", True), check(Z1[hs], Zr, "Z_out", True)
            check(dS0[hs], rS, "dS_in", True), check(dZ0[hs], rZ, "dZ_in", True)
            if n:
                check(O[sl], Or, "O")
                for nm, x, ref in zip(("dQ", "dK", "dV"), grads, (rq, rk, rv)):
                    check(x[sl], ref, nm)


@pytest.mark.parametrize("N", [1, 17, 64, 130])
@pytest.mark.parametrize("B,dtype,phi,D,M", [(56, torch.bfloat16, "elu1", 32, 32), (28, torch.float32, "elu1", 64, 64),
                                             (28, torch.bfloat16, "identity", 128, 64)])
def test_a_zero_state_changes_nothing(B, dtype, phi, D, M, N):
    """A sequence that is trained in pieces may start from a state of zeros: the same results bit for bit as from none
    (the first rows, whose gradients cancel almost entirely, above all).  One warp per strip: at least 222 CTAs."""
    dev = [t.to(DEV) for t in draw_qkvg(B, 8, N, D, M, 3 + N, dtype, 1.0)]
    if phi == "identity":
        dev[0], dev[1] = dev[0].abs() + 0.1, dev[1].abs() + 0.1
    state = {"S_in": torch.zeros(B, 8, D, M, device=DEV), "Z_in": torch.zeros(B, 8, D, device=DEV)}
    plain = (la.la_causal_forward(*dev[:3], phi=phi), *la.la_causal_backward(*dev, phi=phi))
    from_zero = (la.la_causal_forward(*dev[:3], phi=phi, **state), *la.la_causal_backward(*dev, phi=phi, **state))
    la.la_last_device_status()
    assert all(torch.equal(a, b) for a, b in zip(plain, from_zero))


@pytest.mark.parametrize("D,M", [(32, 32), (64, 64), (72, 40)])
def test_the_largest_numbers_keep_their_value(D, M):
    """fp32 numbers above the largest bf16 (3.39e38) are finite and stay what they are; keys of minus infinity have no
    weight, whatever finite values lie beside them."""
    B, H, N = 2, 2, 70
    g = torch.Generator().manual_seed(4)
    top = torch.finfo(torch.float32).max
    K = torch.full((B, H, N, D), -torch.inf)
    K[:, :, ::7] = torch.rand((B, H, 10, D), generator=g) - 8          # ten keys, weights that add up to less than one
    Q = torch.rand((B, H, N, D), generator=g) - 6
    V = top * (1 - torch.rand((B, H, N, M), generator=g) * 2 ** -10) * 2.0 ** -torch.randint(0, 3, (1, H, 1, M), generator=g)
    q, k, v = (t.double().numpy() for t in (Q, K, V))
    dev = [t.to(DEV) for t in (Q, K, V)]
    for causal, call in ((True, la.la_causal_forward), (False, la.la_linear_attention)):
        O = call(*dev)
        la.la_last_device_status()
        assert torch.isfinite(O).all()
        _close(O, oracle.linear_attention(q, k, v, causal=causal)[0], 2e-6, f"O {causal}")


@pytest.mark.parametrize("N", [1, 16, 63, 64, 100])
def test_features_below_the_smallest_normal_number(N):
    """Short bf16 sequences whose keys all lie where exp(x) is below 2^-126: their weights are small numbers like any other.
    The reference takes the features as bf16 holds them (multiples of 2^-133); queries are large enough that scores are normal
    numbers.  2-norms: operands (q, scores, state) and result are each rounded to bf16, 2^-9, so 2^-7 for O and den; the
    gradients are differences of terms of about twice their size, 2^-6."""
    B, H, D = 56, 8, 32
    g = torch.Generator().manual_seed(N)
    Q = (torch.rand((B, H, N, D), generator=g) * 20 + 40).bfloat16()
    K = (torch.randint(0, 4, (B, H, N, D), generator=g) * -0.5 - 87.5).bfloat16()          # -87.5 .. -89
    V, G = (torch.randn((B, H, N, D), generator=g).bfloat16() for _ in range(2))
    dev = [t.to(DEV) for t in (Q, K, V, G)]
    den = torch.empty(B, H, N, device=DEV)
    O = la.la_causal_forward(*dev[:3], den=den)
    grads = la.la_causal_backward(*dev)
    la.la_last_device_status()
    sl = (slice(0, B, 55), slice(0, H, 7))
    q, k, v, gg = (t[sl].double().numpy() for t in (Q, K, V, G))
    fq, fk = q + 1, np.round(np.exp(k) * 2.0 ** 133) * 2.0 ** -133
    fq = torch.from_numpy(fq).bfloat16().double().numpy()
    Or, denr = oracle.linear_attention(fq, fk, v, causal=True, phi="identity")[:2]
    _close(O[sl], Or, 2 ** -7, "O")
    _close(den[sl].double() * 2.0 ** 120, denr * 2.0 ** 120, 2 ** -7, "den")
    rq, rk, rv = oracle.linear_attention_backward(fq, fk, v, gg, causal=True, phi="identity")
    for nm, x, ref in zip(("dQ", "dK", "dV"), grads, (rq, rk * fk, rv)):           # slopes: 1 and the feature itself
        if N > 1 or nm == "dV":                                                     # (one key: the others are analytically zero)
            _close(x[sl], ref, 2 ** -6, nm)


def test_every_launch_can_be_profiled():
    """la_profile_enable() brackets every main kernel, these ones included."""
    dev = [t.to(DEV) for t in draw_qkvg(56, 8, 96, 32, 32, 1, torch.bfloat16, 1.0)]
    f32 = [t[:2].float().contiguous() for t in dev]
    la.la_plan_override(2, -1, -1)
    want = {"causal_mma_forward_kernel": 2, "causal_mma_dq_kernel": 1, "causal_mma_dkv_kernel": 1, "causal_mma_sum_kernel": 6,
            "linear_mma_apply_kernel": 3}
    la.la_profile_enable(True)
    try:
        la.la_causal_forward(*dev[:3])          # two pieces: sums, forward
        la.la_causal_backward(*dev)             # sums, dQ, reverse sums, dK and dV
        la.la_causal_forward(*f32[:3], ws=torch.empty(0, dtype=torch.uint8, device=DEV))        # no room for pieces: one kernel
        la.la_linear_attention(*f32[:3])
        la.la_linear_attention_backward(*f32, saved=None)
        got = {k: n for k, (_, n) in la.la_profile_read().items()}
    finally:
        la.la_profile_enable(False)
    assert got == want


@pytest.mark.parametrize("splits", [-1, 1, 3])
@pytest.mark.parametrize("N", [1, 16, 63, 64, 65, 400])
@pytest.mark.parametrize("dims", [(8, 8), (32, 32), (40, 24), (64, 64), (72, 64), (128, 64)], ids=str)
def test_noncausal_tiles(dims, N, splits):
    """The non-causal form on the same products: strips, splits, a ragged batch with an empty sequence, kept sums."""
    D, M = dims
    for dtype, phi in ((torch.float32, "elu1"), (torch.float32, "identity"), (torch.bfloat16, "identity"), (torch.bfloat16, "elu1")):
        if dtype == torch.bfloat16 and D == M and D in (32, 64):
            continue                                    # another kernel's problem
        Q, K, V, G = draw_qkvg(3, 2, N, D, M, 3 + N, dtype, 1.0)
        if phi == "identity":
            Q, K = Q.abs() + 0.1, K.abs() + 0.1
        la.la_plan_override(-1, -1, splits)
        dev = [t.to(DEV) for t in (Q, K, V, G)]
        eps = 0.5 if N % 2 else 0.0
        lengths = [N, 0, (N + 1) // 2]
        for ln in (None, torch.tensor(lengths, dtype=torch.int32, device=DEV)):
            saved = la.linear_saved_buffer(dev[0], dev[2], phi=phi)
            den = torch.empty(3, 2, N, device=DEV)
            O = la.la_linear_attention(*dev[:3], phi=phi, eps=eps, lengths=ln, saved=saved, den=den)
            grads = la.la_linear_attention_backward(*dev, phi=phi, eps=eps, lengths=ln, saved=saved)
            plain = la.la_linear_attention_backward(*dev, phi=phi, eps=eps, lengths=ln)
            la.la_last_device_status()
            assert all(torch.equal(a, b) for a, b in zip(grads, plain))
            f32 = dtype == torch.float32
            for b in range(3):
                n = N if ln is None else lengths[b]
                assert not O[b, :, n:].any() and not den[b, :, n:].any() and not any(x[b, :, n:].any() for x in grads)
                if n == 0:
                    continue
                sl = (slice(b, b + 1), slice(None), slice(0, n))
                q, k, v, g = (t[sl].double().numpy() for t in (Q, K, V, G))
                Or, denr = oracle.linear_attention(q, k, v, causal=False, phi=phi, eps=eps)[:2]
                _close(O[sl], Or, 2e-6 if f32 else 2 ** -8, "O")
                _close(den[sl], denr, 2e-6, "den")
                if n == 1 and not eps:
                    continue                            # dQ and dK are analytically zero
                # (one key: O = V dn' / (dn' + eps), so that of dQ's and dK's terms only their eps / dn is left)
                left = eps / (np.abs(denr).max() + eps) if n == 1 else 1.0
                for nm, x, ref in zip(("dQ", "dK", "dV"), grads,
                                      oracle.linear_attention_backward(q, k, v, g, causal=False, phi=phi, eps=eps)):
                    _close(x[sl], ref, (8e-6 if f32 else 2 ** -8) / (left if f32 else 1.0), nm)
