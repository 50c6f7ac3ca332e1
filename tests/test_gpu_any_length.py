"""Sequence lengths that are not a multiple of the 128-position chunk on the tensor-core kernels.

The last chunk of such a sequence is partly beyond its end, where memory holds the NEXT sequence
(or nothing): tile loads must read zeros there and nothing may be stored there.  Every tensor of
these tests sits at the front of a larger buffer filled with a marker, so that a store past a
tensor's end would be seen (and would be harmless); stores into the next sequence show up in the
comparison with the oracle.
"""
import os

import numpy as np
import pytest
import torch

import oracle
import paper_2006_16236_b200 as la
from paper_2006_16236_b200.inputs import draw_qkvg
from parity import assert_close

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda")
SLACK = 32768           # elements behind every tensor
MARK = 1234.0


def _front(shape, dtype):
    n = int(np.prod(shape))
    flat = torch.full((n + SLACK,), MARK, dtype=dtype, device=DEV)
    return flat[:n].view(shape), flat[n:]


def _place(t):
    v, tail = _front(tuple(t.shape), t.dtype)
    v.copy_(t)
    return v, tail


def _untouched(tails):
    for nm, tail in tails.items():
        assert bool((tail == MARK).all()), f"{nm}: something was stored behind the tensor's end"


@pytest.fixture
def tcgen05(request):
    """Whether the calls are kept to the tcgen05 kernels (non-causal: to those with a warp per sixteen positions): plans that are forced, to
    pieces and splits as the automatic ones choose about, leave out the kernels with a cluster per sequence that would take short problems."""
    yield request.param
    la.la_plan_override()


ROUTES = pytest.mark.parametrize("tcgen05", [False, True], ids=["automatic", "tcgen05"], indirect=True)
CLUSTER, TC = {"causal_cluster_forward_kernel", "causal_cluster_backward_kernel"}, {"causal_fwd_kernel", "causal_bwd_dq_kernel", "causal_bwd_dkv_kernel"}

SHAPES = [(2, 3, 100, 64), (2, 3, 129, 64), (1, 5, 200, 32), (2, 8, 784, 32), (3, 2, 1000, 64), (1, 70, 700, 64),
          (2, 2, 1, 64), (1, 3, 127, 32), (1, 2, 2, 32)]


@pytest.mark.parametrize("keep", [False, True], ids=["recompute", "saved"])
@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "B%d_H%d_N%d_D%d" % s)
@ROUTES
def test_causal_any_length(tcgen05, shape, keep):
    B, H, N, D = shape
    p = la.make_problem(B, H, N, D, D, la.LA_BF16)
    assert la.la_causal_plan(p) is not None, "this shape is meant to run the tensor-core kernels"
    if tcgen05:
        la.la_plan_override(causal_pieces=min(3, (N + 127) // 128))
    Q, K, V, G = draw_qkvg(B, H, N, D, D, 7 + N, torch.bfloat16, 1.0)
    tails = {}
    dev = {}
    for nm, t in zip("QKVG", (Q, K, V, G)):
        dev[nm], tails[nm] = _place(t.to(DEV))
    outs = {}
    for nm, like in (("O", V), ("dQ", Q), ("dK", K), ("dV", V)):
        outs[nm], tails[nm] = _front(tuple(like.shape), torch.bfloat16)
    den, tails["den"] = _front((B, H, N), torch.float32)
    S, tails["S"] = _front((B, H, D, D), torch.float32)
    Z, tails["Z"] = _front((B, H, D), torch.float32)
    saved = la.saved_buffer(dev["Q"], dev["V"]) if keep else None
    kw = {"saved": saved} if keep else {}
    la.la_profile_enable(True)
    la.la_causal_forward(dev["Q"], dev["K"], dev["V"], O=outs["O"], den=den, S_out=S, Z_out=Z, **kw)
    la.la_causal_backward(dev["Q"], dev["K"], dev["V"], dev["G"], dQ=outs["dQ"], dK=outs["dK"], dV=outs["dV"], **kw)
    la.la_last_device_status()
    names = set(la.la_profile_read()) - {"segment_sum_kernel"}
    la.la_profile_enable(False)
    assert names == TC if tcgen05 else names <= TC | CLUSTER
    _untouched(tails)
    q, k, v, g = (t.double().numpy() for t in (Q, K, V, G))
    O_ref, den_ref = oracle.linear_attention(q, k, v, causal=True)[:2]
    assert_close(outs["O"], O_ref, torch.bfloat16, "O")
    assert_close(den, den_ref, torch.bfloat16, "den")
    for nm, ref in zip(("dQ", "dK", "dV"), oracle.linear_attention_backward(q, k, v, g, causal=True)):
        assert_close(outs[nm], ref, torch.bfloat16, nm, grad=True)
    # the state at the sequence's end: what the unrolled recurrence holds after N steps
    fk = oracle.feature_map(k)
    assert_close(S, np.einsum("bhnd,bhnm->bhdm", fk, v), torch.bfloat16, "S_out")
    assert_close(Z, fk.sum(2), torch.bfloat16, "Z_out")


@pytest.mark.parametrize("shape", SHAPES[:5] + SHAPES[6:], ids=lambda s: "B%d_H%d_N%d_D%d" % s)
@ROUTES
def test_noncausal_any_length(tcgen05, shape):
    B, H, N, D = shape
    if tcgen05:
        la.la_plan_override(linear_splits=min(3, (N + 127) // 128))
    Q, K, V, G = draw_qkvg(B, H, N, D, D, 11 + N, torch.bfloat16, 0.5)
    tails, dev, outs = {}, {}, {}
    for nm, t in zip("QKVG", (Q, K, V, G)):
        dev[nm], tails[nm] = _place(t.to(DEV))
    for nm, like in (("O", V), ("dQ", Q), ("dK", K), ("dV", V)):
        outs[nm], tails[nm] = _front(tuple(like.shape), torch.bfloat16)
    den, tails["den"] = _front((B, H, N), torch.float32)
    la.la_profile_enable(True)
    la.la_linear_attention(dev["Q"], dev["K"], dev["V"], O=outs["O"], den=den)
    la.la_linear_attention_backward(dev["Q"], dev["K"], dev["V"], dev["G"], dQ=outs["dQ"], dK=outs["dK"], dV=outs["dV"])
    la.la_last_device_status()
    names = set(la.la_profile_read())
    la.la_profile_enable(False)
    assert names == {"linear_warp_sum_kernel", "linear_warp_apply_kernel", "linear_warp_dq_kernel"} | (set() if tcgen05 else {"linear_cluster_forward_kernel"}), names
    _untouched(tails)
    q, k, v, g = (t.double().numpy() for t in (Q, K, V, G))
    O_ref, den_ref = oracle.linear_attention(q, k, v, causal=False)[:2]
    assert_close(outs["O"], O_ref, torch.bfloat16, "O")
    assert_close(den, den_ref, torch.bfloat16, "den")
    for nm, ref in zip(("dQ", "dK", "dV"), oracle.linear_attention_backward(q, k, v, g, causal=False)):
        assert_close(outs[nm], ref, torch.bfloat16, nm, grad=True)


SUMS_AND_DQ = {"linear_sum_kernel", "linear_apply_kernel"}         # the non-causal kernels on tcgen05: D = 64, more than 512 and 65536 positions


@pytest.mark.parametrize("ragged", [False, True])
@pytest.mark.parametrize("phi", ["elu1", "identity"])
@pytest.mark.parametrize("N", [1000, 1001, 1024])
def test_noncausal_of_many_positions(N, phi, ragged):
    B, H, D = 9, 8, 64
    lengths = [N, 0, N - 1, 513, 128, 1, 640, N // 2, 999] if ragged else [N] * B
    Q, K, V, G = draw_qkvg(B, H, N, D, D, 13 + N, torch.bfloat16, 0.5)
    if phi == "identity":                               # features: positive, as the weights of a kernel are
        Q, K = ((t.float().abs() + 0.1).to(torch.bfloat16) for t in (Q, K))
    tails, dev, outs = {}, {}, {}
    for nm, t in zip("QKVG", (Q, K, V, G)):
        dev[nm], tails[nm] = _place(t.to(DEV))
    for nm, like in (("O", V), ("dQ", Q), ("dK", K), ("dV", V)):
        outs[nm], tails[nm] = _front(tuple(like.shape), torch.bfloat16)
    den, tails["den"] = _front((B, H, N), torch.float32)
    KV, tails["KV"] = _front((B, H, D, D), torch.float32)
    Zs, tails["Zs"] = _front((B, H, D), torch.float32)
    saved = la.linear_saved_buffer(dev["Q"], dev["V"], phi=phi)
    kw = {"phi": phi, "lengths": torch.tensor(lengths, dtype=torch.int32, device=DEV) if ragged else None}
    la.la_profile_enable(True)
    la.la_linear_attention(dev["Q"], dev["K"], dev["V"], O=outs["O"], den=den, KV=KV, Zs=Zs, saved=saved, **kw)
    la.la_linear_attention_backward(dev["Q"], dev["K"], dev["V"], dev["G"], saved=saved, dQ=outs["dQ"], dK=outs["dK"], dV=outs["dV"], **kw)
    la.la_last_device_status()
    names = set(la.la_profile_read())
    la.la_profile_enable(False)
    assert names == SUMS_AND_DQ | {"linear_warp_apply_kernel"}, names
    _untouched(tails)
    again = la.la_linear_attention_backward(dev["Q"], dev["K"], dev["V"], dev["G"], **kw)      # the sums that it would make itself
    assert all(torch.equal(outs[nm], x) for nm, x in zip(("dQ", "dK", "dV"), again))
    for b, n in enumerate(lengths):
        for nm in ("O", "dQ", "dK", "dV"):
            assert not outs[nm][b, :, n:].any(), f"{nm}: padding of sequence {b} is not zero"
        h = b % H
        sl = (slice(b, b + 1), slice(h, h + 1), slice(0, n))
        if n == 0:
            assert not KV[b].any() and not Zs[b].any()
            continue
        q, k, v, g = (t[sl].double().numpy() for t in (Q, K, V, G))
        O_ref, den_ref = oracle.linear_attention(q, k, v, causal=False, phi=phi)[:2]
        assert_close(outs["O"][sl], O_ref, torch.bfloat16, f"O of sequence {b}")
        assert_close(den[sl], den_ref, torch.bfloat16, f"den of sequence {b}")
        fk = oracle.feature_map(k) if phi == "elu1" else k
        assert_close(KV[b:b + 1, h:h + 1], np.einsum("bhnd,bhnm->bhdm", fk, v), torch.bfloat16, f"KV of sequence {b}")
        assert_close(Zs[b:b + 1, h:h + 1], fk.sum(2), torch.bfloat16, f"Zs of sequence {b}")
        if n > 1:                                       # (of one position dQ and dK are analytically zero)
            for nm, ref in zip(("dQ", "dK", "dV"), oracle.linear_attention_backward(q, k, v, g, causal=False, phi=phi)):
                assert_close(outs[nm][sl], ref, torch.bfloat16, f"{nm} of sequence {b}", grad=True)


def test_noncausal_of_many_positions_refuses_sums_of_another_plan():
    if os.environ.get("LA_DEBUG"):
        pytest.skip("in checked mode the call itself reads the status and raises; this test reads it afterwards")
    dev = [t.to(DEV) for t in draw_qkvg(9, 8, 1000, 64, 64, 5, torch.bfloat16, 0.5)]
    try:
        la.la_plan_override(linear_splits=4)
        saved = la.linear_saved_buffer(dev[0], dev[2])
        la.la_linear_attention(*dev[:3], saved=saved)
        for splits in (2, 3, -1):
            la.la_plan_override(linear_splits=splits)
            outs = [torch.full_like(dev[0], 7.0) for _ in range(3)]
            la.la_profile_enable(True)
            la.la_linear_attention_backward(*dev, saved=saved, dQ=outs[0], dK=outs[1], dV=outs[2])
            with pytest.raises(la.LaError) as e:
                la.la_last_device_status()
            names = set(la.la_profile_read())
            la.la_profile_enable(False)
            assert e.value.status == -1 and "plan" in str(e.value) and names == {"linear_apply_kernel", "linear_warp_apply_kernel"}
            assert all(torch.all(t == 7.0) for t in outs)           # nothing was written
            la.la_last_device_status()
    finally:
        la.la_plan_override()


@pytest.mark.parametrize("causal", [False, True])
@ROUTES
def test_lengths_inside_a_batch_whose_own_length_is_odd(tcgen05, causal):
    """Both kinds of raggedness at once: N = 700 and per-sequence lengths below it (one of them 0, one of them N)."""
    if tcgen05:
        la.la_plan_override(causal_pieces=3, linear_splits=3)
    B, H, N, D = 4, 2, 700, 64
    lengths = [700, 0, 333, 129]
    Q, K, V, G = draw_qkvg(B, H, N, D, D, 5, torch.bfloat16, 1.0)
    tails, dev, outs = {}, {}, {}
    for nm, t in zip("QKVG", (Q, K, V, G)):
        dev[nm], tails[nm] = _place(t.to(DEV))
    for nm, like in (("O", V), ("dQ", Q), ("dK", K), ("dV", V)):
        outs[nm], tails[nm] = _front(tuple(like.shape), torch.bfloat16)
    ln = torch.tensor(lengths, dtype=torch.int32, device=DEV)
    if causal:
        la.la_causal_forward(dev["Q"], dev["K"], dev["V"], lengths=ln, O=outs["O"])
        la.la_causal_backward(dev["Q"], dev["K"], dev["V"], dev["G"], lengths=ln, dQ=outs["dQ"], dK=outs["dK"], dV=outs["dV"])
    else:
        la.la_linear_attention_varlen(dev["Q"], dev["K"], dev["V"], ln, O=outs["O"])
        la.la_linear_attention_varlen_backward(dev["Q"], dev["K"], dev["V"], dev["G"], ln, dQ=outs["dQ"], dK=outs["dK"], dV=outs["dV"])
    la.la_last_device_status()
    _untouched(tails)
    for b, n in enumerate(lengths):
        for nm in ("O", "dQ", "dK", "dV"):
            assert not bool(outs[nm][b, :, n:].float().abs().max() > 0) if n < N else True, f"{nm}: padding of sequence {b} is not zero"
        if n == 0:
            continue
        q, k, v, g = (t[b:b + 1, :, :n].double().numpy() for t in (Q, K, V, G))
        O_ref = oracle.linear_attention(q, k, v, causal=causal)[0]
        assert_close(outs["O"][b:b + 1, :, :n], O_ref, torch.bfloat16, f"O of sequence {b}")
        for nm, ref in zip(("dQ", "dK", "dV"), oracle.linear_attention_backward(q, k, v, g, causal=causal)):
            assert_close(outs[nm][b:b + 1, :, :n], ref, torch.bfloat16, f"{nm} of sequence {b}", grad=True)


def test_prefill_in_odd_pieces_then_decode():
    """A prompt of 300 positions fed in calls of 77, 200 and 23 positions (none a multiple of the chunk), each
    continuing from the state the call before left, then two decode steps: the same outputs as the whole sequence."""
    B, H, D = 2, 3, 64
    cuts = [77, 200, 23]
    N = sum(cuts) + 2
    Q, K, V, _ = draw_qkvg(B, H, N, D, D, 3, torch.bfloat16, 1.0, with_grad=False)
    O_ref = oracle.linear_attention(*(t.double().numpy() for t in (Q, K, V)), causal=True)[0]
    S = torch.zeros((B, H, D, D), device=DEV)
    Z = torch.zeros((B, H, D), device=DEV)
    lo = 0
    for n in cuts:
        q, k, v = (t[:, :, lo:lo + n].contiguous().to(DEV) for t in (Q, K, V))
        S2, Z2 = torch.empty_like(S), torch.empty_like(Z)
        O = la.la_causal_forward(q, k, v, S_in=S, Z_in=Z, S_out=S2, Z_out=Z2)
        assert_close(O, O_ref[:, :, lo:lo + n], torch.bfloat16, f"positions {lo}..{lo + n}")
        S, Z, lo = S2, Z2, lo + n
    for i in range(lo, N):
        out = la.la_recurrent_step(Q[:, :, i].contiguous().to(DEV), K[:, :, i].contiguous().to(DEV), V[:, :, i].contiguous().to(DEV), S, Z)
        assert_close(out, O_ref[:, :, i], torch.bfloat16, f"decode step {i}")
    la.la_last_device_status()
