"""Stream order around the calls: what a kernel enqueued just before a call wrote is what the call reads.

The kernels of one call follow each other as programmatic dependents, and several of them request
their first tiles (or read the decode state) before they wait for the kernel in front of them.
That is only right if everything enqueued BEFORE the call is complete by then.  Here the inputs
of every call are rewritten in the stream immediately before it (long copies, no host
synchronisation anywhere, two alternating sets of values, so that stale data would be the other
set's), and every result has to be bit-identical to the one of a fully synchronised run.
"""
import os

import pytest
import torch

import paper_2006_16236_b200 as la
from paper_2006_16236_b200.inputs import WORKLOADS, draw_workload

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda")


def _calls(kind):
    if kind == "causal":
        return la.la_causal_forward, la.la_causal_backward, la.saved_buffer
    return la.la_linear_attention, la.la_linear_attention_backward, la.linear_saved_buffer


@pytest.mark.parametrize("keep", [False, True], ids=["recompute", "saved"])
@pytest.mark.parametrize("name", ["causal_sweep_bf16_N16384", "causal_sweep_bf16_N65536", "noncausal_bf16_speech"])
def test_inputs_written_in_stream_just_before_a_call_are_seen(name, keep):
    w = WORKLOADS[name]
    fwd, bwd, make_saved = _calls(w.kind)
    set_a = [t.to(DEV) for t in draw_workload(w)]
    set_b = [(t.flip(2) * 0.75).contiguous() for t in set_a]            # other values at every position
    Q, K, V, G = (torch.empty_like(t) for t in set_a)
    O, dQ, dK, dV = torch.empty_like(V), torch.empty_like(Q), torch.empty_like(K), torch.empty_like(V)
    saved = make_saved(Q, V) if keep else None
    kw = {"saved": saved} if keep else {}

    def run(src, synced):
        def gap():
            if synced:
                torch.cuda.synchronize()
        Q.copy_(src[0]); K.copy_(src[1]); V.copy_(src[2]); gap()
        fwd(Q, K, V, O=O, **kw); gap()
        G.copy_(src[3]); gap()
        bwd(Q, K, V, G, dQ=dQ, dK=dK, dV=dV, **kw); gap()
        return [t.clone() for t in (O, dQ, dK, dV)]

    want = {0: run(set_a, True), 1: run(set_b, True)}
    assert not torch.equal(want[0][0], want[1][0])
    torch.cuda.synchronize()
    got = [(i & 1, run(set_b if i & 1 else set_a, False)) for i in range(6)]
    torch.cuda.synchronize()
    la.la_last_device_status()
    for i, (which, res) in enumerate(got):
        for a, b, nm in zip(want[which], res, ("O", "dQ", "dK", "dV")):
            assert torch.equal(a, b), f"{name}: {nm} of unsynchronised repeat {i} differs from the synchronised run"


def test_decode_layer_fed_back_on_the_device_without_synchronisation():
    """Generation loop on the device: the next input is made from the previous output by ordinary stream-ordered
    kernels; the step kernel reads the state, and the output projection its weights, before waiting for the
    kernel in front of them.  Same bits as with a host synchronisation after every operation."""
    B, H, D, T = 256, 8, 64, 24
    F = H * D
    g = torch.Generator().manual_seed(5)
    s = 1.0 / F ** 0.5
    Wqkv = (torch.randn((3 * F, F), generator=g) * s).to(torch.bfloat16).to(DEV)
    Wo = (torch.randn((F, F), generator=g) * s).to(torch.bfloat16).to(DEV)
    x0 = torch.randn((B, F), generator=g).to(torch.bfloat16).to(DEV)

    def run(synced):
        S = torch.zeros((B, H, D, D), device=DEV)
        Z = torch.zeros((B, H, D), device=DEV)
        x, ys = x0.clone(), []
        for t in range(T):
            y = la.la_decode_layer_step(x, Wqkv, Wo, S, Z)
            if synced:
                torch.cuda.synchronize()
            ys.append(y)
            x = torch.tanh(y.float()).to(torch.bfloat16)
            if t == T // 2:
                S.mul_(0.5)         # the state rewritten in the stream between two calls
                Z.mul_(0.5)
            if synced:
                torch.cuda.synchronize()
        torch.cuda.synchronize()
        return ys, S, Z

    ys1, S1, Z1 = run(True)
    ys2, S2, Z2 = run(False)
    la.la_last_device_status()
    for t, (a, b) in enumerate(zip(ys1, ys2)):
        assert torch.equal(a, b), f"token {t}"
    assert torch.equal(S1, S2) and torch.equal(Z1, Z2)


@pytest.mark.parametrize("name", ["causal_sweep_bf16_N16384", "noncausal_bf16_speech"])
def test_training_step_replayed_from_a_cuda_graph(name):
    """Forward + backward captured into a CUDA graph after one eager call (the first call of a kernel opts in to
    its shared memory, which is not a stream operation) and replayed: the chained launches keep their order
    inside the graph, and the replays give the eager call's bits."""
    if os.environ.get("LA_DEBUG"):
        pytest.skip("checked mode synchronises after every call, which a stream capture does not allow")
    w = WORKLOADS[name]
    fwd, bwd, make_saved = _calls(w.kind)
    Q, K, V, G = (t.to(DEV) for t in draw_workload(w))
    O, dQ, dK, dV = torch.empty_like(V), torch.empty_like(Q), torch.empty_like(K), torch.empty_like(V)
    saved = make_saved(Q, V)
    ws_f = la.workspace(la.make_problem(w.B, w.H, w.N, w.D, w.M, la.LA_BF16),
                        la.LA_OP_CAUSAL_FORWARD if w.kind == "causal" else la.LA_OP_LINEAR_FORWARD, DEV)
    ws_b = la.workspace(la.make_problem(w.B, w.H, w.N, w.D, w.M, la.LA_BF16),
                        la.LA_OP_CAUSAL_BACKWARD if w.kind == "causal" else la.LA_OP_LINEAR_BACKWARD, DEV)

    def step():
        fwd(Q, K, V, O=O, saved=saved, ws=ws_f)
        bwd(Q, K, V, G, dQ=dQ, dK=dK, dV=dV, saved=saved, ws=ws_b)

    step()
    torch.cuda.synchronize()
    want = [t.clone() for t in (O, dQ, dK, dV)]
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.stream(side):
        with torch.cuda.graph(graph, stream=side):
            step()
    torch.cuda.current_stream().wait_stream(side)
    for _ in range(3):
        for t in (O, dQ, dK, dV):
            t.fill_(7.0)
        graph.replay()
        torch.cuda.synchronize()
        for a, b, nm in zip(want, (O, dQ, dK, dV), ("O", "dQ", "dK", "dV")):
            assert torch.equal(a, b), f"{name}: {nm} of a graph replay differs from the eager call"
    la.la_last_device_status()


@pytest.mark.parametrize("kind,H,N,D", [("causal", 8, 1100, 64), ("causal", 4, 500, 64), ("causal", 8, 1100, 32), ("linear", 8, 1000, 64),
                                        ("linear", 3, 300, 32)])
def test_short_training_step_replayed_from_a_cuda_graph(kind, H, N, D):
    """Steps of a cluster per sequence, captured with the copies that write their inputs just before them: with a saved buffer the
    cluster kernel starts beside the pre-pass in front of it and waits for it at its own end, and what follows needs both.  Two
    sets of values in turn, so that stale data would be the other set's; the replays give the bits of a synchronised run."""
    if os.environ.get("LA_DEBUG"):
        pytest.skip("checked mode synchronises after every call, which a stream capture does not allow")
    fwd, bwd, make_saved = _calls(kind)
    g = torch.Generator().manual_seed(3)
    set_a = [torch.randn((1, H, N, D), generator=g).bfloat16().to(DEV) for _ in range(4)]
    sets = [set_a, [(t.flip(2) * 0.75).contiguous() for t in set_a]]
    src = [torch.empty_like(t) for t in set_a]
    Q, K, V, G = (torch.empty_like(t) for t in set_a)
    O, dQ, dK, dV = torch.empty_like(V), torch.empty_like(Q), torch.empty_like(K), torch.empty_like(V)
    saved = make_saved(Q, V)

    def step(gap=lambda: None):
        Q.copy_(src[0]); K.copy_(src[1]); V.copy_(src[2]); G.copy_(src[3]); gap()
        fwd(Q, K, V, O=O, saved=saved); gap()
        bwd(Q, K, V, G, dQ=dQ, dK=dK, dV=dV, saved=saved); gap()

    want = []
    for values in sets:
        for a, b in zip(src, values):
            a.copy_(b)
        step(torch.cuda.synchronize)
        want.append([t.clone() for t in (O, dQ, dK, dV)])
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.stream(side):
        with torch.cuda.graph(graph, stream=side):
            for _ in range(3):
                step()
    torch.cuda.current_stream().wait_stream(side)
    for i in range(6):
        for a, b in zip(src, sets[i % 2]):
            a.copy_(b)
        for t in (O, dQ, dK, dV):
            t.fill_(7.0)
        graph.replay()
        for a, b, nm in zip(want[i % 2], (O, dQ, dK, dV), ("O", "dQ", "dK", "dV")):
            assert torch.equal(a, b), f"replay {i}: {nm} differs from the synchronised run"
    la.la_last_device_status()


@pytest.mark.parametrize("D,H", [(32, 2), (64, 4)])
def test_small_fp32_calls_that_feed_each_other(D, H):
    """The kernels of small fp32 problems start as programmatic dependents of whatever is in front of them, another call's
    included: the state goes from piece to piece of a prompt between two pairs of buffers, outputs and gradients go
    straight into the next call as its inputs, and nothing is synchronised.  Same bits as with a wait after every call."""
    B, N, T = 1, 200, 12
    g = torch.Generator().manual_seed(11)
    Q, K, V, G = (torch.randn((B, H, T * N, D), generator=g).to(DEV) for _ in range(4))
    pieces = [[t[:, :, i * N:(i + 1) * N].contiguous() for t in (Q, K, V, G)] for i in range(T)]

    def run(synced):
        def gap():
            if synced:
                torch.cuda.synchronize()
        S = [torch.zeros((B, H, D, D), device=DEV) for _ in range(2)]
        Z = [torch.zeros((B, H, D), device=DEV) for _ in range(2)]
        q, k, v, o = (torch.empty_like(pieces[0][0]) for _ in range(4))
        out = []
        for i, (a, b, c, d) in enumerate(pieces):
            q.copy_(a); k.copy_(b); v.copy_(c); gap()
            la.la_causal_forward(q, k, v, O=o, S_in=S[i & 1], Z_in=Z[i & 1], S_out=S[~i & 1], Z_out=Z[~i & 1]); gap()
            dq, dk, dv = la.la_causal_backward(q, k, o, d, S_in=S[i & 1], Z_in=Z[i & 1]); gap()
            e = la.la_linear_attention(dq, dk, dv); gap()
            out += [o.clone(), dq, dk, dv, e, *la.la_linear_attention_backward(q, k, e, dv)]; gap()
        torch.cuda.synchronize()
        return out + S + Z

    want = run(True)
    for _ in range(4):
        for i, (a, b) in enumerate(zip(want, run(False), strict=True)):
            assert torch.equal(a, b), i
    la.la_last_device_status()
