"""Short sequences in one launch (a thread-block cluster per sequence): lengths at the edges of a CTA's rows and of the cluster,
ragged, from a state and with state gradients, and the bidirectional forward pass, against the fp64 oracle.

Tolerances (2-norm of the difference over the 2-norm of the result) as for the other kernels on these instructions: fp32 2e-6
where terms do not cancel (16 * 2^-23), 8e-6 for gradients; bf16 D = M calls are held to the gates of tests/parity.py, bf16
features of 128 columns to one rounding of the output, 2^-8 (their states stay in fp32)."""
import numpy as np
import pytest
import torch

import oracle
import paper_2006_16236_b200 as la
from paper_2006_16236_b200.inputs import draw_qkvg
from parity import assert_close

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
SIZES = {torch.float32: [1, 16, 63, 64, 65, 130, 1000, 1024], torch.bfloat16: [1, 63, 64, 128, 129, 300, 1024, 1025, 2048]}
CAUSAL = [(torch.float32, "elu1", 32, 32), (torch.float32, "identity", 64, 64), (torch.bfloat16, "elu1", 64, 64),
          (torch.bfloat16, "elu1", 32, 32), (torch.bfloat16, "identity", 128, 64)]


def _close(x, ref, tol, what):
    x, ref = x.double().cpu().numpy(), np.asarray(ref)
    assert np.linalg.norm(x - ref) <= tol * np.linalg.norm(ref) + 1e-30, (what, np.linalg.norm(x - ref) / np.linalg.norm(ref))


@pytest.mark.parametrize("dtype,phi,D,M,N", [(*c, n) for c in CAUSAL for n in SIZES[c[0]] if c[2] != 128 or n <= 1024])
def test_causal(dtype, phi, D, M, N):
    causal_against_the_oracle(dtype, phi, D, M, N, 3, 1)


@pytest.mark.parametrize("dtype,phi,D,M", CAUSAL + [(torch.float32, "elu1", 64, 64), (torch.float32, "identity", 32, 32),
                                                    (torch.bfloat16, "identity", 64, 64), (torch.bfloat16, "identity", 32, 32)])
def test_causal_with_several_heads(dtype, phi, D, M):
    """The lengths of a ragged batch belong to its sequences, each of several heads; both feature maps of every kernel."""
    causal_against_the_oracle(dtype, phi, D, M, 500, 3, 2)
    Q, K, V = (torch.zeros(3, 2, 500, c, dtype=dtype, device=DEV) + 1 for c in (D, D, M))
    assert set(kernels_of(lambda: la.la_causal_forward(Q, K, V, phi=phi))) == {"causal_cluster_forward_kernel"}
    assert set(kernels_of(lambda: la.la_causal_backward(Q, K, V, V, phi=phi))) == {"causal_cluster_backward_kernel"}


def causal_against_the_oracle(dtype, phi, D, M, N, B, H):
    eps = 0.5 if N % 2 else 0.0
    Q, K, V, G = draw_qkvg(B, H, N, D, M, 11 + N, dtype, 1.0)
    if phi == "identity":                               # features: positive, as the weights of a kernel are
        Q, K = Q.abs() + 0.1, K.abs() + 0.1
    g = torch.Generator().manual_seed(N)
    S0, Z0 = torch.randn((B, H, D, M), generator=g), torch.rand((B, H, D), generator=g) * 4 + 1
    dS, dZ = torch.randn((B, H, D, M), generator=g) * 0.05, torch.randn((B, H, D), generator=g) * 0.05
    dev = [t.to(DEV) for t in (Q, K, V, G)]
    S0d, Z0d, dSd, dZd = (t.to(DEV) for t in (S0, Z0, dS, dZ))

    def check(x, ref, what, state=False):
        if dtype == torch.bfloat16 and D == M:
            assert_close(x, ref, dtype, what, grad=what[0] == "d")
        else:
            _close(x, ref, (8e-6 if what[0] == "d" else 2e-6) if dtype == torch.float32 or state else 2 ** -8, what)

    for lengths in (None, [N, N // 2, 0]):
        ln = None if lengths is None else torch.tensor(lengths, dtype=torch.int32, device=DEV)
        for state in (False, True):
            S1, Z1, dS0, dZ0 = (torch.full_like(t, 7.0) for t in (S0d, Z0d, S0d, Z0d))
            den = torch.empty(B, H, N, device=DEV)
            kw = {"phi": phi, "eps": eps, "lengths": ln, **({"S_in": S0d, "Z_in": Z0d} if state else {})}
            O = la.la_causal_forward(*dev[:3], den=den, S_out=S1, Z_out=Z1, **kw)
            grads = la.la_causal_backward(*dev, **kw, **({"dS_out": dSd, "dZ_out": dZd, "dS_in": dS0, "dZ_in": dZ0} if state else {}))
            la.la_last_device_status()
            for b in range(B):
                n = N if lengths is None else lengths[b]
                assert not O[b, :, n:].any() and not den[b, :, n:].any() and not any(x[b, :, n:].any() for x in grads)
                sl = (slice(b, b + 1), slice(None), slice(0, n))
                q, k, v, gg = (t[sl].double().numpy() for t in (Q, K, V, G))
                st = [(t[b:b + 1] if state else torch.zeros_like(t[b:b + 1])).double().numpy() for t in (S0, Z0, dS, dZ)]
                Or, denr, Sr, Zr = oracle.causal_from_state(q, k, v, st[0], st[1], phi, eps)
                rq, rk, rv, rS, rZ = oracle.causal_backward_from_state(q, k, v, st[0], st[1], gg, st[2], st[3], phi, eps)
                if n or state:
                    check(S1[b:b + 1], Sr, "S_out", True), check(Z1[b:b + 1], Zr, "Z_out", True)
                if state:
                    check(dS0[b:b + 1], rS, "dS_in", True), check(dZ0[b:b + 1], rZ, "dZ_in", True)
                if n:
                    check(O[sl], Or, "O"), check(den[sl], denr, "O den", True)
                    for nm, x, ref in zip(("dQ", "dK", "dV"), grads, (rq, rk, rv)):
                        check(x[sl], ref, nm)


@pytest.mark.parametrize("phi", ["elu1", "identity"])
@pytest.mark.parametrize("N", [1, 64, 127, 128, 129, 1000, 2048, 2049, 4500])
@pytest.mark.parametrize("D", [32, 64])
def test_bidirectional_forward(D, N, phi):
    B, H = 3, 1
    Q, K, V, _ = draw_qkvg(B, H, N, D, D, 5 + N, torch.bfloat16, 0.125)
    if phi == "identity":
        Q, K = Q.abs() + 0.9, K.abs() + 0.9
    dev = [t.to(DEV) for t in (Q, K, V)]
    for lengths in ([N] * B, [N, N // 2 + 1, 0]):
        den, S, Z = torch.empty(B, H, N, device=DEV), torch.empty(B, H, D, D, device=DEV), torch.empty(B, H, D, device=DEV)
        ln = None if lengths[-1] else torch.tensor(lengths, dtype=torch.int32, device=DEV)
        O = la.la_linear_attention(*dev, phi=phi, lengths=ln, den=den, KV=S, Zs=Z)
        la.la_last_device_status()
        for b, n in enumerate(lengths):
            sl = (slice(b, b + 1), slice(None), slice(0, n))
            assert not O[b, :, n:].any() and not den[b, :, n:].any()
            if not n:
                assert not S[b].any() and not Z[b].any()
                continue
            q, k, v = (t[sl].double().numpy() for t in (Q, K, V))
            Or, denr = oracle.linear_attention(q, k, v, causal=False, phi=phi)[:2]
            fk = oracle.feature_map(k) if phi == "elu1" else k
            assert_close(O[sl], Or, torch.bfloat16, "O")
            assert_close(den[sl], denr, torch.bfloat16, "den")
            assert_close(S[b:b + 1], np.einsum("bhnd,bhnm->bhdm", fk, v), torch.bfloat16, "KV")
            assert_close(Z[b:b + 1], fk.sum(2), torch.bfloat16, "Zs")


@pytest.mark.parametrize("D", [32, 64])
@pytest.mark.parametrize("N", [300, 1024, 1025, 2048])
def test_training_steps_follow_each_other(N, D):
    """Steps with and without a saved buffer, enqueued one behind the other on data that changes in between without any host
    synchronisation: the same bits every time, and the forward's do not depend on the buffer."""
    sets = [[t.to(DEV) for t in draw_qkvg(1, 4, N, D, D, seed, torch.bfloat16, 1.0)] for seed in (1, 2)]
    buf = [torch.empty_like(t) for t in sets[0]]
    saved = la.saved_buffer(buf[0], buf[2])
    sums = la.linear_saved_buffer(buf[0], buf[2])

    def step(i):
        for b, t in zip(buf, sets[i % 2]):
            b.copy_(t)
        out = [la.la_causal_forward(*buf[:3], saved=saved if i % 4 < 2 else None)]
        out += la.la_causal_backward(*buf, saved=saved if i % 4 < 2 else None)
        out.append(la.la_linear_attention(*buf[:3], saved=sums if i % 4 < 2 else None))
        out += la.la_linear_attention_backward(*buf, saved=sums if i % 4 < 2 else None)
        return out

    steps = [step(i) for i in range(12)]
    la.la_last_device_status()
    for i in range(4, 12):
        assert all(torch.equal(a, b) for a, b in zip(steps[i], steps[i % 4])), i
    for i in (0, 1):                            # (the causal dK and dV agree to rounding only, where the buffer is used)
        assert torch.equal(steps[i][0], steps[i + 2][0]) and torch.equal(steps[i][1], steps[i + 2][1])
        assert all(torch.equal(a, b) for a, b in zip(steps[i][4:], steps[i + 2][4:]))
    q, k, v, g = (t.double().cpu().numpy() for t in sets[0])
    assert_close(steps[0][0], oracle.linear_attention(q, k, v, causal=True)[0], torch.bfloat16, "O")
    for nm, x, ref in zip(("dQ", "dK", "dV"), steps[0][1:4], oracle.linear_attention_backward(q, k, v, g, causal=True)):
        assert_close(x, ref, torch.bfloat16, nm, grad=True)


@pytest.mark.parametrize("dtype,N", [(torch.float32, 1000), (torch.bfloat16, 1024)])
@pytest.mark.parametrize("D", [32, 64])
def test_a_large_state_is_rounded_once(D, N, dtype):
    """A state, or the gradient of one, much larger than what a call adds to it: the sum is rounded once at its size (2^-24 of
    the result).  The sums themselves are held to 2e-6 of their terms' size, in the backward pass of bf16, whose q / dn is
    rounded, to 2^-8."""
    B, H = 1, 2
    Q, K, V, G = draw_qkvg(B, H, N, D, D, 21, dtype, 1.0)
    Q, K = Q.abs() + 0.1, K.abs() + 0.1
    g = torch.Generator().manual_seed(22)
    S0, Z0 = (torch.randn((B, H, D, D), generator=g) + 4) * 1e5, (torch.rand((B, H, D), generator=g) + 1) * 1e6
    S0d, Z0d, q, k, v, gg = (t.to(DEV) for t in (S0, Z0, Q, K, V, G))
    S1, Z1, dS, dZ = (torch.empty_like(t) for t in (S0d, Z0d, S0d, Z0d))
    la.la_causal_forward(q, k, v, phi="identity", S_in=S0d, Z_in=Z0d, S_out=S1, Z_out=Z1)
    la.la_causal_backward(q, k, v, gg, phi="identity", dS_out=S0d, dZ_out=Z0d, dS_in=dS, dZ_in=dZ)
    la.la_last_device_status()
    Q, K, V, G = (t.double().numpy() for t in (Q, K, V, G))
    O, den = oracle.linear_attention(Q, K, V, causal=True, phi="identity")[:2]
    qn, dl = Q / den[..., None], -(G * O).sum(-1, keepdims=True)

    def check(x, x0, a, b, tol, what):
        ref = x0.double().numpy() + np.einsum("bhnd,bhnm->bhdm", a, b).reshape(x0.shape)
        size = np.einsum("bhnd,bhnm->bhdm", abs(a), abs(b)).reshape(x0.shape)
        err = abs(x.double().cpu().numpy() - ref) / (2.0 ** -24 * 1.001 * abs(ref) + tol * size)
        assert err.max() <= 1, (what, err.max())

    ones, tol = np.ones_like(dl), 2e-6 if dtype == torch.float32 else 2.0 ** -8
    check(S1, S0, K, V, 2e-6, "S_out"), check(Z1, Z0, K, ones, 2e-6, "Z_out")
    check(dS, S0, qn, G, tol, "dS_in"), check(dZ, Z0, qn, dl, tol, "dZ_in")


def kernels_of(call):
    """The library's kernels that a call launches, with how often."""
    la.la_profile_enable(True)
    try:
        call()
        la.la_last_device_status()
        return {k: n for k, (_, n) in la.la_profile_read().items()}
    finally:
        la.la_profile_enable(False)


def test_these_kernels_are_profiled_under_their_own_names():
    Q, K, V, G = (t.to(DEV) for t in draw_qkvg(1, 2, 500, 64, 64, 1, torch.bfloat16, 1.0))
    assert kernels_of(lambda: la.la_causal_forward(Q, K, V)) == {"causal_cluster_forward_kernel": 1}
    assert kernels_of(lambda: la.la_causal_backward(Q, K, V, G)) == {"causal_cluster_backward_kernel": 1}
    assert kernels_of(lambda: la.la_linear_attention(Q, K, V)) == {"linear_cluster_forward_kernel": 1}
    saved = la.linear_saved_buffer(Q, V)
    assert kernels_of(lambda: la.la_linear_attention(Q, K, V, saved=saved)) == {"linear_warp_sum_kernel": 1, "linear_cluster_forward_kernel": 1}


@pytest.fixture(scope="module")
def small_context():
    """A stream whose context has eight of the device's SMs: no room for a cluster of more than eight CTAs."""
    cu = pytest.importorskip("cuda.bindings.driver")

    def ok(r):
        assert r[0] == cu.CUresult.CUDA_SUCCESS, r[0]
        return r[1] if len(r) == 2 else r[1:]

    torch.zeros(1, device=DEV)
    dev = ok(cu.cuDeviceGet(0))
    sms = ok(cu.cuDeviceGetDevResource(dev, cu.CUdevResourceType.CU_DEV_RESOURCE_TYPE_SM))
    groups, _, _ = ok(cu.cuDevSmResourceSplitByCount(1, sms, 0, 8))
    ctx = ok(cu.cuGreenCtxCreate(ok(cu.cuDevResourceGenerateDesc(groups, 1)), dev, cu.CUgreenCtxCreate_flags.CU_GREEN_CTX_DEFAULT_STREAM))
    # (kept for the life of the process: the allocator remembers the stream)
    return torch.cuda.ExternalStream(int(ok(cu.cuGreenCtxStreamCreate(ctx, cu.CUstream_flags.CU_STREAM_NON_BLOCKING, 0))))


@pytest.mark.parametrize("dtype,phi,D,M,N", [(torch.bfloat16, "elu1", 64, 64, 1030), (torch.bfloat16, "elu1", 32, 32, 1030),
                                             (torch.bfloat16, "elu1", 32, 32, 600), (torch.bfloat16, "elu1", 64, 64, 600),
                                             (torch.float32, "elu1", 64, 64, 600), (torch.float32, "elu1", 32, 32, 600),
                                             (torch.bfloat16, "identity", 128, 64, 600)])
def test_a_context_without_room_for_a_cluster(small_context, dtype, phi, D, M, N):
    """The other kernels take the problem: same results to the usual tolerances, with a saved buffer too, whichever of the two
    calls of a step ran where there was room."""
    Q, K, V, G = draw_qkvg(1, 2, N, D, M, 31, dtype, 1.0 if D != 32 else 0.5)
    if phi == "identity":
        Q, K = Q.abs() + 0.1, K.abs() + 0.1
    dev = [t.to(DEV) for t in (Q, K, V, G)]
    q, k, v, g = (t.double().numpy() for t in (Q, K, V, G))
    Or, grads = oracle.linear_attention(q, k, v, causal=True, phi=phi)[0], oracle.linear_attention_backward(q, k, v, g, causal=True, phi=phi)
    Ob = oracle.linear_attention(q, k, v, causal=False, phi=phi)[0]
    streams = {"here": torch.cuda.current_stream(), "there": small_context}
    torch.cuda.synchronize()
    for f, b in (("there", "there"), ("here", "there"), ("there", "here")):
        saved = la.saved_buffer(dev[0], dev[2], phi=phi)
        torch.cuda.synchronize()
        with torch.cuda.stream(streams[f]):
            if f == "there" and N > 1024:
                n0 = la.la_kernel_launches()
                la.la_causal_forward(*dev[:3], phi=phi)
                assert la.la_kernel_launches() > n0 + 1
            O = la.la_causal_forward(*dev[:3], phi=phi, saved=saved)
            E = la.la_linear_attention(*dev[:3], phi=phi)
            la.la_last_device_status()
        with torch.cuda.stream(streams[b]):
            out = la.la_causal_backward(*dev, phi=phi, saved=saved)
            la.la_last_device_status()
        for x, ref, nm in ((O, Or, "O"), (E, Ob, "E"), *zip(out, grads, ("dQ", "dK", "dV"))):
            if D == M and dtype == torch.bfloat16:
                assert_close(x, ref, dtype, f"{nm}, forward {f}, backward {b}", grad=nm[0] == "d")
            else:
                _close(x, ref, (8e-6 if nm[0] == "d" else 2e-6) if dtype == torch.float32 else 2 ** -7, nm)


SUM, FWD, MMA = "segment_sum_kernel", "causal_fwd_kernel", "causal_mma_forward_kernel"
CLUSTER, GRADIENTS = "causal_cluster_forward_kernel", "causal_cluster_backward_kernel"


@pytest.mark.parametrize("dtype,D,BHN,state,saved,want", [
    (torch.bfloat16, 64, (6, 8, 1024), False, False, {CLUSTER}),               # two waves ...
    (torch.bfloat16, 64, (6, 8, 1024), False, True, {SUM, FWD}),               # ... are none with the records on top
    (torch.bfloat16, 64, (6, 8, 500), False, True, {SUM, CLUSTER}),            # one wave is, beside the pre-pass
    (torch.bfloat16, 64, (4, 8, 2048), False, False, {SUM, FWD}),              # three waves
    (torch.bfloat16, 64, (2, 8, 384), False, False, {CLUSTER}),                # three tiles, an SM each ...
    (torch.bfloat16, 64, (6, 8, 384), False, False, {FWD}),                    # ... or shared ...
    (torch.bfloat16, 64, (6, 8, 384), True, False, {CLUSTER}),                 # ... from a state
    (torch.bfloat16, 64, (1, 8, 256), False, False, {FWD}),
    (torch.bfloat16, 32, (7, 8, 300), False, False, {CLUSTER}),
    (torch.bfloat16, 32, (7, 14, 300), False, False, {FWD}),                   # a second wave of three tiles
    (torch.bfloat16, 32, (5, 8, 1024), False, True, {SUM, CLUSTER}),
    (torch.float32, 64, (4, 8, 128), False, False, {CLUSTER}),
    (torch.float32, 64, (12, 8, 128), False, False, {MMA}),                    # a second wave of two tiles
    (torch.float32, 64, (4, 8, 64), False, False, {MMA}),
    (torch.float32, 32, (12, 8, 192), False, False, {CLUSTER})], ids=str)
def test_which_kernel_takes_a_forward_pass(dtype, D, BHN, state, saved, want):
    B, H, N = BHN
    Q, K, V = (torch.zeros(B, H, N, D, dtype=dtype, device=DEV) for _ in range(3))
    kw = {"S_in": torch.zeros(B, H, D, D, device=DEV), "Z_in": torch.zeros(B, H, D, device=DEV)} if state else {}
    names = kernels_of(lambda: la.la_causal_forward(Q, K, V, saved=la.saved_buffer(Q, V) if saved else None, **kw))
    assert set(names) - {"causal_mma_sum_kernel"} == want


@pytest.mark.parametrize("dtype,D,BHN,cluster", [
    (torch.bfloat16, 64, (1, 8, 257), True), (torch.bfloat16, 64, (1, 8, 256), False), (torch.bfloat16, 64, (1, 12, 1024), True),
    (torch.bfloat16, 64, (1, 13, 1024), False), (torch.bfloat16, 32, (8, 8, 256), True), (torch.bfloat16, 32, (9, 8, 256), False),
    (torch.bfloat16, 32, (6, 8, 384), True), (torch.bfloat16, 32, (1, 8, 64), False), (torch.float32, 64, (4, 8, 128), True),
    (torch.float32, 64, (12, 8, 128), True), (torch.float32, 64, (20, 1, 256), True), (torch.float32, 64, (10, 8, 128), False)], ids=str)
def test_which_kernel_takes_a_backward_pass(dtype, D, BHN, cluster):
    Q, K, V, G = (torch.zeros(*BHN, D, dtype=dtype, device=DEV) for _ in range(4))
    names = kernels_of(lambda: la.la_causal_backward(Q, K, V, G))
    assert (set(names) == {GRADIENTS}) if cluster else (len(names) > 1 and GRADIENTS not in names)


@pytest.mark.parametrize("D,BHN,cluster", [(64, (1, 8, 1536), True), (64, (1, 8, 1537), False), (64, (18, 8, 128), True), (64, (19, 8, 128), False),
                                           (32, (56, 8, 128), True), (32, (57, 8, 128), False), (32, (4, 8, 1700), False), (32, (3, 8, 2048), True),
                                           (32, (1, 8, 8192), True), (32, (1, 8, 8193), False), (32, (2, 8, 2049), False)], ids=str)
def test_which_kernel_takes_a_bidirectional_forward_pass(D, BHN, cluster):
    Q, K, V = (torch.zeros(*BHN, D, dtype=torch.bfloat16, device=DEV) for _ in range(3))
    want = {"linear_cluster_forward_kernel"} if cluster else {"linear_warp_sum_kernel", "linear_warp_apply_kernel"}
    assert set(kernels_of(lambda: la.la_linear_attention(Q, K, V))) == want
    saved = la.linear_saved_buffer(Q, V)
    assert set(kernels_of(lambda: la.la_linear_attention(Q, K, V, saved=saved))) == want | {"linear_warp_sum_kernel"}


@pytest.mark.parametrize("dtype,phi,D,M", CAUSAL)
def test_a_zero_state_changes_nothing(dtype, phi, D, M):
    """A sequence may start from a state of zeros: the same results bit for bit as from none."""
    dev = [t.to(DEV) for t in draw_qkvg(2, 2, 500, D, M, 3, dtype, 1.0)]
    if phi == "identity":
        dev[0], dev[1] = dev[0].abs() + 0.1, dev[1].abs() + 0.1
    state = {"S_in": torch.zeros(2, 2, D, M, device=DEV), "Z_in": torch.zeros(2, 2, D, device=DEV)}
    plain = (la.la_causal_forward(*dev[:3], phi=phi), *la.la_causal_backward(*dev, phi=phi))
    from_zero = (la.la_causal_forward(*dev[:3], phi=phi, **state), *la.la_causal_backward(*dev, phi=phi, **state))
    la.la_last_device_status()
    assert all(torch.equal(a, b) for a, b in zip(plain, from_zero))
