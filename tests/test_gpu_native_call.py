"""The native part of the binding does what the Python code behind it does: the same outputs bit for bit, the same
errors, and it leaves everything but plain tensors of the current device to that code."""
import pytest
import torch

import paper_2006_16236_b200 as la
from paper_2006_16236_b200 import binding

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


class _Declines:
    def __getattr__(self, name):
        return lambda *a: NotImplemented


def _calls(dtype, lengths):
    g = torch.Generator(device=DEV).manual_seed(1)
    n = lambda *s, dt=dtype: torch.randn(s, generator=g, device=DEV).to(dt)
    B, H, N, D, M = 2, 3, 70, 64, 64
    Q, K, V, G = n(B, H, N, D), n(B, H, N, D), n(B, H, N, M), n(B, H, N, M)
    S, Z = n(B, H, D, M, dt=torch.float32), n(B, H, D, dt=torch.float32).abs() + 9
    ln = torch.tensor([70, 33], dtype=torch.int32, device=DEV) if lengths else None
    S1, Z1, den = torch.empty_like(S), torch.empty_like(Z), torch.empty(B, H, N, device=DEV)

    def train(fwd, bwd, buffer, **kw):
        saved = buffer(Q, V)
        O = fwd(Q, K, V, saved=saved, den=den, **kw)
        return (O, den.clone(), *bwd(Q, K, V, G, saved=saved, **kw), *bwd(Q, K, V, G, **kw))

    yield lambda: train(la.la_causal_forward, la.la_causal_backward, la.saved_buffer, lengths=ln)
    yield lambda: train(la.la_linear_attention, la.la_linear_attention_backward, la.linear_saved_buffer, lengths=ln)
    yield lambda: (la.la_causal_forward(Q, K, V, phi=0, eps=1, S_in=S, Z_in=Z, S_out=S1, Z_out=Z1, lengths=ln), S1.clone(), Z1.clone())
    yield lambda: (la.la_linear_attention(Q.abs(), K.abs(), V, "identity", 0.5, lengths=ln),)

    def step():
        s, z = S.clone(), Z.clone()
        return la.la_recurrent_step(Q[:, :, 0].contiguous(), K[:, :, 0].contiguous(), V[:, :, 0].contiguous(), s, z), s, z
    yield step
    if dtype == torch.bfloat16:
        x, Wqkv, Wo = n(B, H * D), n(3 * H * D, H * D) * 0.05, n(H * D, H * D) * 0.05

        def layer():
            s, z = S.clone(), Z.clone()
            return la.la_decode_layer_step(x, Wqkv, Wo, s, z), s, z
        yield layer


@pytest.mark.parametrize("lengths", [False, True])
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
def test_same_results_both_ways(dtype, lengths, monkeypatch):
    here = [f() for f in _calls(dtype, lengths)]
    monkeypatch.setattr(binding, "_native", lambda: _Declines())
    for a, b in zip(here, [f() for f in _calls(dtype, lengths)], strict=True):
        assert all(torch.equal(x, y) for x, y in zip(a, b, strict=True))


def test_same_errors_and_outputs_in_place():
    Q = torch.randn(1, 2, 16, 32, device=DEV)
    V = torch.randn(1, 2, 16, 32, device=DEV)
    O = torch.empty_like(V)
    assert la.la_causal_forward(Q, Q, V, O=O) is O
    for bad in (Q[:, :, :8], Q.transpose(1, 2), Q.bfloat16(), Q.cpu()):
        with pytest.raises(ValueError):
            la.la_causal_forward(Q, bad, V)
    with pytest.raises(TypeError):
        la.la_causal_forward(Q.half(), Q.half(), V.half())
    with pytest.raises(KeyError):
        la.la_causal_forward(Q, Q, V, phi="relu")
    with pytest.raises(la.LaError):
        la.la_causal_forward(Q, Q, V, eps=-1.0)
    with pytest.raises(la.LaError):
        la.la_causal_forward(Q, Q, V, S_in=torch.zeros(1, 2, 32, 32, device=DEV))


def test_an_allocation_that_fails_is_an_out_of_memory_error():
    """Outputs and scratch are allocated in native code; a program that catches torch.OutOfMemoryError to go on with a
    smaller batch has to see that type.  The failure is the allocator's: it is told to hold no more than it already does,
    and what it keeps free is taken first."""
    n = lambda *s, dt=torch.float32: torch.zeros(s, device=DEV, dtype=dt)
    Q, Qb = n(1, 8, 65536, 16), n(1, 8, 65536, 64, dt=torch.bfloat16)       # outputs of 33 MB and more
    q, S, Z = n(32768, 8, 32), n(32768, 8, 32, 32), n(32768, 8, 32)
    x, W, Wo = n(32768, 512, dt=torch.bfloat16), n(1536, 512, dt=torch.bfloat16), n(512, 512, dt=torch.bfloat16)
    Sl, Zl = n(32768, 8, 64, 64), n(32768, 8, 64)
    calls = [lambda: la.la_causal_forward(Q, Q, Q), lambda: la.la_causal_backward(Q, Q, Q, Q),
             lambda: la.la_linear_attention(Q, Q, Q), lambda: la.la_linear_attention_backward(Q, Q, Q, Q),
             lambda: la.la_recurrent_step(q, q, q, S, Z), lambda: la.la_decode_layer_step(x, W, Wo, Sl, Zl),
             lambda: la.saved_buffer(Qb, Qb)]
    binding._ws_cache.clear()
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    torch.cuda.set_per_process_memory_fraction(0.0)
    taken = []
    try:
        with pytest.raises(torch.OutOfMemoryError):
            while True:
                taken.append(torch.empty(Q.nbytes, dtype=torch.uint8, device=DEV))
        for call in calls:
            with pytest.raises(torch.OutOfMemoryError):
                call()
    finally:
        torch.cuda.set_per_process_memory_fraction(1.0)
    del taken
    assert torch.isfinite(la.la_causal_forward(Q, Q, Q)).all()


class _Sub(torch.Tensor):
    pass


def test_what_is_not_ordinary_goes_to_the_python_code():
    """A tensor subclass, an active function mode: the native functions decline, nothing done, and the call still works."""
    from torch.overrides import TorchFunctionMode

    class Mode(TorchFunctionMode):
        def __torch_function__(self, func, types, args=(), kwargs=None):
            return func(*args, **(kwargs or {}))

    Q = torch.randn(1, 2, 40, 32, device=DEV)
    want = la.la_causal_forward(Q, Q, Q)
    native = lambda q: binding._native().linear_forward(q, q, q, "elu1", 0.0, None, None, None, None, None, None, None, {})
    launches = la.la_kernel_launches()
    assert native(Q.as_subclass(_Sub)) is NotImplemented
    with Mode():
        assert native(Q) is NotImplemented
    assert native(Q[:, :, ::2]) is NotImplemented and native(Q.half()) is NotImplemented and native(Q.cpu()) is NotImplemented
    assert la.la_kernel_launches() == launches
    assert torch.equal(la.la_causal_forward(Q.as_subclass(_Sub), Q, Q), want)
    with Mode():
        assert torch.equal(la.la_causal_forward(Q, Q, Q), want)


def test_the_current_stream_is_the_one_that_runs():
    """The call is enqueued on the stream that is current, behind what is already there (a delay and the copy that makes its
    input), and nothing on the default stream."""
    Q = torch.randn(1, 2, 300, 32, device=DEV)
    want = la.la_causal_forward(Q, Q, Q)
    side, q, O = torch.cuda.Stream(), torch.zeros_like(Q), torch.empty_like(Q)
    torch.cuda.synchronize()
    with torch.cuda.stream(side):
        torch.cuda._sleep(20_000_000)           # about 10 ms
        q.copy_(Q)
        la.la_causal_forward(q, q, q, O=O)
    assert torch.cuda.default_stream().query()
    side.synchronize()
    assert torch.equal(O, want)
