"""The binding's C marshalling: the checks and errors of its calls on the CPU (nothing is launched), and
on the GPU the optional arguments (output, workspace, stream, h, top-1 only) against the plain call."""
import pytest
import torch


@pytest.fixture(scope="module")
def B():
    from paper_2608_28003_gb300 import build
    build.build()
    from paper_2608_28003_gb300 import binding
    return binding


def _qweight(B, n, k, device, f16=True):
    g = torch.Generator().manual_seed(n + k)
    wq = torch.randint(-127, 128, (n, k), generator=g, dtype=torch.int32)
    return B.QWeight(wq.to(torch.int8).to(device), torch.full((n,), 1e-3, device=device), torch.ones(k, device=device),
                     torch.ones(k, device=device), wq.to(torch.float16).to(device) if f16 else None)


def _calls_on(B, x, dev, ws):
    q, qd = _qweight(B, 64, 32, dev), _qweight(B, 32, 32, dev)
    f8 = B.Fp8Weight(q.wq.view(torch.uint8), q.s_w, q.delta, q.inv_delta)
    f8d = B.Fp8Weight(qd.wq.view(torch.uint8), qd.s_w, qd.delta, qd.inv_delta)
    w = torch.zeros(64, 32, dtype=torch.bfloat16, device=dev)
    return [lambda: B.linear(q, x, ws=ws), lambda: B.fp8_linear(f8, x, ws=ws), lambda: B.linear_bf16(w, x, ws=ws),
            lambda: B.ffn_block(B.FfnWeights(32, 32, q, qd), 1, x, ws=ws),
            lambda: B.fp8_ffn_block(B.Fp8FfnWeights(32, 32, f8, f8d), x, ws=ws),
            lambda: B.lm_head(B.HeadWeights(64, 32, q), 1, x, ws=ws)]


def test_host_tensors_are_refused(B):
    ws = B.Workspace(torch.device("cpu"))
    for call in _calls_on(B, torch.zeros(2, 32, dtype=torch.bfloat16), "cpu", ws):
        with pytest.raises(AssertionError, match="contiguous CUDA"):
            call()


def test_wrong_objects_raise(B):
    ws = B.Workspace(torch.device("cpu"))
    x = torch.zeros(2, 32, dtype=torch.bfloat16)
    with pytest.raises(AttributeError):
        B.linear(object(), x, ws=ws)
    with pytest.raises(AttributeError):
        B.linear(_qweight(B, 16, 32, "cpu"), object(), ws=ws)
    with pytest.raises(AttributeError):
        B.ffn_block(None, 1, x, ws=ws)
    with pytest.raises((IndexError, TypeError)):
        B.linear_bf16(torch.zeros(16), x, ws=ws)
    with pytest.raises(ValueError):
        B.linear_bf16(torch.zeros(4, 16, 32, dtype=torch.bfloat16), x, ws=ws)


@pytest.mark.gpu
def test_optional_arguments(B):
    dev = torch.device("cuda", 0)
    x = torch.randn(40, 256, device=dev, generator=torch.Generator(dev).manual_seed(1)).to(torch.bfloat16)
    q, qd = _qweight(B, 1024, 256, dev), _qweight(B, 256, 512, dev)
    y = B.linear(q, x)
    out, ws, st = torch.empty_like(y), B.Workspace(dev), torch.cuda.Stream()
    before = ws.buf.numel()
    st.wait_stream(torch.cuda.current_stream())
    assert B.linear(q, x, out=out, ws=ws, stream=st) is out and ws.buf.numel() > before
    st.synchronize()
    assert torch.equal(out.view(torch.int16), y.view(torch.int16))

    class Counted(B.Workspace):  # a workspace of the caller's own kind is asked for its buffer
        asked = 0

        def get(self, n):
            self.asked += 1
            return super().get(n)
    mine = Counted(dev)
    assert torch.equal(B.linear(q, x, ws=mine).view(torch.int16), y.view(torch.int16)) and mine.asked == 1

    f = B.FfnWeights(256, 512, q, qd)
    y2, h = B.ffn_block(f, B.W8A8_PREC_W8A8, x, want_h=True)
    assert h.shape == (40, 512) and torch.equal(B.ffn_block(f, B.W8A8_PREC_W8A8, x).view(torch.int16), y2.view(torch.int16))
    hd = B.HeadWeights(1024, 256, q)
    logits, top1 = B.lm_head(hd, B.W8A8_PREC_W8A8, x)
    none, only = B.lm_head(hd, B.W8A8_PREC_W8A8, x, want_logits=False)
    assert none is None and torch.equal(only, top1) and torch.equal(logits.argmax(1).int(), top1)
    with pytest.raises(AssertionError, match="contiguous CUDA"):
        B.linear(q, x.t().contiguous().t())
    with pytest.raises(B.W8A8Error) as e:
        B.ffn_block(f, 7, x)
    assert e.value.status == 1
    with pytest.raises(B.W8A8Error):
        B.ffn_block(B.FfnWeights(256, 512), B.W8A8_PREC_W8A8, x)  # no weights of that precision
    assert B.linear(q, x[:0]).shape == (0, 1024)


@pytest.mark.gpu
def test_descriptors_give_what_the_calls_give(B):
    """The ctypes descriptors (c() of the weight classes) through the C ABI, as a caller of lib() uses them,
    against the C module's own marshalling of the same objects."""
    from ctypes import byref
    dev = torch.device("cuda", 0)
    x = torch.randn(8, 256, device=dev, generator=torch.Generator(dev).manual_seed(2)).to(torch.bfloat16)
    q, qd = _qweight(B, 1024, 256, dev), _qweight(B, 256, 512, dev)
    f8 = B.Fp8FfnWeights(256, 512, *(B.Fp8Weight(torch.randint(0, 0x70, t.wq.shape, dtype=torch.uint8, device=dev), t.s_w,
                                                 t.delta, t.inv_delta) for t in (q, qd)))
    f, hd = B.FfnWeights(256, 512, q, qd), B.HeadWeights(1024, 256, q)
    ws = B.Workspace(dev).get(16 << 20)
    y, st = torch.empty(8, 256, dtype=torch.bfloat16, device=dev), B._stream()
    B._check("w8a8_ffn_block", B.lib().w8a8_ffn_block(byref(f.c()), B.W8A8_PREC_W8A8, B._p(x), 8, B._p(y), None, B._p(ws),
                                                      ws.numel(), st))
    assert torch.equal(B.ffn_block(f, B.W8A8_PREC_W8A8, x).view(torch.int16), y.view(torch.int16))
    B._check("w8a8_fp8_ffn_block", B.lib().w8a8_fp8_ffn_block(byref(f8.c()), B._p(x), 8, B._p(y), None, B._p(ws),
                                                              ws.numel(), st))
    assert torch.equal(B.fp8_ffn_block(f8, x).view(torch.int16), y.view(torch.int16))
    logits, top1 = torch.empty(8, 1024, device=dev), torch.empty(8, dtype=torch.int32, device=dev)
    B._check("w8a8_lm_head", B.lib().w8a8_lm_head(byref(hd.c()), B.W8A8_PREC_W8A8, B._p(x), 8, B._p(logits), B._p(top1),
                                                  B._p(ws), ws.numel(), st))
    got = B.lm_head(hd, B.W8A8_PREC_W8A8, x)
    assert torch.equal(got[0].view(torch.int32), logits.view(torch.int32)) and torch.equal(got[1], top1)
