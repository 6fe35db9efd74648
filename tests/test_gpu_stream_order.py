"""Calls run in stream order with every argument: weights, scales and biases that the call just before
wrote.  The kernels let their dependents start early, so a call's first launch may read nothing ahead of
its wait.  Each pass clears the produced tensor, produces it and uses it without a synchronisation
between; the result equals the one of the same call on the finished tensor, bit for bit."""
import pytest
import torch

pytestmark = pytest.mark.gpu

H, F = 1152, 2304


@pytest.fixture(scope="module")
def B():
    from paper_2608_28003_gb300 import build
    build.build()
    from paper_2608_28003_gb300 import binding
    return binding


def _randn(shape, seed, scale=1.0):
    g = torch.Generator("cuda").manual_seed(seed)
    return (torch.randn(*shape, device="cuda", generator=g) * scale).to(torch.bfloat16)


def _check(make, buf, use, passes=8):
    make()
    torch.cuda.synchronize()
    want = use()
    torch.cuda.synchronize()
    want = [t.clone() for t in want]
    for _ in range(passes):
        buf.zero_()
        make()
        got = use()
        torch.cuda.synchronize()
        for a, b in zip(got, want):
            assert torch.equal(a.view(torch.uint8), b.view(torch.uint8))


def _product(B, rows, cols, seed, ws):
    """A [rows, cols] bf16 tensor and the call that writes it (a prefill-sized GEMM on many CTAs)."""
    x, w = _randn((rows, 6912), seed), _randn((cols, 6912), seed + 1, 0.002)
    buf = torch.empty(rows, cols, dtype=torch.bfloat16, device="cuda")
    return buf, lambda: B.linear_bf16(w, x, out=buf, ws=ws)


@pytest.mark.parametrize("M", [1, 5, 16, 17, 37, 300])
def test_bf16_weight_from_the_call_before(B, M):
    ws = B.Workspace(torch.device("cuda", 0))
    ws.get(256 << 20)
    k, make = _product(B, 1536, H, 1, ws)
    q = _randn((M, H), 2)
    _check(make, k, lambda: [B.linear_bf16(k, q, ws=ws)])
    gu, make = _product(B, 2 * F, H, 3, ws)
    down = _randn((H, F), 4, 0.02)
    f = B.FfnWeights(H, F, gate_up_bf16=gu, down_bf16=down)
    _check(make, gu, lambda: [B.ffn_block(f, B.W8A8_PREC_BF16, q, ws=ws)])
    table, make = _product(B, 20000, 256, 5, ws)
    x = _randn((M, 256), 6)
    hd = B.HeadWeights(20000, 256, bf16=table)
    _check(make, table, lambda: list(B.lm_head(hd, B.W8A8_PREC_BF16, x, ws=ws)))


@pytest.mark.parametrize("M", [1, 4, 8, 16, 33, 300])
def test_scales_and_bias_from_the_call_before(B, M):
    """fp32 logits of one row stand for 1 / delta, the row scales and a bias."""
    ws = B.Workspace(torch.device("cuda", 0))
    ws.get(64 << 20)
    src = B.HeadWeights(H, 6912, bf16=_randn((H, 6912), 7, 0.02))
    row = _randn((1, 6912), 8)
    v, tok = torch.empty(1, H, device="cuda"), torch.empty(1, dtype=torch.int32, device="cuda")

    def make():
        B.lm_head(src, B.W8A8_PREC_BF16, row, logits=v, top1=tok, ws=ws)

    vec = v.view(H)
    ones = torch.ones(H, device="cuda")
    x = _randn((M, H), 9)
    q = B.prepare_weights(_randn((H, H), 10, 0.02), ones, want_f16=True)
    e = B.fp8_prepare_weights(_randn((H, H), 10, 0.02), ones)
    for w in (B.QWeight(q.wq, q.s_w, ones, vec, q.wq_f16), B.QWeight(q.wq, vec, ones, q.inv_delta, q.wq_f16),
              B.QWeight(q.wq, vec, ones, vec)):
        _check(make, v, lambda: [B.linear(w, x, bias=vec, ws=ws)])
    for w in (B.Fp8Weight(e.wq, e.s_w, ones, vec), B.Fp8Weight(e.wq, vec, ones, e.inv_delta)):
        _check(make, v, lambda: [B.fp8_linear(w, x, bias=vec, ws=ws)])
    _check(make, v, lambda: [t for t in B.quantize_activations(x, vec) if t is not None])
    hd = B.HeadWeights(H, H, B.QWeight(q.wq, vec, ones, vec, q.wq_f16))
    _check(make, v, lambda: list(B.lm_head(hd, B.W8A8_PREC_W8A8, x, ws=ws)))
