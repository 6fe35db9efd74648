"""The decode GEMV's fused quantiser at 5-16 tokens against the stand-alone one, bit for bit, on rows that
leave its fast path (NaN, infinities, rows of zeros and of values so small that 127 / max overflows) beside
ordinary rows, with the constants in shared memory and read from global memory, and against the FFN
block, whose down projection takes its row maxima from the gate/up launch."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K,N", [(1152, 6912), (6912, 1152), (1040, 72), (16, 64)])
@pytest.mark.parametrize("M", [5, 8, 11, 16])
def test_codes_match_the_standalone_quantiser(M, K, N):
    from paper_2608_28003_gb300 import build
    build.build()
    from paper_2608_28003_gb300 import binding as B
    g = torch.Generator("cuda").manual_seed(K + M)
    x = torch.randn(M, K, device="cuda", generator=g)
    x[1, 3], x[1, 5] = float("nan"), -float("nan")
    x[2, 1] = float("inf")
    x[3] = 0.0
    x[4] *= 1e-38           # 127 / max is infinite: codes +-127, 0 for zeros
    x[4, ::2] = 0.0
    x = x.to(torch.bfloat16)
    w = torch.randn(N, K, device="cuda", generator=g).to(torch.bfloat16) * 0.02
    q = B.prepare_weights(w, torch.rand(K, device="cuda", generator=g) + 0.5, want_f16=True)
    y, dbg = B.linear(q, x, debug=True)
    xq, _, s_x = B.quantize_activations(x, q.inv_delta)
    assert torch.equal(dbg["xq"], xq)
    assert torch.equal(dbg["s_x"].view(torch.int32), s_x.view(torch.int32))
    acc = xq.double() @ q.wq.double().t()
    assert torch.equal(dbg["acc"].double(), acc)
    want = (s_x[:, None] * q.s_w[None, :]) * acc.float()
    assert torch.equal(y.view(torch.int16), want.to(torch.bfloat16).view(torch.int16)) or \
        torch.equal(torch.nan_to_num(y.float()), torch.nan_to_num(want.to(torch.bfloat16).float()))


@pytest.mark.parametrize("F", [32, 4112, 6912])  # fused quantiser; known maxima: a ragged second chunk; the decoder's
@pytest.mark.parametrize("M", [5, 8, 16])
def test_ffn_down_equals_the_linear_on_its_input(M, F):
    from paper_2608_28003_gb300 import build
    build.build()
    from paper_2608_28003_gb300 import binding as B
    H = 1152
    g = torch.Generator("cuda").manual_seed(F + M)
    x = torch.randn(M, H, device="cuda", generator=g)
    x[1, 3], x[2], x[3, 1] = float("nan"), 0.0, 1e38
    x = x.to(torch.bfloat16)
    wg, wu = (torch.randn(F, H, device="cuda", generator=g).to(torch.bfloat16) * 0.05 for _ in range(2))
    wd = torch.randn(H, F, device="cuda", generator=g).to(torch.bfloat16) * 0.05
    gu = B.prepare_gate_up(wg, wu, torch.rand(H, device="cuda", generator=g) + 0.5)
    dn = B.prepare_weights(wd, torch.rand(F, device="cuda", generator=g) + 0.5)
    f = B.FfnWeights(H, F, gu, dn, B.interleave_gate_up(wg, wu), wd)
    y, h = B.ffn_block(f, B.W8A8_PREC_W8A8, x, want_h=True)
    want = B.linear(f.down, h)
    assert torch.equal(y.view(torch.int16), want.view(torch.int16))
