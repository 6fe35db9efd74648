"""The per-token codes of the decode GEMV at 3-16 tokens, from its own prologue and from a launch before it,
against a host statement of the rule, bit for bit, on rows that leave the usual range (NaN, infinities, rows
of zeros and of values so small that 127 / max overflows) beside ordinary rows; and the FFN blocks, whose
down projection takes its row maxima from the gate/up launch, against the linear on their h."""
import numpy as np
import pytest
import torch

from oracle import fp8 as OF

pytestmark = pytest.mark.gpu


def _rows(M, K):
    g = torch.Generator("cuda").manual_seed(K + M)
    x = torch.randn(M, K, device="cuda", generator=g)
    x[0, 3], x[0, 5] = float("nan"), -float("nan")
    x[1, 1] = float("inf")
    x[2] *= 1e-38           # 127 / max is infinite: codes +-127, 0 for zeros
    x[2, ::2] = 0.0
    if M > 4:
        x[3] = 0.0
    return x.to(torch.bfloat16), g


def _scaled(x, inv_delta, qmax):
    """s_x and fl(x_hat fl(qmax / m)) of the rows, NaN left out of the maxima."""
    with np.errstate(all="ignore"):
        xh = x.float().cpu().numpy() * inv_delta.cpu().numpy()[None, :]
        m = np.fmax.reduce(np.abs(xh), axis=1)
        r = np.where(m > 0, np.float32(qmax) / m, np.float32(0)).astype(np.float32)
        return (m / np.float32(qmax)).astype(np.float32), (xh * r[:, None]).astype(np.float32)


SHAPES = [(1152, 6912), (6912, 1152), (1040, 72), (16, 64), (2048, 2304)]


@pytest.mark.parametrize("K,N", SHAPES)
@pytest.mark.parametrize("M", [5, 8, 11, 16])
def test_int8_codes(M, K, N):
    from paper_2608_28003_gb300 import build
    build.build()
    from paper_2608_28003_gb300 import binding as B
    x, g = _rows(M, K)
    w = torch.randn(N, K, device="cuda", generator=g).to(torch.bfloat16) * 0.02
    q = B.prepare_weights(w, torch.rand(K, device="cuda", generator=g) + 0.5, want_f16=True)
    y, dbg = B.linear(q, x, debug=True)
    s, p = _scaled(x, q.inv_delta, 127.0)
    codes = np.where(np.isnan(p), 0, np.clip(np.rint(p), -127, 127)).astype(np.int8)
    assert np.array_equal(dbg["xq"].cpu().numpy(), codes)
    assert np.array_equal(dbg["s_x"].cpu().numpy().view(np.uint32), s.view(np.uint32))
    acc = torch.from_numpy(codes).cuda().double() @ q.wq.double().t()
    assert torch.equal(dbg["acc"].double(), acc)
    want = ((dbg["s_x"][:, None] * q.s_w[None, :]) * acc.float()).to(torch.bfloat16)
    assert torch.equal(torch.nan_to_num(y.float(), nan=7.0), torch.nan_to_num(want.float(), nan=7.0))
    assert torch.equal(B.linear(q, x).view(torch.int16), y.view(torch.int16))


@pytest.mark.parametrize("K,N", [(1152, 6912), (6912, 1152), (1040, 80), (16, 64), (2048, 2304)])
@pytest.mark.parametrize("M", [3, 5, 8, 16])
def test_fp8_codes(M, K, N):
    from paper_2608_28003_gb300 import build
    build.build()
    from paper_2608_28003_gb300 import binding as B
    x, g = _rows(M, K)
    w = torch.randn(N, K, device="cuda", generator=g).to(torch.bfloat16) * 0.02
    q = B.fp8_prepare_weights(w, torch.rand(K, device="cuda", generator=g) + 0.5)
    y, dbg = B.fp8_linear(q, x, debug=True)
    s, p = _scaled(x, q.inv_delta, 448.0)
    assert np.array_equal(OF.e4m3_decode(dbg["xq"].cpu().numpy()), OF.e4m3_round(p), equal_nan=True)
    assert np.array_equal(dbg["s_x"].cpu().numpy().view(np.uint32), s.view(np.uint32))
    xv = torch.from_numpy(OF.e4m3_round(p)).cuda()
    wv = torch.from_numpy(OF.e4m3_decode(q.wq.cpu().numpy())).cuda()
    scale = dbg["s_x"].double()[:, None] * q.s_w.double()[None, :]
    acc, mag = xv @ wv.t(), xv.abs() @ wv.abs().t()
    ok = torch.isfinite(acc * scale)
    # fp32 sums of K products in the kernel's order, then two fp32 roundings and the bf16 one
    bound = ((K * 2.0 ** -23 * mag + 2.0 ** -8 * acc.abs()) * scale + 1e-38)[ok]
    assert bool(((y.double() - acc * scale)[ok].abs() <= bound).all())


@pytest.mark.parametrize("F", [32, 2064, 4112, 6912])  # fused quantiser; its launch, one and several blocks a row
@pytest.mark.parametrize("M", [3, 5, 8, 16])
def test_ffn_down_equals_the_linear_on_its_input(M, F):
    from paper_2608_28003_gb300 import build
    build.build()
    from paper_2608_28003_gb300 import binding as B
    H = 1152
    g = torch.Generator("cuda").manual_seed(F + M)
    x = torch.randn(M, H, device="cuda", generator=g)
    x[1, 3] = float("nan")
    if M > 3:
        x[2], x[3, 1] = 0.0, 1e38
    x = x.to(torch.bfloat16)
    wg, wu = (torch.randn(F, H, device="cuda", generator=g).to(torch.bfloat16) * 0.05 for _ in range(2))
    wd = torch.randn(H, F, device="cuda", generator=g).to(torch.bfloat16) * 0.05
    st, sd = torch.rand(H, device="cuda", generator=g) + 0.5, torch.rand(F, device="cuda", generator=g) + 0.5
    f = B.FfnWeights(H, F, B.prepare_gate_up(wg, wu, st), B.prepare_weights(wd, sd), B.interleave_gate_up(wg, wu), wd)
    y, h = B.ffn_block(f, B.W8A8_PREC_W8A8, x, want_h=True)
    assert torch.equal(y.view(torch.int16), B.linear(f.down, h).view(torch.int16))
    e = B.Fp8FfnWeights(H, F, B.fp8_prepare_gate_up(wg, wu, st), B.fp8_prepare_weights(wd, sd))
    y, h = B.fp8_ffn_block(e, x, want_h=True)
    want = B.fp8_linear(e.down, h)
    assert torch.equal(torch.nan_to_num(y.float(), nan=7.0), torch.nan_to_num(want.float(), nan=7.0))
