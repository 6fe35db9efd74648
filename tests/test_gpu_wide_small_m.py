"""lm_head-sized outputs at few tokens: the streaming kernel to 16, the tensor-core GEMM from 17, on both
sides of the line and at a ragged vocabulary, logits and top-1 against the oracle, and the precision of the
bf16 logits that the line keeps."""
import numpy as np
import pytest
import torch

import synth
from oracle import blocks as OB
from oracle import w8a8 as OW

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("vocab", [16400, 20000])
@pytest.mark.parametrize("M", [1, 2, 7, 16, 17, 33, 63])
def test_wide_output_few_tokens(M, vocab):
    from paper_2608_28003_gb300 import build
    build.build()
    from paper_2608_28003_gb300 import binding as B
    c = synth.lm_head_case(M, seed=M, hidden=1040, vocab=vocab, calib_rows=32)
    stat = OW.act_absmax(c["calib32"])
    w = c["w"].cuda()
    hd = B.HeadWeights(vocab, 1040, B.prepare_weights(w, torch.from_numpy(stat).cuda(), want_f16=True), w)
    logits, top1 = B.lm_head(hd, B.W8A8_PREC_W8A8, c["x"].cuda())
    r = OB.lm_head_w8a8(c["x32"], OW.prepare_weights(c["w32"], stat))
    assert np.array_equal(logits.cpu().numpy().view(np.uint32), r["logits"].view(np.uint32))
    assert np.array_equal(top1.cpu().numpy(), r["top1"])
    logits, top1 = B.lm_head(hd, B.W8A8_PREC_BF16, c["x"].cuda())
    r = OB.lm_head_bf16(c["x32"], c["w32"])
    mag = np.abs(c["x32"]).astype(np.float64) @ np.abs(c["w32"]).astype(np.float64).T
    lg = logits.cpu().numpy()
    assert np.all(np.abs(lg - r["logits"]) <= 1040 * 2.0 ** -24 * mag + 1e-30)  # fp32 sums, any order
    assert np.array_equal(top1.cpu().numpy(), lg.argmax(axis=1))


@pytest.mark.parametrize("M,K", [(32, 1152), (33, 1152), (33, 1792), (33, 1808), (64, 1152), (100, 1024)])
def test_split_line_of_short_k_ranges(M, K):
    """Both sides of the rule that leaves short k ranges whole from 33 tokens: the plan, and the W8A8
    linear bit for bit."""
    from paper_2608_28003_gb300 import build
    build.build()
    from paper_2608_28003_gb300 import binding as B
    N = 1152
    split = B.tc_gemm_plan("int8", M, N, K)[2]
    assert (split > 1) == (M <= 32 or K > 28 * 64), split
    x32, x, ch = synth.activations(M, K, 8, seed=M)
    w32, w = synth.weight(N, K, seed=K)
    stat = OW.act_absmax(x32)
    q = B.prepare_weights(w.cuda(), torch.from_numpy(stat).cuda(), want_f16=True)
    y = B.linear(q, x.cuda())
    r = OW.w8a8_linear(x32, OW.prepare_weights(w32, stat), out="bf16")
    assert np.array_equal(y.float().cpu().numpy(), r["y"])


@pytest.mark.parametrize("vocab", [16400, 16392, 600, 40960])  # ragged, not a multiple of 16, few rows; no split row group
@pytest.mark.parametrize("M", [1, 4, 8])
def test_bf16_head_runs_in_the_queried_workspace(M, vocab):
    from paper_2608_28003_gb300 import build
    build.build()
    from paper_2608_28003_gb300 import binding as B
    c = synth.lm_head_case(M, seed=M, hidden=1152, vocab=vocab, calib_rows=8)
    ws = B.Workspace(torch.device("cuda", 0))
    ws.buf = torch.zeros(B._size("w8a8_lm_head_workspace_size", M, vocab, 1152), dtype=torch.uint8, device="cuda")
    hd = B.HeadWeights(vocab, 1152, bf16=c["w"].cuda())
    logits, top1 = B.lm_head(hd, B.W8A8_PREC_BF16, c["x"].cuda(), ws=ws)
    r = OB.lm_head_bf16(c["x32"], c["w32"])
    mag = np.abs(c["x32"]).astype(np.float64) @ np.abs(c["w32"]).astype(np.float64).T
    lg = logits.cpu().numpy()
    assert np.all(np.abs(lg - r["logits"]) <= 1152 * 2.0 ** -24 * mag + 1e-30)
    assert np.array_equal(top1.cpu().numpy(), lg.argmax(axis=1))


@pytest.mark.parametrize("M,bound", [(1, 4e-7), (5, 4e-7), (8, 4e-7), (9, 8e-7), (16, 8e-7)])
def test_bf16_logits_keep_the_split_sums(M, bound):
    """Relative error against 64 bits: four chains per output to 8 tokens (measured 2.5e-7) and two to 16
    (5.4e-7); one accumulator over all of K has 1.1e-6."""
    from paper_2608_28003_gb300 import build
    build.build()
    from paper_2608_28003_gb300 import binding as B
    g = torch.Generator("cuda").manual_seed(M)
    w = (torch.randn(32768, 1152, device="cuda", generator=g) * 0.02).to(torch.bfloat16)
    x = torch.randn(M, 1152, device="cuda", generator=g).to(torch.bfloat16)
    logits, _ = B.lm_head(B.HeadWeights(32768, 1152, bf16=w), B.W8A8_PREC_BF16, x)
    want = x.double() @ w.double().t()
    assert float((logits.double() - want).norm() / want.norm()) <= bound
