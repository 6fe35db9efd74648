"""The tcgen05 GEMM's epilogue at the edges of its fast paths: GeGLU of gates inside and outside the
range that the packed recipe takes (zeros, tiny, far negative and huge gates, on full and ragged
column groups), and the lm_head's top-1 with ties across column groups, all-negative logits beside the
zero columns past a ragged vocabulary, and equal maxima in different tiles."""
import numpy as np
import pytest
import torch

import synth
from oracle import blocks as OB
from oracle import w8a8 as OW

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2608_28003_gb300 import build
    build.build()
    from paper_2608_28003_gb300 import binding
    return binding


@pytest.mark.parametrize("inter", [528, 1536])  # 2 x 528 columns: the last 32-column group is whole, the tile ragged
@pytest.mark.parametrize("M", [40, 130, 700])   # 64-, 128-column and pair tiles
def test_geglu_gate_ranges_bit_exact(B, M, inter):
    H = 256
    c = synth.ffn_case(M, seed=M, hidden=H, inter=inter, calib_rows=32)
    wg32, wg = c["wg32"].copy(), c["wg"].clone()
    wg32[3:inter:7] = 0.0  # gates that are exactly zero
    wg[3:inter:7] = 0.0
    scale = np.array([1.0, 0.0, 2.0 ** -40, 16.0, 2.0 ** -80, 2.0 ** 14, 4.0, 2.0 ** 45], np.float32)
    x32 = c["x32"] * scale[np.arange(M) % 8][:, None]  # powers of two: still bf16 values
    x = torch.from_numpy(x32).to(torch.bfloat16)
    stat = OW.act_absmax(c["calib32"])
    f = B.FfnWeights(H, inter, B.prepare_gate_up(wg.cuda(), c["wu"].cuda(), torch.from_numpy(stat).cuda(), want_f16=True),
                     B.prepare_weights(c["wd"].cuda(), torch.from_numpy(c["stat_h"]).cuda(), want_f16=True))
    _, h = B.ffn_block(f, B.W8A8_PREC_W8A8, x.cuda(), want_h=True)
    r = OB.ffn_w8a8(x32, OB.prepare_ffn(wg32, c["wu32"], c["wd32"], stat, c["stat_h"]))
    got = h.cpu().float().numpy()
    assert np.array_equal(got.view(np.uint32), r["h"].astype(np.float32).view(np.uint32))


@pytest.mark.parametrize("vocab", [4112, 4096])  # 16 columns past the last whole group; none
@pytest.mark.parametrize("M", [70, 300])
@pytest.mark.parametrize("prec", [0, 1])
def test_top1_ties_and_negative_logits(B, prec, M, vocab):
    H = 256
    g = np.random.default_rng([M, vocab])
    w32, w = synth.to_bf16(-np.abs(synth.normal((vocab, H), 0.02, g)) - np.float32(0.004))
    x32, x = synth.to_bf16(np.abs(synth.normal((M, H), 1.0, g)) + np.float32(0.1))
    best = synth.to_bf16(np.full(H, -0.001, np.float32))[0]
    for row in (37, 40, 1029, vocab - 1):  # equal, and the largest: the lowest index wins
        w32[row] = best
    w = torch.from_numpy(w32).to(torch.bfloat16)
    x32[M // 2] = 0.0                      # all logits equal (zero)
    x = torch.from_numpy(x32).to(torch.bfloat16)
    stat = OW.act_absmax(np.abs(x32) + np.float32(1.0))
    hd = B.HeadWeights(vocab, H, B.prepare_weights(w.cuda(), torch.from_numpy(stat).cuda(), want_f16=True), w.cuda())
    logits, top1 = B.lm_head(hd, B.W8A8_PREC_W8A8 if prec else B.W8A8_PREC_BF16, x.cuda())
    lg, t = logits.cpu().numpy(), top1.cpu().numpy()
    assert np.all(lg <= 0.0)
    assert np.array_equal(t, np.argmax(lg, axis=1))
    want = np.full(M, 37)
    want[M // 2] = 0
    assert np.array_equal(t, want)
    if prec:
        r = OB.lm_head_w8a8(x32, OW.prepare_weights(w32, stat))
        assert np.array_equal(lg.view(np.uint32) & 0x7fffffff, r["logits"].view(np.uint32) & 0x7fffffff)
