"""The residual step inside the decode GEMV equals the stand-alone kernel bit for bit: a decode step (fused)
and the same step traced (unfused) give the same logits, at every number of token slots that fuses it."""
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu

L, F, V = 2, 2304, 1024


@pytest.fixture(scope="module", params=[1152, 1536])  # 1536: more vectors a row than a warp keeps in registers
def dec(request):
    from paper_2608_28003_gb300 import build
    build.build()
    from paper_2608_28003_gb300 import binding as B
    H = request.param
    _, bf, norms = synth.decoder_weights(L, H, F, V, seed=H, want_f32=False)
    w = {k: [t.cuda() for t in v] if isinstance(v, list) else v.cuda() for k, v in bf.items()}
    g = torch.Generator().manual_seed(H)
    n = {k: [torch.rand(len(a), generator=g).add_(0.5).cuda() for a in v] if isinstance(v, list)
         else torch.from_numpy(v).cuda() for k, v in norms.items()}
    d = B.Decoder(B.DecoderConfig(layers=L, hidden=H, inter=F, vocab=V, max_batch=8, max_seq=64, max_tokens=512), w, n)
    d.calibrate(torch.from_numpy(synth.tokens(4 * 32, V, seed=1).reshape(4, 32)).cuda())
    d.prepare()
    return d


@pytest.mark.parametrize("int8", [0, 1])
@pytest.mark.parametrize("batch", [1, 2, 3, 4])
def test_fused_step_equals_the_traced_one(dec, batch, int8):
    mask = (1 << L) - 1 if int8 else 0
    dec.set_mask(mask, mask, bool(int8))
    toks = torch.from_numpy(synth.tokens(batch * 9, V, seed=batch)).cuda().view(batch, 9)
    dec.forward(toks[:, :8].contiguous(), 0, want_logits=False)
    tok = toks[:, 8].clone()
    out = torch.empty(batch, V, device="cuda")
    fused = dec.decode_step(tok, 8, logits=out)[0].clone()
    dec.set_trace(batch)
    plain = dec.decode_step(tok, 8, logits=out)[0].clone()
    dec.set_trace(None)
    assert torch.equal(fused.view(torch.int32), plain.view(torch.int32))
