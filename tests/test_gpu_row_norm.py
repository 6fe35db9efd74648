"""The residual + norm step of long prompts (a warp per row) in a traced prefill, against fp64 on the
step's own inputs: rows that do not fill the last block, one to five vectors per lane, and the row count
at which the block-per-row kernel hands over."""
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H", [256, 1152, 1280, 1296])  # 1296: past the warp kernel's width
@pytest.mark.parametrize("T", [511, 512, 513])
def test_residual_norm_rows(H, T):
    from paper_2608_28003_gb300 import build
    build.build()
    from paper_2608_28003_gb300 import binding as B
    V, F = 512, 64
    _, bf, norms = synth.decoder_weights(1, H, F, V, seed=H, want_f32=False)
    w = {k: [t.cuda() for t in v] if isinstance(v, list) else v.cuda() for k, v in bf.items()}
    g = torch.Generator().manual_seed(H)
    n = {k: [torch.rand(len(a), generator=g).add_(0.5).cuda() for a in v] if isinstance(v, list)
         else torch.from_numpy(v).cuda() for k, v in norms.items()}
    dec = B.Decoder(B.DecoderConfig(layers=1, hidden=H, inter=F, vocab=V, max_batch=1, max_seq=640, max_tokens=640), w, n)
    toks = torch.from_numpy(synth.tokens(T, V, seed=5)).cuda().view(1, T)
    tr = dec.set_trace(T)
    dec.forward(toks, 0)
    torch.cuda.synchronize()

    def unit(x):
        return x * torch.rsqrt(x.square().mean(-1, keepdim=True) + 1e-6)

    r = (w["embed"][toks[0].long()].float() * torch.tensor(H, dtype=torch.float64).sqrt().float().cuda()).double()
    r = r + unit(tr["y_o"][0, :T].double()) * n["ln_post_attn"][0].double()
    a = unit(r) * n["ln_pre_ffn"][0].double()
    # bf16 rounding (8 significant bits: half an ulp is at most 2^-8 of the value) of a value whose fp32 sums over H terms are within H 2^-24 of exact
    bound = (2.0 ** -8 + 4 * H * 2.0 ** -24) * a.abs() + 1e-6
    assert bool(((tr["a_ffn"][0, :T].double() - a).abs() <= bound).all())
    r = r + unit(tr["y_f"][0, :T].double()) * n["ln_post_ffn"][0].double()
    assert bool(((tr["r"][0, :T].double() - r).abs() <= 4 * H * 2.0 ** -24 * (r.abs() + 4.0)).all())
    dec.set_trace(None)
