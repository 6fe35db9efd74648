"""Prefill attention on the tensor cores against the oracle decoder (two layers, one global and one with
a window shorter than a key tile): query blocks and key tiles with ragged ends, one and two CTAs per
query block, a second CTA without keys, and prompts fed in chunks that start at any position; and the head
layouts: several key/value heads, one or more query heads on each, with and without the QK-norm."""
import numpy as np
import pytest
import torch

import synth
from oracle import decoder as OD
from oracle import masks as OM

pytestmark = pytest.mark.gpu

L, H, F, V, WINDOW, SEQ = 2, 1152, 256, 1024, 100, 320


def _decoders(batch, n_q=4, n_kv=1, qk_norm=True):
    """The decoder and the oracle's on the same weights."""
    from paper_2608_28003_gb300 import build
    build.build()
    from paper_2608_28003_gb300 import binding as B
    f32, bf, norms = synth.decoder_weights(L, H, F, V, n_q=n_q, n_kv=n_kv, seed=9)
    w = {k: [t.cuda() for t in v] if isinstance(v, list) else v.cuda() for k, v in bf.items()}
    n = {k: [torch.from_numpy(a).cuda() for a in v] if isinstance(v, list) else torch.from_numpy(v).cuda()
         for k, v in norms.items()}
    shape = dict(layers=L, inter=F, vocab=V, window=WINDOW, global_layers=(0,), n_q=n_q, n_kv=n_kv, qk_norm=qk_norm)
    ow = dict(f32)
    ow.update(norms)
    return (B.Decoder(B.DecoderConfig(max_batch=batch, max_seq=SEQ, max_tokens=batch * SEQ, **shape), w, n),
            OD.OracleDecoder(OD.DecoderConfig(**shape), ow, batch=batch, max_len=SEQ))


@pytest.fixture(scope="module")
def setup():
    dec, od = _decoders(8)
    toks = synth.tokens(8 * 300, V, seed=4).reshape(8, 300)
    return dec, toks, od.forward(toks, 0, OM.make_mask())["logits"]


@pytest.mark.parametrize("batch,chunks", [(8, [300]),            # 96 query blocks: one CTA each
                                          (1, [257]), (2, [128]), (1, [2]),
                                          (2, [37, 130, 3]),     # keys of earlier calls, unaligned starts
                                          (1, [129, 127, 44])])
def test_chunked_prefill_matches_oracle(setup, batch, chunks):
    dec, toks, ref = setup
    _check_chunks(dec, toks[:batch], ref[:batch], chunks)


def _check_chunks(dec, toks, ref, chunks):
    batch = len(toks)
    t = torch.from_numpy(toks).cuda()
    pos = 0
    for c in chunks:
        logits, top1 = dec.forward(t[:, pos:pos + c].clone(memory_format=torch.contiguous_format), pos)
        got = logits.view(batch, c, V).cpu().numpy().astype(np.float64)
        want = ref[:, pos:pos + c]
        rel = np.linalg.norm(got - want, axis=-1) / np.linalg.norm(want, axis=-1)
        assert rel.max() <= 1e-2, (pos, float(rel.max()))  # the decoder's stated tolerance, all bf16
        pos += c


@pytest.mark.parametrize("n_q,n_kv,qk_norm", [(4, 2, True), (4, 4, False), (6, 2, False)])
def test_head_layouts_match_oracle(n_q, n_kv, qk_norm):
    dec, od = _decoders(3, n_q, n_kv, qk_norm)
    toks = synth.tokens(3 * 170, V, seed=5).reshape(3, 170)
    _check_chunks(dec, toks, od.forward(toks, 0, OM.make_mask())["logits"], [37, 130, 3])
