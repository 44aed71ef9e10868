"""Infinite and NaN encoder frames in one stream of a call: the other streams'
results keep their bits, every label stays in range and the decoder goes on."""
import numpy as np
import pytest

import synth
from tests import parity_util as pu

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _decode(inp, w, enc, **kw):
    """Tokens, frames, scores and counts of every chunk."""
    import paper_2609_14991_gb300 as tsd

    dev = torch.device("cuda", 0)
    lm = tsd.NGram.from_arrays(inp.lmA)
    bo = tsd.Boost.from_phrases(w.V, inp.ph, w.bonus)
    dec = tsd.Decoder(w.V, w.H, torch.from_numpy(inp.W.view(np.int16)).to(dev), torch.from_numpy(inp.E.view(np.int16)).to(dev),
                      lm=lm, boost=bo, max_symbols=w.max_sym, max_streams=w.B, max_T=w.T, **kw)
    slots = [dec.open() for _ in range(w.B)]
    out = []
    for e in enc:
        o = dec.decode_chunk(slots, torch.from_numpy(e.view(np.int16)).to(dev), inp.lam, inp.beta)
        torch.cuda.synchronize()
        out.append([x.cpu().numpy() for x in (o.tokens, o.frames, o.scores, o.counts)])
    dec.check()
    hyps = [dec.hyps(s) for s in slots] if kw.get("beam_k", 1) > 1 else None
    return out, hyps


# +inf, -inf, NaN, and the largest finite value (whose logits overflow)
BAD = [0x7F80, 0xFF80, 0x7FC0, 0x7F7F]


@pytest.mark.parametrize("K,S", [(2, 1), (4, 1), (8, 1), (3, 3), (8, 2)])
def test_beam(K, S):
    w = synth.scaled(synth.WORKLOADS[0], V=100, H=128, B=6, T=5, beam=K, max_sym=S, lm_total=2000)
    inp = pu.Inputs(w, lmA=synth.ngram_lm(7, w.V, 3, 2000, 1.1), ph=synth.phrases(7, w.V, 6, 1, 3, 0.0))
    enc = [synth.enc_chunk(w, range(w.B), c) for c in range(3)]
    good, good_h = _decode(inp, w, enc, beam_k=K)
    bad = [e.copy() for e in enc]
    for i, v in enumerate(BAD):  # streams 1 .. 4, one element and a whole frame
        bad[0][1 + i, 2, 5] = v
        bad[1][1 + i, 1, :] = v
    got, got_h = _decode(inp, w, bad, beam_k=K)
    for i in (0, 5):
        for c in range(3):
            assert got[c][3][i] == good[c][3][i]
        assert got_h[i] == good_h[i]
    for c in range(3):
        for i in range(w.B):
            n = got[c][3][i]
            assert 0 <= n <= 3 * w.T * S
    for h in got_h:
        assert len(h) <= K and all(0 <= t < w.V for toks, _ in h for t in toks)
