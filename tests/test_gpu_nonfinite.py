"""Infinite and NaN encoder frames in one stream of a call: the other streams'
results keep their bits, every label stays in range and the decoder goes on.
A NaN logit makes its row's scores NaN."""
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


@pytest.mark.parametrize("form", ["one launch", "row pass, few rows", "row pass, many rows", "several lms"])
def test_a_nan_logit_reaches_the_scores(form):
    import paper_2609_14991_gb300 as tsd

    w = synth.scaled(synth.WORKLOADS[0], V=300, H=128, B=480 if form == "row pass, many rows" else 4, T=4, lm_total=6000)
    lmA, ph = synth.ngram_lm(7, w.V, 3, 6000, 1.1), synth.phrases(7, w.V, 6, 1, 3, 0.0)
    E, W = synth.joint_weights(w)
    W = W.copy()
    W[5, 250] = 0x7FC0
    dev = torch.device("cuda", 0)
    lm = tsd.NGram.from_arrays(lmA)
    how = dict(lms=[(lm, 1.0), (lm, 0.5)]) if form == "several lms" else dict(lm=lm)
    dec = tsd.Decoder(w.V, w.H, torch.from_numpy(W.view(np.int16)).to(dev), torch.from_numpy(E.view(np.int16)).to(dev),
                      boost=tsd.Boost.from_phrases(w.V, ph, w.bonus), max_symbols=w.max_sym, max_streams=w.B, max_T=w.T, **how)
    dec.set_option("one_launch", 1 if form == "one launch" else 0)
    slots = [dec.open() for _ in range(w.B)]
    o = dec.decode_chunk(slots, torch.from_numpy(synth.enc_chunk(w, range(w.B), 0).view(np.int16)).to(dev), w.lam, w.beta)
    torch.cuda.synchronize()
    tok, sc, n = (x.cpu().numpy() for x in (o.tokens, o.scores, o.counts))
    dec.check()
    assert n.sum() > 0
    for i in range(w.B):
        assert (tok[i, :n[i]] != 250).all() and np.isnan(sc[i, :n[i]]).all(), (i, sc[i, :n[i]])
