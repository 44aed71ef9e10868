"""The row pass with several LMs (and with one LM of a weight other than 1)
at the sizes where it can go wrong: vocabularies around its threads and quads,
chains and trie nodes past what its threads hold, more chain elements than
warps, hidden sizes past one piece per thread, the CUDA-core joint, saved
state."""
import numpy as np
import pytest

import oracle
import synth
import paper_2609_14991_gb300 as tsd
from tests import parity_util as pu

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _check(w, arrays, weights, ph, chunks=2, joint_kind=0, move=False):
    E, W = synth.joint_weights(w)
    dev = torch.device("cuda", 0)
    gl = [tsd.NGram.from_arrays(a) for a in arrays]
    bo = tsd.Boost.from_phrases(w.V, ph, w.bonus) if ph else None
    on = lambda x: torch.from_numpy(x.view(np.int16)).to(dev)
    make = lambda: tsd.Decoder(w.V, w.H, on(W), on(E), lms=list(zip(gl, weights)), boost=bo, max_symbols=w.max_sym,
                               max_streams=w.B, max_T=w.T)
    dec = make()
    if joint_kind:
        dec.set_joint_kernel(joint_kind)
    slots = [dec.open() for _ in range(w.B)]
    olms = [(oracle.LM.from_arrays(a), wt) for a, wt in zip(arrays, weights)]
    obo = oracle.Boost.from_phrases(w.V, ph, w.bonus) if ph else None
    model = oracle.Model(w.V, w.H, E, W)
    rows = sorted({0, w.B // 2, w.B - 1})
    streams = {i: oracle.Stream(w.V) for i in rows}
    for c in range(chunks):
        enc = synth.enc_chunk(w, range(w.B), c)
        out = dec.decode_chunk(slots, on(enc), w.lam, w.beta)
        torch.cuda.synchronize()
        toks, frames, scores, counts = (x.cpu().numpy() for x in (out.tokens, out.frames, out.scores, out.counts))
        for i in rows:
            n = int(counts[i])
            _, _, _, rep = oracle.decode_chunk(streams[i], model, olms, obo, enc[i], w.lam, w.beta, w.max_sym,
                                               follow=(toks[i, :n], frames[i, :n], scores[i, :n]))
            assert rep[oracle.REP_INCONSISTENT] == 0 and rep[oracle.REP_MISMATCH] == 0, rep
            assert rep[oracle.REP_MAX_SCORE_DIFF] <= pu.SCORE_TOL, rep
            for m, g in enumerate(gl):
                assert g.state_tuple(dec.lm_state(slots[i], m)) == olms[m][0].state(streams[i].history()), (c, i, m)
        if move:  # every stream goes on in a new decoder from its saved state
            blobs = [dec.export_state(s) for s in slots]
            dec = make()
            slots = [dec.open() for _ in blobs]
            for s, b in zip(slots, blobs):
                dec.import_state(s, b)


BASE = synth.scaled(synth.WORKLOADS[0], B=3, T=5, H=128, beta=1.5)


@pytest.mark.parametrize("V,H,B", [(5, 64, 1), (255, 128, 3), (1023, 2112, 2), (1025, 64, 3), (4100, 64, 2), (300, 64, 320)])
@pytest.mark.parametrize("n_lm", [2, 3, 4])
def test_sizes(V, H, B, n_lm):
    w = synth.scaled(BASE, V=V, H=H, B=B)
    arrays = [synth.ngram_lm(11 + i, V, 2 + i % 3, max(30, (8 - i) * V), 1.1) for i in range(n_lm)]
    _check(w, arrays, [1.0, 0.5, 0.25, -0.2][:n_lm], synth.phrases(5, V, 12, 1, 4, 0.0))


def test_long_chains():
    w = synth.scaled(BASE, V=8, H=64, T=12, beta=4.0)
    arrays = [synth.ngram_lm(3 + i, 8, 16, 60000, 1.05) for i in range(4)]
    _check(w, arrays, [1.0, 0.5, 0.5, 0.25], synth.phrases(5, 8, 12, 16, 32, 0.0))


@pytest.mark.parametrize("move", [False, True])
def test_wide_nodes_and_saved_state(move):
    w = synth.scaled(BASE, V=600, beta=3.0)
    arrays = [synth.ngram_lm(9, 600, 5, 200_000, 1.02), synth.ngram_lm(10, 600, 3, 90_000, 1.02)]
    _check(w, arrays, [1.0, 0.5], synth.phrases(9, 600, 30000, 2, 4, 0.9), move=move)


@pytest.mark.parametrize("case", ["one weighted", "no trie", "unigram and bigram", "cuda cores"])
def test_forms(case):
    w = synth.scaled(BASE, V=300)
    a = synth.ngram_lm(3, 300, 3, 6000, 1.1)
    ph = synth.phrases(5, 300, 20, 2, 4, 0.1)
    if case == "one weighted":
        _check(w, [a], [0.5], ph)
    elif case == "no trie":
        _check(w, [a, synth.ngram_lm(4, 300, 2, 3000, 1.1)], [1.0, 0.5], None)
    elif case == "unigram and bigram":
        _check(w, [synth.ngram_lm(4, 300, 1, 300, 1.1), synth.ngram_lm(5, 300, 2, 3000, 1.1)], [1.0, 0.5], ph)
    else:
        _check(w, [a, synth.ngram_lm(4, 300, 2, 3000, 1.1)], [1.0, 0.5], ph, joint_kind=1)
