"""The stateful form's joint kernel for few rows gives the bits of the
stateless form's one launch: identity projection and a silent predictor, over
label slices around its blocks of 80 and its 16 CTAs, rows around 8 and 16 per
CTA, hidden sizes that leave warps without work."""
import numpy as np
import pytest

import synth
from tests.test_gpu_pred import _chunk, _decoder

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("V,H,B", [(15, 64, 1), (127, 192, 8), (499, 320, 9), (1023, 1024, 17), (1100, 640, 33),
                                   (1279, 512, 64), (2100, 320, 5), (1024, 1024, 112), (512, 640, 200)])
def test_bits_of_the_stateless_form(V, H, B):
    import paper_2609_14991_gb300 as tsd

    w = synth.scaled(synth.WORKLOADS[0], V=V, H=H, B=B, T=4)
    p = synth.pred_weights(w, D=64, Henc=H)
    p.We = np.eye(H, dtype=np.float32).view(np.uint32).__rshift__(16).astype(np.uint16)
    p.be = np.zeros(H, dtype=np.float32)
    p.Wp = np.zeros_like(p.Wp)
    p.bp = np.zeros(H, dtype=np.float32)
    lmA = synth.ngram_lm(w.lm_seed, V, 4, max(60, 20 * V), w.zipf)
    ph = synth.phrases(w.boost_seed, V, 20, 1, 4, 0.3)
    E, W = synth.joint_weights(w)
    dec, _, _ = _decoder(w, p, lmA, ph, E, W)
    dec._slots = [dec.open() for _ in range(B)]
    dev = torch.device("cuda", 0)
    plain = tsd.Decoder(V, H, torch.from_numpy(W.view(np.int16)).to(dev), torch.zeros((w.N, H), dtype=torch.int16, device=dev),
                        lm=tsd.NGram.from_arrays(lmA), boost=tsd.Boost.from_phrases(V, ph, w.bonus), max_symbols=w.max_sym,
                        max_streams=B, max_T=w.T)
    plain._slots = [plain.open() for _ in range(B)]
    assert plain.launches_per_chunk(B, w.T) == 1
    for c in range(2):
        enc = synth.enc_chunk(w, range(B), c)
        for x, y in zip(_chunk(dec, w, enc), _chunk(plain, w, enc)):
            for u, v in zip(x, y):
                assert np.array_equal(u, v)
    for a, b in zip(dec._slots, plain._slots):
        assert dec.state(a) == plain.state(b)
