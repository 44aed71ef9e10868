"""The per-step GEMMs of the stateful form in their 64-row tiles (while every
tile has an SM of its own) against the 128-row ones a larger batch takes: the
same streams give the same bits, for widths that fill the last LSTM tile of 80
columns and that leave it partial, and rows around the tiles' edges."""
import numpy as np
import pytest

import synth
from tests.test_gpu_pred import _chunk, _decoder

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("D,H,large,small", [(640, 1024, 300, (1, 17, 64, 65, 256)), (192, 320, 1000, (3, 63, 129, 960))])
def test_small_and_large_batches_agree(D, H, large, small):
    w = synth.scaled(synth.WORKLOADS[0], V=200, H=H, B=large, T=2, n_phr=20, phr_len=(2, 5))
    p = synth.pred_weights(w, D=D, Henc=H)
    lmA = synth.ngram_lm(w.lm_seed, w.V, 3, 6000, w.zipf)
    ph = synth.phrases(w.boost_seed, w.V, w.n_phr, 2, 5, 0.2)
    E, W = synth.joint_weights(w)
    enc = [synth.enc_chunk_wide(w, range(large), c, H) for c in range(2)]

    def decode(n):
        dec, _, _ = _decoder(synth.scaled(w, B=n), p, lmA, ph, E, W)
        dec.set_option("joint_bn", 64)
        dec._slots = [dec.open() for _ in range(n)]
        return [_chunk(dec, w, e[:n]) for e in enc], [dec.pred_state(s) for s in dec._slots]

    ref, state = decode(large)
    for n in small:
        got, st = decode(n)
        for c in range(2):
            for i in range(n):
                for a, b in zip(got[c][i], ref[c][i]):
                    assert np.array_equal(a, b), (n, c, i)
        for i in range(n):
            assert all(np.array_equal(a, b) for a, b in zip(st[i], state[i])), (n, i)
