"""The measurement hook replays the joint kernel that the last chunk ran: its
byte count has that kernel's softmax partials (and, pruned, best labels)."""
import pytest

import synth
from tests.test_gpu_pred import _chunk, _decoder

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("form", ["stateful, few rows", "stateful, many rows", "streaming", "pruned"])
def test_joint_bytes(form):
    import paper_2609_14991_gb300 as tsd

    V, H, B, T, k = 1024, 320, 400 if form == "stateful, many rows" else 3, 2, 4
    w = synth.scaled(synth.WORKLOADS[0], V=V, H=H, B=B, T=T)
    lmA = synth.ngram_lm(w.lm_seed, V, 3, 30_000, w.zipf)
    E, W = synth.joint_weights(w)
    if form.startswith("stateful"):
        dec, lm, bo = _decoder(w, synth.pred_weights(w, D=64, Henc=H), lmA, None, E, W)
    else:
        dev = torch.device("cuda", 0)
        lm = tsd.NGram.from_arrays(lmA)
        dec = tsd.Decoder(V, H, torch.from_numpy(W.view("int16")).to(dev), torch.from_numpy(E.view("int16")).to(dev),
                          lm=lm, max_symbols=w.max_sym, max_streams=B, max_T=T, prune_k=k if form == "pruned" else 0)
    dec._slots = [dec.open() for _ in range(B)]
    dec.set_option("joint_bn", 64)
    if form == "stateful, few rows":
        dec.set_option("one_launch", 1)  # joint_bn turned it off
    _chunk(dec, w, synth.enc_chunk(w, range(B), 0))
    # partials per row: one per 64-label tile; few rows: one per unit of labels (16, of 68 and 64)
    partials = 16 if form == "stateful, few rows" else (V + 1 + 63) // 64
    operands = 2 * H * (B + V + 1)
    want = operands + 8 * B * partials * (1 + k) if form == "pruned" else operands + 4 * B * (V + 1) + 8 * B * partials
    assert dec.replay(1, 2, count_bytes=True) == want
    assert dec.replay(0, 2, count_bytes=True) > 0
    dec.check()
