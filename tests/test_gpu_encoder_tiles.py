"""The encoder's GEMM tile shapes (CTA pairs of 256 x 256, 128 x 128 / 64 /
32, and 64 staged rows for small calls) at their edges: every stream's output
is bit-identical to the same stream encoded alone (another tile shape), and
one stream is checked against the oracle."""
import numpy as np
import pytest

import synth
from oracle import encoder as oe

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _run(w, cfg, n, C, chunks, streams=None):
    import paper_2609_14991_gb300 as tsd

    streams = list(range(n)) if streams is None else streams
    enc = tsd.Encoder(w, max_streams=len(streams), max_chunk=C)
    slots = [enc.open() for _ in streams]
    out = []
    for c in range(chunks):
        f = torch.from_numpy(synth.features(cfg, streams, c * C, C).view(np.int16)).cuda()
        out.append(enc.encode_chunk(slots, f).cpu().numpy())
    enc.check()
    return out


# (d, heads, ff, kernel) x (streams, frames): rows at and around the 32-row
# slabs, 64 staged rows, the 128-row tile, the 256-row pair tile
@pytest.mark.parametrize("d,heads,ff,kernel", [(256, 4, 512, 9), (384, 6, 640, 9), (640, 5, 2560, 7)])
@pytest.mark.parametrize("n,C", [(1, 1), (2, 16), (3, 11), (4, 16), (5, 13), (8, 16), (12, 11), (20, 13), (37, 7)])
def test_small_calls(d, heads, ff, kernel, n, C):
    cfg = synth.EncoderCfg("t", d=d, layers=1, heads=heads, ff=ff, kernel=kernel, left=12, chunk=C, feat=16, stack=4)
    w = synth.encoder_weights(cfg)
    many = _run(w, cfg, n, C, 2)
    for s in sorted({0, n // 2, n - 1}):
        alone = _run(w, cfg, 1, C, 2, [s])
        for c in range(2):
            assert np.array_equal(many[c][s], alone[c][0]), (s, c)
    E, st = oe.Encoder(w), oe.EncoderStream(cfg)
    for c in range(2):
        want = oe.bits_to_f64(oe.encode_chunk(E, st, synth.features(cfg, [n - 1], c * C, C)[0]))
        err = np.abs(oe.bits_to_f64(many[c][n - 1].view(np.uint16)) - want)
        # a block's roundings to bf16 land on either side of a boundary: a few flips of one output ulp (2^-7)
        assert err.mean() <= 0.0095 and err.max() <= 0.033, (err.mean(), err.max())


@pytest.mark.parametrize("n,C", [(79, 13), (128, 8), (100, 13), (257, 13)])
def test_pair_tiles(n, C):
    """Calls large enough for the CTA pairs, whole and partial last tiles."""
    cfg = synth.EncoderCfg("t", d=1024, layers=1, heads=8, ff=4096, left=12, chunk=C, feat=80, stack=8)
    w = synth.encoder_weights(cfg)
    many = _run(w, cfg, n, C, 1)
    for s in (0, 19, n - 1):
        assert np.array_equal(many[0][s], _run(w, cfg, 1, C, 1, [s])[0][0]), s


def test_branches_only_while_a_gemm_leaves_most_sms_idle():
    import paper_2609_14991_gb300 as tsd

    for d, heads, ff, n, branches in ((256, 4, 512, 100, 2), (512, 8, 2048, 60, 1), (256, 4, 1024, 256, 1)):
        cfg = synth.EncoderCfg("t", d=d, layers=1, heads=heads, ff=ff, left=12, chunk=13, feat=16, stack=4)
        enc = tsd.Encoder(synth.encoder_weights(cfg), max_streams=n)
        assert enc.launches_per_chunk(n, 13) == branches * 16 + 1
