"""Where a chunk runs in one launch and where the two-kernel step is faster
(both measured beside the rule in csrc/chunk_cluster.cu): on either side of
each of its lines, with the oracle's decisions."""
import pytest

import synth
from tests import parity_util as pu

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n,V,H,one", [(120, 1024, 640, True), (128, 1024, 640, False),   # one group; clusters of 16, three
                                       (70, 2048, 512, True), (112, 2048, 512, False),    # two passes, 10 and 16 rows
                                       (200, 639, 512, True), (200, 700, 512, False),     # a slice of one block, of two
                                       (200, 1024, 448, True), (160, 1500, 512, False),   # two blocks, H < 512
                                       (300, 512, 640, True), (300, 600, 640, False),     # three groups: bytes of W_out
                                       (300, 512, 704, False), (300, 300, 768, False)])
def test_both_sides(n, V, H, one):
    w = synth.scaled(synth.WORKLOADS[0], V=V, H=H, B=n, T=2, lm_total=20 * V, n_phr=12, phr_len=(1, 4))
    inp = pu.Inputs(w, lmA=synth.ngram_lm(7, V, 3, w.lm_total, 1.1), ph=synth.phrases(7, V, 12, 1, 4, 0.0))
    run = pu.GpuRun(inp, range(n), 1)
    assert run.dec.launches_per_chunk(n, w.T) == (1 if one else 2 * w.T * w.max_sym + 2)
    pu.assert_reports(pu.replay(inp, run, [0, n // 2, n - 1]))
