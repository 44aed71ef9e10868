"""The joint kernel's 64-row tile (streaming epilogue, label tiles of 64, used
while every tile has an SM of its own): rows around its quadrants of 16 and
its tiles of 64, label counts around 64, more and fewer K blocks than operand
stages, and the first row count past the rule's line."""
import pytest

import synth
from tests import parity_util as pu

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("B,V,H", [(1, 63, 64), (15, 64, 128), (16, 62, 512), (17, 127, 576), (63, 128, 320),
                                   (64, 499, 640), (65, 1024, 1024), (130, 300, 704), (256, 1023, 1024),
                                   (500, 1024, 1024), (577, 1000, 1024), (96, 4000, 320)])
def test_logits(B, V, H):
    """Every label's captured logit against the double product of the same
    bf16 inputs, and the decisions taken from the stored ones."""
    w = synth.scaled(synth.WORKLOADS[0], B=B, V=V, H=H, T=3, lm_total=max(60, 20 * V), n_phr=12, phr_len=(1, 4))
    inp = pu.Inputs(w)
    run = pu.GpuRun(inp, range(B), 1, capture_steps=3, options={"one_launch": 0})
    models = pu.oracle_models(inp)
    rows = sorted({0, B // 3, B // 2, B - 1} | {i for i in (15, 16, 47, 48, 63, 64, 127, 128) if i < B})
    err, n = pu.captured_logit_error(run, models[2], 3, rows)
    assert n >= len(rows) and err < pu.LOGIT_TOL, (err, n)
    pu.assert_reports(pu.replay(inp, run, rows, models=models))
