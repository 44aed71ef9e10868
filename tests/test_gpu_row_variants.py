"""The streaming row pass with few rows (eight warps per row, up to two or
three rows per SM) and with many (four warps) take the same decisions bit for bit, where
the two could differ: more chain elements than warps, chains at their
capacities, trie nodes with more children than a warp holds, hidden sizes past
one 16-byte piece per thread, no tables."""
import numpy as np
import pytest

import synth
from tests import parity_util as pu

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _inputs(case):
    w = synth.scaled(synth.WORKLOADS[0], B=320, V=300, H=128, T=4, lm_total=6000, n_phr=40, phr_len=(1, 5))
    if case == "long chains":
        w = synth.scaled(w, V=8, H=64, T=12, lm_order=16, lm_total=60000, beta=4.0)
        return pu.Inputs(w, lmA=synth.ngram_lm(w.lm_seed, 8, 16, 60000, 1.05), ph=synth.phrases(5, 8, 12, 16, 32, 0.0))
    if case == "wide nodes":
        w = synth.scaled(w, V=600, lm_total=280_000, beta=3.0)
        return pu.Inputs(w, lmA=synth.ngram_lm(9, 600, 5, 280_000, 1.02), ph=synth.phrases(9, 600, 30000, 2, 4, 0.9))
    if case == "hidden sizes":
        return pu.Inputs(synth.scaled(w, V=70, H=2112, T=2))
    if case == "wide labels":  # past three rows per SM: the joint kernel's 64-row tiles do not apply
        return pu.Inputs(synth.scaled(w, V=2100, B=460, T=2, lm_total=20000))
    if case == "no tables":
        return pu.Inputs(w, with_lm=False, with_boost=False)
    return pu.Inputs(w)


@pytest.mark.parametrize("case", ["plain", "long chains", "wide nodes", "hidden sizes", "wide labels", "no tables"])
def test_few_and_many_rows_agree(case):
    inp = _inputs(case)
    off = {"one_launch": 0, "joint_bn": 64}
    many = pu.GpuRun(inp, range(inp.w.B), 2, options=off)  # past the line
    few = pu.GpuRun(inp, range(5), 2, options=off)
    for c in range(2):
        for s in range(5):
            assert many.states[c][s] == few.states[c][s]
            for a, b in zip(many.emitted(s, c), few.emitted(s, c)):
                assert np.array_equal(a, b), (c, s)
    pu.assert_reports(pu.replay(inp, few, range(5)))
