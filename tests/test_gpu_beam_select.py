"""Beam selection (each hypothesis' top K by its own CTA, the block-wide
ranking, the merges by one warp) over beam widths and vocabularies around its
tilings, checked candidate by candidate against the oracle."""
import pytest

import synth
from tests import parity_util as pu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K", [2, 3, 5, 6, 7, 8])
@pytest.mark.parametrize("V", [7, 255, 1100])
def test_beam_widths(K, V):
    w = synth.scaled(synth.WORKLOADS[0], V=V, H=64, B=3, T=5, beam=K, max_sym=1, lm_total=max(40, 4 * V))
    inp = pu.Inputs(w, lmA=synth.ngram_lm(7, V, 3, w.lm_total, 1.1), ph=synth.phrases(7, V, 6, 1, 3, 0.0))
    run = pu.GpuRun(inp, range(w.B), 3, capture_steps=w.T)
    pu.assert_reports(pu.replay_beam(inp, run, range(w.B)))


@pytest.mark.parametrize("K,S", [(3, 2), (8, 3)])
def test_several_labels_per_frame(K, S):
    w = synth.scaled(synth.WORKLOADS[0], V=40, H=64, B=3, T=6, beam=K, max_sym=S, lm_total=400)
    inp = pu.Inputs(w, lmA=synth.ngram_lm(7, 40, 3, 400, 1.1), ph=synth.phrases(7, 40, 6, 1, 3, 0.0))
    run = pu.GpuRun(inp, range(w.B), 3, capture_steps=w.T * S)
    pu.assert_reports(pu.replay_beam(inp, run, range(w.B)))


def test_beam_with_the_cuda_core_joint():
    """The CUDA-core joint kernel feeds the same selection."""
    w = synth.scaled(synth.WORKLOADS[0], V=255, H=64, B=3, T=5, beam=4, max_sym=1, lm_total=2000)
    inp = pu.Inputs(w)
    run = pu.GpuRun(inp, range(w.B), 2, capture_steps=w.T, joint_kind=1)
    pu.assert_reports(pu.replay_beam(inp, run, range(w.B)))
