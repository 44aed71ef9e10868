"""The chunk in one launch (option "one_launch", the default where a cluster's
shared memory holds W_out) against the two-kernel step and the oracle, where
its tilings can go wrong: label slices around multiples of 8 and 80 labels,
row counts around 8 and 16 and around one wave of clusters, hidden sizes that
leave warps without work, chains with many arcs, empty tables."""
import numpy as np
import pytest

import synth
from tests import parity_util as pu

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

BASE = synth.scaled(synth.WORKLOADS[0], T=6, lm_total=6000, n_phr=40, phr_len=(1, 5))


def _runs(inp, streams, chunks=2, **kw):
    one = pu.GpuRun(inp, streams, chunks, **kw)
    two = pu.GpuRun(inp, streams, chunks, options={"one_launch": 0}, **kw)
    assert one.dec.launches_per_chunk(len(one.streams), one.T) == 1
    assert two.dec.launches_per_chunk(len(one.streams), one.T) == 2 * one.T * inp.w.max_sym + 2
    return one, two


def _agree(one, two):
    """Both forms take the same decisions; their sums differ in order only
    (scores: |logit| <= ~15 and a log-sum-exp, a few fp32 ulps each)."""
    for c in range(len(one.chunks)):
        assert one.states[c] == two.states[c]
        for i in range(len(one.streams)):
            a, b = one.emitted(i, c), two.emitted(i, c)
            assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1]), (c, i)
            np.testing.assert_allclose(a[2], b[2], atol=2e-5)


@pytest.mark.parametrize("V,H", [(15, 64), (63, 64), (64, 128), (127, 320), (255, 192), (499, 320), (1023, 1024),
                                 (1024, 1024), (1100, 640), (1279, 512), (2100, 320)])
def test_label_slices(V, H):
    w = synth.scaled(BASE, V=V, H=H, B=3, lm_total=max(60, 20 * V))
    inp = pu.Inputs(w, lmA=synth.ngram_lm(7, V, 3, w.lm_total, 1.1), ph=synth.phrases(7, V, 12, 1, 4, 0.0))
    one, two = _runs(inp, range(w.B))
    _agree(one, two)
    pu.assert_reports(pu.replay(inp, one, range(w.B)))


@pytest.mark.parametrize("B", [1, 7, 8, 9, 17, 64, 111, 113, 200, 336])
def test_row_counts(B):
    w = synth.scaled(BASE, V=512, H=640, B=B, T=3, lm_total=20000)
    inp = pu.Inputs(w)
    one, two = _runs(inp, range(B))
    _agree(one, two)
    pu.assert_reports(pu.replay(inp, one, sorted({0, B // 2, B - 1})))


def test_two_passes_of_the_product():
    """More than eight rows per cluster with a slice of W_out that leaves room for eight."""
    w = synth.scaled(BASE, V=2100, H=512, B=70, T=2, lm_total=40000)
    inp = pu.Inputs(w)
    one, two = _runs(inp, range(w.B))
    _agree(one, two)
    pu.assert_reports(pu.replay(inp, one, [0, 34, 69]))


@pytest.mark.parametrize("case", ["no tables", "unigram lm", "no boost", "no lm", "zero weights", "long chains",
                                  "wide contexts"])
def test_tables(case):
    w = synth.scaled(BASE, B=3)
    if case == "no tables":
        inp = pu.Inputs(w, with_lm=False, with_boost=False)
    elif case == "unigram lm":
        inp = pu.Inputs(w, lmA=synth.ngram_lm(3, w.V, 1, w.V, 1.1))
    elif case == "no boost":
        inp = pu.Inputs(w, with_boost=False)
    elif case == "no lm":
        inp = pu.Inputs(w, with_lm=False)
    elif case == "zero weights":
        inp = pu.Inputs(synth.scaled(w, lam=0.0, beta=0.0))
    elif case == "long chains":  # LM and trie chains up to their capacities
        w = synth.scaled(w, V=8, H=64, T=40, lm_order=16, lm_total=60000, beta=4.0)
        inp = pu.Inputs(w, lmA=synth.ngram_lm(w.lm_seed, 8, 16, 60000, 1.05), ph=synth.phrases(5, 8, 12, 16, 32, 0.0))
    else:  # more arcs and trie children than a group's threads hold at once, trie chains longer than they hold
        w = synth.scaled(w, V=40, lm_total=280_000, beta=3.0)
        inp = pu.Inputs(w, lmA=synth.ngram_lm(9, 40, 8, 280_000, 1.02), ph=synth.phrases(9, 40, 20000, 4, 9, 0.2))
    one, two = _runs(inp, range(w.B))
    _agree(one, two)
    pu.assert_reports(pu.replay(inp, one, range(w.B)))


@pytest.mark.parametrize("V,H", [(15, 64), (255, 320), (511, 320), (639, 640), (700, 448), (1023, 640), (1300, 512),
                                 (600, 832), (500, 1024), (300, 192)])
def test_results_do_not_depend_on_the_other_rows(V, H):
    """The same bits alone and in calls whose rows take clusters of 8 and of
    16, one to three row groups and one or two passes of the product."""
    w = synth.scaled(BASE, V=V, H=H, T=2, lm_total=max(60, 20 * V))
    inp = pu.Inputs(w, lmA=synth.ngram_lm(7, V, 3, w.lm_total, 1.1), ph=synth.phrases(7, V, 12, 1, 4, 0.0))
    watch = (0, 5)
    alone = [pu.GpuRun(inp, [s], 2) for s in watch]
    used = 1
    for n in (6, 16, 33, 64, 100, 113, 128, 160, 200, 260, 336):
        run = pu.GpuRun(inp, range(n), 2)
        if run.dec.launches_per_chunk(n, w.T) != 1:
            continue  # (the two-kernel step, whose sums have another order)
        used += 1
        for s, a in zip(watch, alone):
            for c in range(2):
                for x, y in zip(a.emitted(0, c), run.emitted(s, c)):
                    assert np.array_equal(x, y), (n, s, c)
    assert used >= 4


def test_shapes_that_do_not_fit_take_the_two_kernel_step():
    """W_out larger than a cluster's shared memory, more rows than one wave, a hidden size past the warps' pieces."""
    for kw in (dict(V=4096, H=1024, B=2), dict(V=512, H=640, B=400), dict(V=64, H=1088, B=2)):
        w = synth.scaled(BASE, T=1, **kw)
        run = pu.GpuRun(pu.Inputs(w, with_lm=False, with_boost=False), range(w.B), 1)
        assert run.dec.launches_per_chunk(w.B, 1) == 2 * w.max_sym + 2
        pu.assert_reports(pu.replay(pu.Inputs(w, with_lm=False, with_boost=False), run, [0, w.B - 1]))
