"""The softmax partials of the one-launch decode (csrc/chunk_partials.h) under
every order in which a cluster's messages may arrive: a row's owner reads each
step's partials, all of them and no others.  An exhaustive search over a
model of one row: CTA 0 owns it, every CTA sends its logits and then its
partial of a step, any message in flight may land next, and a barrier's phase
completes when its arrival and as many partials as announced have been counted."""
import ctypes
import os
import subprocess

import pytest

from paper_2609_14991_gb300 import _build


@pytest.fixture(scope="module")
def header(tmp_path_factory):
    """(barrier, parity, buffer) of a step, as the kernel takes them, and the two counts."""
    d = tmp_path_factory.mktemp("partials")
    (d / "p.cpp").write_text('#include "chunk_partials.h"\n' + "".join(
        f'extern "C" int {f}(int s) {{ return tsd::part_{f}(s); }}\n' for f in ("bar", "parity", "buf")) +
        'extern "C" int bars() { return tsd::kPartBars; }\nextern "C" int bufs() { return tsd::kPartBufs; }\n')
    subprocess.run([os.environ.get("CXX", "g++"), "-std=c++17", "-shared", "-fPIC", "-I", _build.CSRC, "-o", str(d / "p.so"),
                    str(d / "p.cpp")], check=True)
    lib = ctypes.CDLL(str(d / "p.so"))
    return lib.bar, lib.parity, lib.buf, lib.bars(), lib.bufs()


def _search(scheme, n_cta, steps):
    """The first fault over all orders, or None."""
    bar_of, parity_of, buf_of, bars, bufs = scheme
    # a CTA's program per step; the owner also waits for the partials of the step before, announces this step's
    # and writes the score of the step before
    owner = ["label", "wait", "arm", "logits", "partial", "score"]
    other = ["label", "logits", "partial"]
    # state: per CTA (step, place), labels each CTA has, row's step, its logits in, barriers, buffers, messages
    start = (((0, 0),) * n_cta, (0,) * n_cta, 0, frozenset(), ((0, 1, 0),) * bars, ((-1,) * n_cta,) * bufs, frozenset())
    seen, todo = {start}, [start]
    while todo:
        pcs, labels, row, have, bar, buf, msgs = todo.pop()
        nxt = []

        def count(bs, i, arrive, tx):  # an arrival that announces tx partials, or one partial that landed (tx = -1)
            phase, pending, left = bs[i]
            pending, left = pending - arrive, left + tx
            if pending == 0 and left == 0:
                phase, pending, left = phase + 1, 1, 0
            return bs[:i] + ((phase, pending, left),) + bs[i + 1:]

        for c in range(n_cta):
            step, at = pcs[c]
            prog = owner if c == 0 else other
            op = prog[at]
            if op == "label" and labels[c] < step:
                continue
            if step == steps and c != 0:
                continue  # the row has finished
            b2, m2 = bar, msgs
            if op == "wait" and step > 0 and (bar[bar_of(step - 1)][0] & 1) == parity_of(step - 1):
                continue
            if op == "score" and step > 0 and any(x != step - 1 for x in buf[buf_of(step - 1)]):
                return f"step {step - 1}: the owner reads the partials of steps {buf[buf_of(step - 1)]}"
            if step == steps and op in ("arm", "logits", "partial"):
                pass
            elif op == "arm":
                b2 = count(bar, bar_of(step), 1, n_cta)
            elif op in ("logits", "partial"):
                m2 = msgs | {(op, c, step)}
            if step == steps and op == "score":
                continue  # the end
            pc = (step, at + 1) if at + 1 < len(prog) else (step + 1, 0)
            nxt.append((pcs[:c] + (pc,) + pcs[c + 1:], labels, row, have, b2, buf, m2))
        for m in msgs:  # any message lands
            kind, c, step = m
            rest = msgs - {m}
            if kind == "label":
                nxt.append((pcs, labels[:c] + (step,) + labels[c + 1:], row, have, bar, buf, rest))
            elif kind == "logits":
                h2, r2 = have | {c}, row
                if len(h2) == n_cta:  # the row's label of the next step, to every CTA
                    h2, r2 = frozenset(), row + 1
                    rest = rest | {("label", x, r2) for x in range(n_cta)}
                nxt.append((pcs, labels, r2, h2, bar, buf, rest))
            else:
                k = buf_of(step)
                f2 = buf[:k] + (buf[k][:c] + (step,) + buf[k][c + 1:],) + buf[k + 1:]
                nxt.append((pcs, labels, row, have, count(bar, bar_of(step), 0, -1), f2, rest))
        if not nxt and pcs[0] != (steps, owner.index("score")):
            return f"nothing can move: {pcs}"
        for s in nxt:
            if s not in seen:
                seen.add(s)
                todo.append(s)
    return None


@pytest.mark.parametrize("n_cta,steps", [(2, 9), (3, 7)])
def test_every_order_of_arrival(header, n_cta, steps):
    assert _search(header, n_cta, steps) is None


def test_the_search_finds_what_one_barrier_or_two_buffers_miss(header):
    bar, parity, buf, bars, bufs = header
    assert "reads the partials" in _search((lambda s: 0, lambda s: s & 1, buf, 1, bufs), 2, 7)
    assert _search((bar, parity, lambda s: s % 2, bars, 2), 2, 7) is not None
