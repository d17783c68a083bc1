"""No lane's answer to a bounded wait decides where its warp goes, read from the kernels' source.

A bounded wait can run out, and the abort flag can be set, between two lanes' reads.  Where
warp-collective instructions follow (elect.sync, __syncwarp, the TMEM loads), the lanes of a warp must
still meet: a wait is a vote, or only one lane runs, or its answer is only accumulated in `ok`, which
then decides no branch, unless by a vote, but what the elected lane issues.
"""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2607_11185_gb300", "csrc")
VOTES = ("__all_sync(", "__any_sync(", "named_bar_and(")


def read(src):
    """(line, text) of the reads of a wait or the abort flag that neither a vote nor one lane takes nor
    `ok` accumulates, and of the branches on `ok` in blocks that accumulate."""
    src = re.sub(r"//[^\n]*", lambda m: " " * len(m.group()), src)
    blocks, lone, start = [], [], 0      # open blocks as [header, from, accumulates]; statement start
    branches = []
    for m in re.finditer(r"[{};]|\bmbar_wait\(|\baborted(?:_now)?\(", src):
        tok, stmt = m.group(), src[start:m.start()]
        if tok == "{":
            blocks.append([stmt, m.end(), False])
            start = m.end()
        elif tok == "}":
            head, at, acc = blocks.pop()
            if acc and re.search(r"\bwarp == 1\b", head):   # the whole role
                for b in re.finditer(r"\bbreak\b|\breturn(?: true| false)?;|; ok\b|\bif \(!?ok\b[^;]*;",
                                     src[at:m.start()]):
                    voted = src[:at + b.start()].endswith("if (!__all_sync(0xffffffffu, ok)) ")
                    if not voted and not re.match(r"if \(!ok\) (abort_now\(\)|on_timeout\(bars, status\));", b.group()):
                        branches.append((src[:at + b.start()].count("\n") + 1, b.group()))
            elif blocks:
                blocks[-1][2] |= acc
            start = m.end()
        elif tok == ";":
            start = m.end()
        elif not any(v in stmt for v in VOTES) and not any(re.search(r"\blane == 0", b[0]) for b in blocks):
            if re.search(r"\bok (= ok &&|&=) |\bbool ok = ", stmt):
                blocks[-1][2] = True
            elif "auto aborted_now =" not in stmt:
                lone.append((src[:m.start()].count("\n") + 1, (stmt + tok).strip()[-60:]))
    assert not blocks
    return lone, branches


@pytest.mark.parametrize("name,head", [("attn_fwd.cu", "__launch_bounds__(kThreads, 1)"),
                                       ("attn_bwd.cu", "__launch_bounds__(Bwd<D>::THREADS, 1)")])
def test_no_lane_decides_alone(name, head):
    with open(os.path.join(CSRC, name)) as f:
        src = f.read()
    src = src[src.index(head):]
    lone, branches = read(src[src.index("{"):src.index("\n}\n") + 2])
    assert lone == [] and branches == []


def test_the_reader_sees_lone_waits_and_branches():
    src = """{ if (warp == 1) { bool ok = mbar_wait(a, 0); for (int j = 0; ok && j < n; ++j) { if (!ok) break; }
      ok &= mbar_wait(e, 0); if (!__all_sync(0xffffffffu, ok)) break;
      if (lane == 0) { if (mbar_wait(b, 0)) x(); } ok = ok && mbar_wait(c, 0) && !aborted_now(); if (!ok) abort_now(); }
      if (warp == 5) { if (!mbar_wait(d, 0)) { } if (__any_sync(m, aborted_now())) { } if (aborted(bars)) { } } }"""
    lone, branches = read(src)
    assert [x[1] for x in lone] == ["if (!mbar_wait(", "if (aborted("]
    assert [x[1] for x in branches] == ["; ok", "if (!ok) break;"]
