"""Every arrival of the tensor core on a barrier of the FP64 convolution kernel is waited for
before its block ends (CPU model): an asynchronous arrival after the end would write into
shared memory that the next block on the SM already uses.  The issuing warp's loops are
restated; the condition under which it commits to `done`, and the turns whose readers wait for
it, are read from the kernel source."""
import os
import re

import pytest

SRC = os.path.join(os.path.dirname(__file__), "..", "paper_1204_5434_gb300", "csrc", "pft_tc64.cuh")
NS = 6


def _config(n):
    cw = n if n <= 96 else 64
    return n // cw, 4 if n <= 64 else 2  # chunks, accumulators


def _done_condition(src):
    m = re.search(r"if \(([^\n]*)\) tc_commit\(done\);", src)
    assert m
    return m.group(1).replace("&&", "and")


@pytest.mark.parametrize("n", [16, 32, 48, 64, 96, 128])
@pytest.mark.parametrize("more", [False, True])
def test_every_commit_is_waited_for(n, more):
    with open(SRC) as f:
        src = f.read()
    nch, nb = _config(n)
    nj = nch * NS
    turns = 2 if more else 1
    full = [[0] * nb for _ in range(nch)]
    done = 0
    cond = _done_condition(src)
    for turn in range(turns):
        for ch in range(nch):
            for lev in range(NS):
                t = ch * NS + lev
                full[ch][t % nb] += 1
                done += bool(eval(cond, {}, {"t": t, "NJ": nj, "turn": turn, "more": more}))
    # a chunk's readers wait for each of its levels at every turn
    for ch in range(nch):
        for b in range(nb):
            waits = turns * sum(1 for lev in range(NS) if lev % nb == b)
            assert full[ch][b] == waits, (ch, b)
    # `done` is waited for where a later turn overwrites X
    assert re.search(r"if \(turn\) \{[^\n]*\n\s*mbar_wait\(done, 0, err, 1\);", src)
    assert done == turns - 1
