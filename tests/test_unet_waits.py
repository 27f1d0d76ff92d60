"""The bounded waits of the tcgen05 kernels end the same way for every thread that acts on them
together (a check of the source: the moment at which a wait runs out cannot be set up). Each thread
decides by itself whether its wait ran out, so a result that a warp branches on is voted on by the
warp, and one that a group with a barrier of its own leaves a loop on by the group."""
import os
import re

HERE = os.path.dirname(os.path.abspath(__file__))
SRC = os.path.join(os.path.dirname(HERE), "paper_2003_11069_gb300", "csrc", "unet_conv.cuh")


def _code():
    txt = open(SRC).read()
    return re.sub(r"//[^\n]*", lambda m: " " * len(m.group()), txt)


def _block(code, at):
    """The braces' content that opens at or after `at`."""
    i = code.index("{", at)
    depth = 0
    for j in range(i, len(code)):
        depth += {"{": 1, "}": -1}.get(code[j], 0)
        if depth == 0:
            return i, j
    raise AssertionError("unbalanced braces")


def test_waits_of_whole_warps_are_votes():
    code = _code()
    single = [_block(code, m.start()) for m in re.finditer(r"if \(lane == 0\) \{", code)]  # the copying lane
    count = 0
    for m in re.finditer(r"lbnci::mbar_wait\(", code):
        count += 1
        if any(a < m.start() < b for a, b in single):
            continue
        # the statement that holds the wait, and the one after it: a vote of the warp
        start = max(code.rfind(c, 0, m.start()) for c in ";{}")
        end = code.index(";", code.index(";", m.start()) + 1)
        if re.search(r"__(any|all)_sync\(~0u", code[start:end]):
            continue
        # or the group's reduction, with nothing on the way that lanes could leave by or meet at
        until = code[m.start():code.index("bar_all(", m.start())]
        assert not re.search(r"\b(break|continue|return|while)\b|__syncwarp|bar\.sync|&& ok", until), until
    assert count >= 10


def test_drain_groups_leave_their_loop_together():
    """Every path of the row strips' drain loop that may end it has reduced `ok` over the group of
    128 threads whose barriers (bar_all, bar.sync) the next row uses."""
    code = _code()
    at = code.index("for (int q = 0; q < nq && ok; ++q) {")
    a, b = _block(code, at)
    body = code[a:b]
    waits = [m.start() for m in re.finditer(r"ok = (?:warp|lbnci::mbar)_wait\(done", body)]
    assert len(waits) == 2
    for w in waits:
        vote = body.index("ok = bar_all(1 + g, 128, ok)", w)
        leave = body.find("continue", w)
        assert leave < 0 or vote < leave
