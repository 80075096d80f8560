"""The tensor-core kernels' warps run their loops with all lanes and use
instructions of the whole warp (elect.sync, tcgen05 loads, shuffles), so a
lane whose wait gives up may not leave the others there.  Read from the sources:
it needs no GPU, and a lane left behind would hang one."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2608_01845_gb300", "csrc")
WARP = re.compile(r"\belect_one\(|__syncwarp\(|_sync\(|\bleads\(|\brejoin\(")


def _code(name):
    return re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())


def _blocks(code, head):
    """(start, end) of every block that `head` opens."""
    for m in re.finditer(head, code):
        depth, i = 1, m.end()
        while depth:
            depth += {"{": 1, "}": -1}.get(code[i], 0)
            i += 1
        yield m.end(), i


@pytest.mark.parametrize("name", ["gemm_tc.cu", "attn_tc.cu"])
def test_a_wait_that_gives_up_leaves_no_lane_behind(name):
    """A wait either votes (mbar_wait_warp), or is remembered by its lane, which
    stays in the loop, or is in a part that one lane runs by itself."""
    code = _code(name)
    alone = [(a, b) for a, b in _blocks(code, r"if \(elect_one\(\)\) \{") if not WARP.search(code[a:b])]
    waits = list(re.finditer(r"\bmbar_wait\(", code))
    assert waits and "mbar_wait_warp(" in code
    for m in waits:
        if any(a <= m.start() < b for a, b in alone):
            continue
        line = code[code.rindex("\n", 0, m.start()) + 1:code.index("\n", m.start())]
        assert re.search(r"\bok = (ok && )?mbar_wait\(", line), line
    # the loops with remembered waits have no early way out
    for a, b in _blocks(code, r"\bfor \([^{}]*\) \{"):
        if "ok = ok && mbar_wait(" in code[a:b] and "mbar_wait_warp(" not in code[a:b]:
            assert not re.search(r"\bbreak\b|\breturn (?!kOneLane)", code[a:b]), code[a:b]
            head = code[code.rindex("for (", 0, a):a]
            assert "ok" not in head, head


def test_the_warp_wait_votes():
    """Every return of the wait follows a vote, never one lane's own look."""
    body = re.search(r"bool mbar_wait_warp\([^{]*\{(.*?)\n\}", _code("ptx.cuh"), re.S).group(1)
    looks = re.findall(r"[^\n]*mbar_try_wait[^\n]*", body)
    assert looks and all("__all_sync(kAll, mbar_try_wait(" in x for x in looks)
    assert re.findall(r"[^\n]*return false[^\n]*", body) == ["        if (__any_sync(kAll, stop)) return false;"]


@pytest.mark.gpu
def test_a_whole_warps_wait_gives_up():
    """The self-test's warps, one released by the abort flag and one by its own
    limit, return with all their lanes and report the timeout only."""
    import torch

    from paper_2608_01845_gb300 import wdc
    ctx = wdc.Context(wdc.make_config(width=4096), 4)
    for limit_ns in (1000, 50_000, 2_000_000):
        ctx.selftest_wait_timeout(limit_ns)
        torch.cuda.synchronize()
        assert ctx.device_errors() == 1
    assert ctx.device_errors() == 0
