"""A bounded wait that runs out ends a loop for all threads that meet in that loop's barriers, or for none.  A thread that left on
its own would meet the others in different barriers, which cannot be provoked on a GPU (the waits only run out when something
else is broken): the shape of the code is checked instead."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1806_04090_b200", "csrc")


def _source(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def test_tridiagonal_reduction_gives_up_as_a_block():
    src = _source("atomo_tridiag.cu")
    calls = [m for m in re.finditer(r"\btri_wait\(", src) if "bool tri_wait" not in src[max(0, m.start() - 40):m.end()]]
    assert len(calls) == 1
    after = src[calls[0].start():]
    # what the block decides on is shared memory that the wait's own statement sets ...
    flag = re.match(r"[^;]*\)\s*(\w+)\s*=\s*1u\s*;", after).group(1)
    assert re.search(r"__shared__\s+uint32_t\s+%s\b" % flag, src)
    # ... read after the block has met, and nobody leaves before that
    read = re.search(r"const bool (\w+) = %s != 0u;" % flag, after)
    assert after.index("__syncthreads()") < read.start()
    assert "break" not in after[:read.start()] and "return" not in after[:read.start()]
    assert re.search(r"if \(%s\) \{[^}]*break;" % read.group(1), after[read.start():])


def test_gram_drain_gives_up_as_a_group():
    src = _source("atomo_tc.cu")
    drain = src[src.index("tfull_bar(buf), (uint32_t)(kb >> 1) & 1u"):]
    # a warp decides as one (the TMEM loads are warp-wide) ...
    assert "__all_sync(0xffffffffu, tc_mbar_wait(tfull_bar" in src
    # ... and the four warps meet before the abort word says what they do next
    group = drain.index('"bar.sync 2, 128;"')
    decide = drain.index("ok = *s_abort == 0u;")
    assert group < decide < drain.index("bool write_tile = ok;")
