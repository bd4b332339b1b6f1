"""Rules of the device code that no run can show, read off its source."""
import os
import re

from paper_1808_03801_gb300 import build


def _code(name):
    with open(os.path.join(build.CSRC, name)) as f:
        return re.sub(r"//[^\n]*|/\*.*?\*/", "", f.read(), flags=re.S)


def test_a_bounded_wait_is_decided_by_the_whole_warp():
    """A copy that lands at the limit of a wait is seen by some lanes and not
    by others.  The warp goes on to full-mask collectives, so a wait whose
    outcome is used takes a vote."""
    code = _code("usp_fused.cu")
    body = code[code.index("k_g2(const SimDev"):]
    used = re.findall(r"=\s*(__all_sync\(0xffffffffu,\s*)?mbar_wait\(", body)
    assert used and all(used)


def test_launchers_keep_no_state_that_threads_write():
    """Handles are stepped from several threads: what a launcher finds out
    once is initialised as a constant, which the language does under a lock."""
    for name in os.listdir(build.CSRC):
        code = _code(name)
        assert not re.findall(r"\bstatic\s+(?:int|bool|unsigned|uint32_t|size_t|float|double)\s+\w+\s*(?:=|;|\[)", code), name
