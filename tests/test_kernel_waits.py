"""Every wait of the projection kernel between its first tile and its last ends by itself: a
time-out of one warp must not leave another in a barrier that never fills.  Read from the source,
since a run that times out is never provoked."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1805_08995_gb300", "csrc")


def _body(text, head):
    """The braces that follow `head`, without comments."""
    text = re.sub(r"//[^\n]*", "", text)
    i = text.index("{", text.index(head))
    depth = 0
    for j in range(i, len(text)):
        depth += {"{": 1, "}": -1}.get(text[j], 0)
        if depth == 0:
            return text[i + 1:j]
    raise AssertionError("unbalanced")


def test_projection_waits_are_bounded():
    src = open(os.path.join(CSRC, "project_tc.cu")).read()
    kernel = _body(src, "k_project(")
    # CTA-wide barriers: before the loops and after them only (nested in no block of the kernel)
    depth, at = 0, []
    for m in re.finditer(r"[{}]|__syncthreads\(\)", kernel):
        if m.group() == "__syncthreads()":
            at.append(depth)
        else:
            depth += 1 if m.group() == "{" else -1
    assert at == [0, 0]
    # no named barrier anywhere: a warp that skips a wait would arrive twice in one of its phases
    code = re.sub(r"//[^\n]*", "", src)
    assert not re.search(r"\bbar\.|(?<!m)barrier\.|__barrier_sync", code)
    # mbarriers are waited for in mbar_wait alone, and there a limited number of times
    assert "try_wait" not in code and "test_wait" not in code
    wait = _body(open(os.path.join(CSRC, "tc_common.cuh")).read(), "bool mbar_wait(")
    assert re.search(r"for \(uint32_t i = 0; i < TC_SPIN_LIMIT; \+\+i\)", wait) and "return false" in wait
    # a failed wait ends its loop; only the last ones, for MMAs in flight, have nothing left to skip
    uses = [u.rstrip() for u in re.findall(r"([^\n]*)wait_all\(&", kernel)]
    assert len(uses) == 4 and sum(not u.endswith(("ok =", "!")) for u in uses) == 1, uses
