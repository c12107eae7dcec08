"""The roles of the tensor-core search meet in waits that end (no GPU).

The kernel's warps take three roles (reduce, produce, issue) that leave their
loops when a bounded wait runs out.  From there on no other role may wait for
them without a limit, and no lane of a warp may go on alone into the
tensor-memory loads and warp barriers that take all 32.  That is a property of
the source, and it is read from there: making a wait run out inside the kernel
would need a GPU that stalls for a second.
"""

import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SEARCH = os.path.join(ROOT, "paper_2311_07561_gb300", "csrc", "k_search_tc.cu")


def _code():
    text = open(SEARCH).read()
    return re.sub(r"//[^\n]*|/\*.*?\*/", "", text, flags=re.S)


def _roles():
    """Source of the whole-warp roles (reduce, produce) and of the issuing thread."""
    text = _code()
    begin = text.index("if (warp < kReduceWarps) {")
    issue = text.index("if (lane == 0 && mine > 0) {", begin)
    end = text.index("__syncthreads_and(ok)", issue)
    return text[begin:issue], text[issue:end]


def test_roles_wait_on_mbarriers_only():
    warps, issue = _roles()
    unlimited = re.compile(r"\bbar\.(?:sync|arrive|red)|\bbarrier\.|__syncthreads|__nanosleep")
    assert not unlimited.findall(warps)
    assert not unlimited.findall(issue)


def test_whole_warps_leave_together():
    warps, issue = _roles()
    assert not re.findall(r"\bmbar_wait(?:_bounded)?\s*\(", warps), "a wait without a vote"
    assert re.findall(r"\bmbar_wait_warp\s*\(", warps)
    assert not re.findall(r"\bmbar_wait_warp\s*\(", issue), "a vote by one lane"
    vote = re.search(r"bool mbar_wait_warp\([^)]*\)\s*\{([^}]*)\}", _code()).group(1)
    assert "__all_sync(0xffffffffu, mbar_wait(" in vote


def test_issuer_drains_its_mmas_on_every_path():
    """A reducing warp may give up after the last chunk was issued: the issuing
    thread then leaves its loop without a fault of its own, and still has to see
    the MMAs done before the kernel frees the tensor memory they write."""
    _, issue = _roles()
    drain = issue[issue.index("for (uint32_t hh = 0"):]
    before = issue[:issue.index("for (uint32_t hh = 0")].rstrip()
    assert "mbar_wait(full0 + 8 * hh" in drain
    assert not re.search(r"if\s*\([^)]*ok[^)]*\)\s*\{$", before), "drained only after a wait of its own ran out"


def test_row_pass_counts_a_copy_it_gave_up_on_as_in_flight():
    """The inverse row pass waits once more for its copies in flight before it
    returns with TTM_ERR_TIMEOUT; the one whose wait ran out is among them."""
    text = open(os.path.join(os.path.dirname(SEARCH), "k_fft.cuh")).read()
    text = re.sub(r"//[^\n]*", "", text)
    kernel = text[text.index("rows_c2r_t(const PS*"):]
    kernel = kernel[:kernel.index("stages_io<")]
    wait = kernel.index("const bool ok = bar_wait(")
    left = kernel.index("return;", wait)
    assert "bar_wait(" in kernel[wait + 30:left], "no second wait"
    assert not re.search(r"pending &=|phase \^=", kernel[wait:left])
    assert re.search(r"pending &= ~", kernel[left:]) and re.search(r"phase \^=", kernel[left:])


def test_refinement_reads_only_grid_points():
    """A search that gave up leaves candidates unwritten, and the refinement is
    queued behind it: what is no index of the grid counts as no candidate, not
    only the mark for none."""
    text = open(os.path.join(os.path.dirname(SEARCH), "k_rotation.cuh")).read()
    text = re.sub(r"//[^\n]*", "", text)
    assert not re.search(r"[=!]= 0xFFFF", text)
    reads = re.findall(r"a\.gq \+ 4 \* (\w+)", text)
    assert sorted(set(reads)) == ["gi", "ia", "ib"]
    for index in set(reads):
        assert re.search(rf"\b{index} (?:>=|<) a\.n_grid", text), index
