"""Give-up paths of the tensor-core kernels, checked in the source (they run only
after a wait of about two seconds has expired, which no test may bring about).

A warp with collective operations ahead has to leave its loop as a whole: every
bounded wait of such a kernel is the voting one, so that no lane branches on its
own outcome."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2108_01186_gb300", "csrc")


def _code(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def test_the_voting_wait_returns_the_vote():
    body = re.search(r"bool tc_mbar_warp_wait\([^)]*\) \{(.*?)\n\}", _code("tcgen05.cuh"), re.S).group(1)
    assert re.search(r"return __all_sync\(0xffffffffu, tc_mbar_sleep_or_abort\(bar, parity, abort\)\);", body)


@pytest.mark.parametrize("name", ["kron_tc.cu", "gram_tc.cu"])
def test_no_lane_branches_on_its_own_wait(name):
    code = _code(name)
    assert "tc_mbar_warp_wait" in code
    assert not re.findall(r"tc_mbar_(?:sleep|wait)_or_abort", code)
    assert not re.findall(r"if \(!?s_abort\)|= !?s_abort;", code), "warps decide on the flag by a vote"
    assert not re.findall(r"if \(!?__all_sync", code), "a vote has to be kept: what follows must not use a lane's own value"


def test_teardown_waits_for_the_last_unit_committed():
    """Units of a tile given up half-way are in flight too: the count that the teardown
    takes its slot and phase from goes up with every commit to a unit's mbarrier."""
    code = _code("kron_tc.cu")
    commits = re.findall(r"umma_commit\(&bar_full\[sl\]\);\s*(\S+)", code)
    assert commits == ["++s_units;"]
    assert code.count("++s_units") == 1 and "tc_mbar_wait(&bar_half" not in code
    teardown = code[code.index("if (s_abort && tid == 0)"):code.index("tmem_dealloc")]
    assert re.search(r"tc_last_commit\(s_units, S::kUnits\);\s*"
                     r"if \(lc\.slot >= 0\) tc_mbar_wait\(&bar_full\[lc\.slot\], lc\.parity\);", teardown)
