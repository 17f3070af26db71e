"""An expired wait reaches the caller, checked in the source (no test may bring one about):
every warp of the overlap kernels that gives up sets the status bit, since its partial
sums are missing, and every entry that reads the status words looks at that one."""
import re

from test_tc_abort_paths import _code


def test_every_warp_of_the_overlap_kernels_reports():
    code = _code("gram_tc.cu")
    assert len(re.findall(r"if \(!ok && lane == 0\)\s*\{?\s*atomicOr\(status \+ 3, 2\);", code)) == 2
    assert code.count("atomicOr(status + 3, 2)") == 2


def test_every_entry_that_reads_the_status_looks_at_the_expired_waits():
    code = _code("api.cu")
    parts = re.split(r"read_status\(c, s, st\);", code)[1:]
    assert len(parts) == 3     # FLO build, Poisson, exact adjoint
    for p in parts:
        assert re.search(r"if \(st\[3\]\)\s*return fail\(c, FLOSIC_ERR_CUDA", p[:p.index("return FLOSIC_OK;")])
