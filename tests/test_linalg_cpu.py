"""Host-side checks of the linear algebra unit (no GPU)."""
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1601_02713_gb300", "csrc")


def _code(path):
    """The file without its comments."""
    with open(path) as fh:
        return re.sub(r"//[^\n]*", "", fh.read())


def test_jacobi_norm_update_is_ordered_after_every_lanes_read():
    """All lanes of a warp read a column pair's norms, lane 0 then overwrites
    them: between the two stands a warp barrier that orders memory (shuffles do
    not), outside any branch."""
    code = _code(os.path.join(CSRC, "linalg.cu"))
    read = code.index("al = nrm[p], be = nrm[q]")
    write = code.index("nrm[p] = al - tg")
    between = code[read:write]
    assert "__syncwarp();" in between
    head = between[:between.index("__syncwarp();")]
    assert head.count("{") == head.count("}") == 0
