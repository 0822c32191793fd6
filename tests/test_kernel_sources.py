"""Rules of the kernels that no run on a GPU can show: what a source line may
read, and when.  Each rule is checked on the text of the CUDA files."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2507_02401_gb300", "csrc")


def source(name):
    """A file's text without its comments."""
    with open(os.path.join(CSRC, name)) as f:
        text = f.read()
    return re.sub(r"//[^\n]*", "", re.sub(r"/\*.*?\*/", "", text, flags=re.S))


def test_step2d_tma_reads_cells_only_under_a_bounds_test():
    """A tile at the grid's edge has threads whose cells lie beyond the field.
    A subscript such as a.kappa[gi + j], evaluated before the test that the
    cell exists, reads past the end of the allocation; the kernel's per-cell
    accesses are loads and stores of whole quads, each under its own test."""
    text = source("wave2d_tma.cu")
    fields = r"a\.(kappa|kappa_lo|sp_a|sp_b|cur_lo|next|next_lo|dbuf_lo|lp|gsum_hi|gsum_lo)\s*\["
    assert re.findall(fields, text) == []
    # the injection's and the sensors' lists hold cells of the field
    assert re.findall(r"a\.dbuf\s*\[([^\]]*)\]", text) == ["c.local"]
    assert re.findall(r"a\.cur\s*\[(\S+?)\[", text) == ["a.sens_cell"]
