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


def test_programmatic_kernels_read_only_path_takes_plan_constants():
    """A kernel launched programmatically starts while the previous grid of its
    stream still writes.  The read-only path (ld.global.nc, __ldg) is defined
    only for data that stay unwritten for the kernel's whole life, so there it
    may serve a plan's constants, never a field of the recurrence."""
    constants = r"a\.(kappa|kappa_lo|sp_a|sp_b|active_dev)\b|I\.(kappa|kappa_lo)\b|^p( \+ 1)?$"  # p: the tile table
    seen = 0
    for name in sorted(os.listdir(CSRC)):
        if not name.endswith(".cu") or "griddep_wait()" not in source(name):
            continue
        text = source(name)
        assert "ld.global.nc" not in text
        for m in re.finditer(r"(?:__ldg|\.ldg)\(((?:[^()]|\((?:[^()]|\([^()]*\))*\))*)\)", text):
            seen += 1
            assert re.search(constants, m.group(1)), (name, m.group(0))
    assert seen >= 8
