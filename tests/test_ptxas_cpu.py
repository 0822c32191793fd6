"""What the compiler makes of the kernels that keep their state in registers
(nvcc -Xptxas -v; no GPU needed)."""
import os
import re
import subprocess


def spills(tmp_path, source, pattern):
    """{integers of the mangled template arguments: bytes of spill stores} of a file's kernels."""
    from paper_2507_02401_gb300 import build
    src = os.path.join(build.CSRC, source)
    r = subprocess.run([build.nvcc()] + build.ARCH + build.FLAGS + ["-Xptxas", "-v", "-c", src, "-o",
                                                                    str(tmp_path / "k.o")],
                       capture_output=True, text=True, check=True)
    found = {}
    for name, spill in re.findall(r"Compiling entry function '(\S+)'.*?(\d+) bytes spill stores", r.stderr, re.S):
        m = re.search(pattern, name)
        if m:
            found[tuple(int(g) for g in m.groups())] = int(spill)
    return found


def test_persistent_forms_with_an_sm_to_themselves_do_not_spill(tmp_path):
    # R, adjoint, varying, layer, right-hand sides, CTAs per SM
    found = spills(tmp_path, "wave2d_persist.cu", r"wave2d_persist_kernelILi(\d+)ELb(\d)ELb(\d)ELb(\d)ELi(\d+)ELi(\d+)E")
    forms = {k: v for k, v in found.items() if k[4] == 1 and k[5] == 1}
    assert len(forms) == 4 * 2 * 2 * 2
    assert {k: v for k, v in forms.items() if v} == {}


def test_batched_one_launch_forms_keep_their_state_in_registers(tmp_path):
    """At most a few words of the tile loop's bookkeeping are spilled, never cells of the update (16 words a row)."""
    # R, tile rows, adjoint, all steps in one launch
    found = spills(tmp_path, "batch_kernels.cu", r"batch_step_kernelILi(\d+)ELi(\d+)ELb(\d)ELb(\d)E")
    forms = {k: v for k, v in found.items() if k[3] == 1}
    assert len(forms) == 4 * 2 * 2
    assert {k: v for k, v in forms.items() if v >= 64} == {}
