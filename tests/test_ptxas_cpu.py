"""What the compiler makes of the kernels that keep their state in registers
(nvcc -Xptxas -v; no GPU needed)."""
import os
import re
import subprocess

import pytest


@pytest.fixture(scope="module")
def persistent(tmp_path_factory):
    """{(R, adjoint, varying, layer, right-hand sides, CTAs per SM): bytes of spill stores}"""
    from paper_2507_02401_gb300 import build
    out = str(tmp_path_factory.mktemp("ptxas") / "k.o")
    src = os.path.join(build.CSRC, "wave2d_persist.cu")
    r = subprocess.run([build.nvcc()] + build.ARCH + build.FLAGS + ["-Xptxas", "-v", "-c", src, "-o", out],
                       capture_output=True, text=True, check=True)
    found = {}
    for name, spill in re.findall(r"Compiling entry function '(\S+)'.*?(\d+) bytes spill stores", r.stderr, re.S):
        m = re.search(r"wave2d_persist_kernelILi(\d+)ELb(\d)ELb(\d)ELb(\d)ELi(\d+)ELi(\d+)E", name)
        if m:
            found[tuple(int(g) for g in m.groups())] = int(spill)
    return found


def test_forms_with_an_sm_to_themselves_do_not_spill(persistent):
    forms = {k: v for k, v in persistent.items() if k[4] == 1 and k[5] == 1}
    assert len(forms) == 4 * 2 * 2 * 2
    assert {k: v for k, v in forms.items() if v} == {}
