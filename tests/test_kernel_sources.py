"""Rules of the kernels that no run on a GPU can show: what a source line may
read, and when.  Each rule is checked on the text of the CUDA files."""
import os
import re
import shutil
import subprocess

import pytest

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


def test_no_value_of_one_device_serves_another():
    """Occupancies and kernel attributes belong to a device.  A function-local
    static that is not constant holds the first caller's, for every device and
    without synchronisation; PerDevice (csrc/per_device.h) keeps one per device.
    (The tensor-map encoder, under a once_flag, is the driver's, not a device's.)"""
    for name in sorted(os.listdir(CSRC)):
        for m in re.finditer(r"^[ \t]+static\s+(?!const|inline)([^;({=]*)[;({=]", source(name), re.M):
            encoder = name == "wave3d_tma.cu" and re.search(r"\b(fn|once)\s*$", m.group(1))
            ok = m.group(1).startswith("PerDevice ") or encoder
            assert ok, (name, m.group(0))


PER_DEVICE_MAIN = r"""
#include <cstdio>
#include <thread>
#include <vector>
#include "per_device.h"
static pat::PerDevice kept;
int main() {
  std::atomic<int> calls{0};
  auto value = [&](int d) { return kept.get(d, [&] { ++calls; return d == 5 ? 0 : 100 + d; }); };
  std::vector<std::thread> t;
  std::atomic<int> bad{0};
  for (int i = 0; i < 8; ++i)
    t.emplace_back([&, i] {
      for (int k = 0; k < 2000; ++k) {
        const int d = (k + i) % 5;
        if (value(d) != 100 + d) ++bad;
      }
    });
  for (auto& x : t) x.join();
  if (calls > 8 * 5) ++bad;            // kept: at most once per thread and device
  if (value(5) != 0 || value(5) != 0) ++bad;  // a failure is not kept
  const int before = calls;
  if (kept.get(5, [] { return 7; }) != 7 || value(5) != 7 || calls != before) ++bad;
  if (kept.get(64, [] { return 3; }) != 3 || kept.get(-1, [] { return 4; }) != 4) ++bad;  // no entry: worked out anew
  std::printf("%d\n", (int)bad);
  return bad != 0;
}
"""


def test_per_device_values(tmp_path):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no host compiler")
    (tmp_path / "m.cpp").write_text(PER_DEVICE_MAIN)
    exe = str(tmp_path / "m")
    subprocess.run([cxx, "-std=c++17", "-O2", "-pthread", "-I", CSRC, str(tmp_path / "m.cpp"), "-o", exe], check=True)
    subprocess.run([exe], check=True)
