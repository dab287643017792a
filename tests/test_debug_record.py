"""The bounds-checked build's records: every source file's is read, wherever
its checks are (host code, no GPU)."""
import os
import re
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1701_03038_gb300", "csrc")

UNIT = r"""
#include "debug_record.cuh"
static unsigned long long held = VIOLATIONS;
static int read_own(fstgpu::DebugCounts* out) {
  *out = fstgpu::DebugCounts{held, CODE, CODE * 10, CODE * 100};
  held = 0;
  return 0;
}
static fstgpu::DebugRecord record(read_own);
"""
MAIN = r"""
#include <cstdio>
#include "debug_record.cuh"
int main() {
  for (int i = 0; i < 2; ++i) {
    fstgpu::DebugCounts d;
    if (fstgpu::debug_read_all(&d)) return 1;
    printf("%llu %llu %llu %llu\n", d.violations, d.code, d.index, d.bound);
  }
}
"""


def test_every_files_record_is_read(tmp_path):
    if shutil.which("g++") is None:
        pytest.skip("g++ not available")
    files = [tmp_path / "main.cpp"]
    files[0].write_text(MAIN)
    for i, (n, code) in enumerate([(0, 1), (3, 5), (0, 2), (4, 5)]):
        p = tmp_path / f"u{i}.cpp"
        p.write_text(UNIT.replace("VIOLATIONS", str(n)).replace("CODE", str(code)))
        files.append(p)
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, "-o", str(tmp_path / "t"), *map(str, files)], check=True)
    out = subprocess.run([str(tmp_path / "t")], check=True, capture_output=True, text=True).stdout.splitlines()
    assert out == ["7 5 50 500", "0 0 0 0"]


def test_the_checks_and_their_record_come_together():
    # the header that defines the checks lists the including file's record;
    # no other source has a record of its own
    with open(os.path.join(CSRC, "frontier.cuh")) as fh:
        text = fh.read()
    assert re.search(r"static DebugRecord \w+\(debug_read_own\);", text)
    for name in sorted(os.listdir(CSRC)):
        with open(os.path.join(CSRC, name)) as fh:
            text = fh.read()
        if name != "frontier.cuh":
            assert "g_dbg" not in text, name
        if "in_bounds(" in text and name != "frontier.cuh":
            assert '#include "frontier.cuh"' in text, name
