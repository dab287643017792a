"""The size rule of the (symbol, state) table, compiled for the host, and the
bucketed table at the loads it allows (no GPU)."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1701_03038_gb300", "csrc")

HARNESS = r"""
#include <cstdio>
#include <cstdlib>
#include <initializer_list>
#include "seg_table.cuh"
int main(int, char** v) {
  printf("%lld\n", (long long)fstgpu::seg_buckets(atoll(v[1]), atoll(v[2])));
}
"""
MOST = 2**31 - 1


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("g++ not available")
    d = tmp_path_factory.mktemp("seg")
    (d / "t.cpp").write_text(HARNESS)
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, "-o", str(d / "t"), str(d / "t.cpp")], check=True)
    return lambda n, free: int(subprocess.run([str(d / "t"), str(n), str(free)], check=True, capture_output=True,
                                              text=True).stdout)


@pytest.mark.parametrize("nseg", [0, 1, 2, 1000, 90_000_000, 1_431_655_765, 1_600_000_000, 2_000_000_000, MOST])
@pytest.mark.parametrize("free", [0, 10**6, 8 * 10**9, 100 * 10**9, 280 * 10**9])
def test_size_rule(harness, nseg, free):
    b = harness(nseg, free)
    assert 1 <= b <= MOST and 2 * b >= nseg * 1.125  # (every segment has a slot, and some stay empty)
    full, least = 1 + max(nseg, 1) * 3 // 2, 1 + max(nseg, 1) * 9 // 16
    if full <= MOST and full * 64 <= free // 3:
        assert b == full  # three slots a segment wherever they fit
    elif b * 64 > free // 3:
        assert b == min(least, MOST)  # nothing smaller would do
