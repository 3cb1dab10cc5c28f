"""A lane that has held no task yet takes the walk's deep steps along with the
others, and the steps read a row's features without a predicate: what such a
lane reads has to lie in the tile (feature 0 of its first row), not at shared
address 0, which is no object of the kernel's.  The lane's first state is made
by host code too, so it is checked here without a GPU."""
import os
import re
import subprocess

import pytest

from paper_1806_07300_gb300 import _build

MAIN = """
#include <cstdio>
#include "fp_traverse.cuh"
int main() {
    const uint32_t bases[] = {1024u, 1040u, 4096u};
    for (uint32_t base : bases) {
        const LaneTask L = idle_task(base);
        std::printf("%u %u %u %u %d\\n", base, L.ref, L.xb, L.rt, L.bad);
    }
}
"""


def test_a_lane_without_a_task_reads_the_tile(tmp_path):
    try:
        nvcc = _build.nvcc()
    except RuntimeError as e:
        pytest.skip(str(e))
    src, exe = tmp_path / "idle.cu", tmp_path / "idle"
    src.write_text(MAIN)
    subprocess.run([nvcc, *_build.ARCH, "-std=c++17", "-O0", "-I", _build.CSRC, str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout
    lines = [list(map(int, line.split())) for line in out.splitlines()]
    assert lines == [[b, 0xFFFFFFFF, b, 0, 0] for b in (1024, 1040, 4096)]


def test_the_walk_starts_from_that_state():
    with open(os.path.join(_build.CSRC, "fp_traverse.cuh")) as f:
        text = f.read()
    text = text.replace("__host__ __device__ __forceinline__ LaneTask idle_task(uint32_t base) {\n    LaneTask L;", "")
    assert re.findall(r"LaneTask L\b(?!\s*[,)])[^;]*;", text) == ["LaneTask L = idle_task(base);"]
