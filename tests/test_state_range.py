"""The rule by which rlb_get_state and rlb_set_state let a kernel reach a
device buffer (rlb_internal.h: holds): the whole state lies in the allocation
that the buffer starts in.  A shorter buffer goes through a copy that the
runtime checks, so that no kernel leaves an allocation."""
import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PROGRAM = r"""
#include <cstdio>
#include "rlb_internal.h"
int main()
{
    const unsigned long long a = 0x7f0000000000ull, top = ~0ull;
    struct { unsigned long long start; size_t size; unsigned long long at; size_t bytes; int want; } t[] = {
        {a, 1000, a, 1000, 1},      {a, 1000, a, 1001, 0},    {a, 1000, a + 4, 996, 1}, {a, 1000, a + 4, 997, 0},
        {a, 1000, a + 1000, 0, 1},  {a, 1000, a + 1001, 0, 0}, {a, 1000, a - 4, 8, 0},   {a, 0, a, 4, 0},
        {a, 1000, a, (size_t)top, 0}, {a, 1000, a + 8, (size_t)(top - 4), 0}};
    for (auto &c : t)
        if (rlb::holds(c.start, c.size, c.at, c.bytes) != (c.want != 0)) return 1;
    return std::puts("ok") < 0;
}
"""


def test_only_whole_buffers_are_reached_by_a_kernel(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    src = tmp_path / "t.cpp"
    src.write_text(PROGRAM)
    csrc = os.path.join(ROOT, "paper_1302_1125_gb300", "csrc")
    subprocess.run([nvcc, "-std=c++20", "-I", csrc, "-o", str(tmp_path / "t"), str(src)], check=True)
    assert subprocess.run([str(tmp_path / "t")], capture_output=True, text=True).stdout == "ok\n"
    api = open(os.path.join(csrc, "rlb_api.cu")).read()
    assert re.search(r"&& in_one_allocation\(\w+, (bytes|rlb_state_bytes\(ctx\))\)", api)
