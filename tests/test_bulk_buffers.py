"""Shared memory of the bulk-staged FP32 step (csrc/rlb_bulk.cuh,
rlb_step_f32_bulk.cu): six items in flight, the number the copy plan of
test_bulk_plan.py is checked with, and two blocks on an SM (228 KB, of which
each block takes 1 KB more than it asks for)."""
import os
import re

from test_bulk_plan import NB, TILE

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1302_1125_gb300", "csrc")


def constant(name, *files):
    text = "".join(open(os.path.join(CSRC, f)).read() for f in files)
    m = re.search(rf"(?:#define\s+{name}\s+|constexpr int {name}\s*=\s*)(\d+)", text)
    assert m, name
    return int(m.group(1))


def test_six_items_in_flight_and_two_blocks_per_sm():
    bufs = constant("RLB_BULK_BUFS", "rlb_bulk.cuh")
    assert bufs == NB == 6
    slots = constant("kParkH", "rlb_step_f32.cuh")
    kernel = open(os.path.join(CSRC, "rlb_step_f32_bulk.cu")).read()
    # the parked coefficients: the slots the size of the dynamic shared memory counts
    park = re.search(r"sizeof\(f2\) \* size_t\(([^)]*)\)", kernel).group(1)
    slots += constant("kEqSlots", "rlb_step_f32.cuh") if "kEqSlots" in park else 0
    block = 4 * bufs * TILE + 8 * slots * 256 + 8 * bufs + 2 * 4 * bufs + 4 * 16
    assert 2 * (block + 1024) <= 228 * 1024
