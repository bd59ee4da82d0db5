"""The benchmark's view of the library's timing slots and bin statistics:
every slot has a name, and no kernel is charged for rows that it does not
take. CPU only."""

import os
import re
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

import bench  # noqa: E402


def test_every_timing_slot_has_a_name():
    text = open(os.path.join(ROOT, "include", "opsparse.h")).read()
    assert bench.NSLOTS == int(re.search(r"\((\d+) slots\)", text).group(1))
    api = open(os.path.join(ROOT, "paper_2206_07244_gb300", "csrc", "api.cu")).read()
    assert bench.NSLOTS == int(re.search(r"kSlots = (\d+)", api).group(1))
    assert bench.SLOT_NAMES[bench.REPEAT_SLOT] == "repeat_rows" and bench.REPEAT_SLOT in bench.KERNEL_SLOTS


def stats(rows, size, nnza, own):
    return [x for v in (rows, size, nnza, own) for x in [v] + [0] * 15]


def test_bytes_are_charged_to_the_kernels_that_take_the_rows():
    b = 1000
    every = stats(100, 5000, 700, 100)
    assert bench._kernel_bytes(every, every, 16, b)[0] == 8 * 100 + 12 * 700 + b + 16 * 100 + 12 * 5000
    assert bench._kernel_bytes(every, every, 0, b)[0] == 8 * 100 + 12 * 700 + b + 16 * 100
    assert bench._kernel_bytes(every, every, bench.REPEAT_SLOT, b)[0] is None
    most = stats(100, 5000, 700, 4)   # 96 rows repeat the row before
    assert bench._kernel_bytes(most, most, 16, b)[0] is None
    assert bench._kernel_bytes(most, most, 0, b)[0] is None
    assert bench._kernel_bytes(most, most, bench.REPEAT_SLOT, b)[0] == 24 * 100 + 12 * (700 + 5000) + b
