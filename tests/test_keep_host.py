"""CPU: sizes of what the wide tier keeps (csrc/kk_keep.h), compiled for the host:
within the budget with all that belongs to it, an index no larger than B, and nothing
at all where the budget does not reach."""
import ctypes
import os
import random
import subprocess

import pytest

from paper_2103_11991_gb300 import _build

CODE = r"""
#include "kk_keep.h"
extern "C" void plan(long long budget, const long long* in, long long* out) {
  const kk::KeepSizes s{in[0], in[1], in[2], in[3], in[4], in[5], in[6], in[7]};
  const kk::KeepPlan p = kk::keep_plan(budget, s);
  out[0] = p.slots; out[1] = p.tasks; out[2] = p.index_rows; out[3] = kk::keep_bytes(s, p);
}
"""


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    d = tmp_path_factory.mktemp("keep")
    src, lib = d / "keep.cpp", d / "keep.so"
    src.write_text(CODE)
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-I", _build.CSRC, str(src), "-o", str(lib)],
                   check=True)
    so = ctypes.CDLL(os.fspath(lib))

    def call(budget, *sizes):
        a, out = (ctypes.c_longlong * 8)(*sizes), (ctypes.c_longlong * 4)()
        so.plan(ctypes.c_longlong(budget), a, out)
        return list(out)
    return call


GB = 1 << 30


def test_half_a_million_rows_of_the_widest_b(plan):
    # 16,384 words and a table of 215 chunks a row, 1,600 products a row, no long rows of B
    slot = (16384 + 432) * 4
    slots, tasks, index, total = plan(36 * GB, 520000, 520000, 520000, slot, 10, 832000000 // 2560, 0, 513 * 4)
    assert total <= 36 * GB and slots * slot >= 0.99 * min(36 * GB, 520000 * slot) and index == 0
    assert tasks == 832000000 // 2560 + 10 * slots


def test_index_is_no_larger_than_b(plan):
    # 1,000 rows of 100,000 entries: 781,250 rows of 128 entries would fit nnz
    slots, tasks, index, total = plan(36 * GB, 1000, 1000, 1000, 70000, 10, 10000, 781250, 513 * 4)
    assert index == 1000 and slots == 1000 and total < 0.1 * GB


@pytest.mark.parametrize("chunks", [True, False])
def test_plans_stay_within_the_budget(plan, chunks):
    rng = random.Random(7)
    log = lambda hi: int(2 ** rng.uniform(0, hi))  # noqa: E731
    for _ in range(3000):
        rows, b_rows = log(27), log(27)
        sizes = (rows, b_rows, min(rows, log(27)), 4 * (1024 * rng.randint(1, 17) + 500), rng.randint(2, 10) if chunks else 0,
                 log(28) if chunks else 0, log(23) if chunks else 0, 4 * rng.randint(3, 513))
        budget = log(36)
        slots, tasks, index, total = plan(budget, *sizes)
        assert slots <= sizes[2] and index <= min(sizes[6], b_rows) and min(slots, tasks, index) >= 0
        if slots > 0:
            assert total <= budget
            assert not chunks or tasks >= min(slots * sizes[4], 1 << 28)
        bigger = plan(2 * budget, *sizes)
        assert bigger[0] >= slots
