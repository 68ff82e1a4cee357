"""Where event_pool_kernel keeps an event's rows while it scores them (akv_score_order.cuh), compiled for the host."""
import ctypes as C
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
HOST = r"""
#include "akv_score_order.cuh"
extern "C" int steps(int n) { return akv::score_steps(n); }
extern "C" int shift(int step, int steps, int chain) { return akv::late_slot_shift(step, steps, chain); }
extern "C" int late_steps() { return akv::kLateSteps; }
extern "C" int chain_slots() { return akv::kChainSlots; }
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("score_order")
    src, so = d / "host.cpp", d / "host.so"
    src.write_text(HOST)
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", os.path.join(ROOT, "paper_2605_14292_b200", "csrc"), "-o", str(so), str(src)])
    return C.CDLL(str(so))


def rows_of_step(i, chain, steps, n):
    first = 16 * (i + chain * steps)
    return range(first, min(first + 16, n))


@pytest.mark.parametrize("n", [0, 1, 15, 16, 17, 31, 32, 33, 128, 129, 192, 193, 208, 209, 241, 255, 256])
def test_two_chains_hold_every_row_once(lib, n):
    steps = lib.steps(n)
    assert sorted(j for i in range(steps) for c in (0, 1) for j in rows_of_step(i, c, steps, n)) == list(range(n))


@pytest.mark.parametrize("n", range(193, 257))
def test_late_rows_come_into_slots_that_have_been_scored(lib, n):
    """192 slots: every row lies in one when it is scored, the late ones overwrite none that is still to be, and each of the kernel's
    four copies is one stretch of rows into one stretch of slots."""
    steps, late = lib.steps(n), lib.late_steps()
    assert 2 * late < steps and 2 * lib.chain_slots() == 192
    late0 = 16 * (steps - late)
    held, scored = {}, set()

    def copy(r0, r1, slot0):
        for j in range(r0, r1):
            slot = slot0 + j - r0
            assert 0 <= j < n and 0 <= slot < 192 and (slot not in held or held[slot] in scored)
            held[slot] = j

    copy(0, late0, 0)
    copy(16 * steps, 16 * steps + late0, lib.chain_slots())
    for i in range(steps):
        if i == late:
            copy(late0, 16 * steps, 0)
            copy(16 * steps + late0, n, lib.chain_slots())
        for chain in (0, 1):
            for j in rows_of_step(i, chain, steps, n):
                assert held[j + lib.shift(i, steps, chain)] == j
                scored.add(j)
    assert scored == set(range(n))
