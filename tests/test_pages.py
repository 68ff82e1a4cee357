"""How many pages an event has (akv_pages.cuh), compiled for the host: for every page size that a layout may have."""
import ctypes as C
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def event_pages(tmp_path_factory):
    d = tmp_path_factory.mktemp("pages")
    src, so = d / "host.cpp", d / "host.so"
    src.write_text('#include "akv_pages.cuh"\nextern "C" int pages(int N, int shift) { return akv::event_pages(N, shift); }\n')
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", os.path.join(ROOT, "paper_2605_14292_b200", "csrc"), "-o", str(so), str(src)])
    return C.CDLL(str(so)).pages


@pytest.mark.parametrize("N", [1, 2, 15, 16, 17, 129, 192, 255, 256, 5120, 65535])
def test_pages_are_those_whose_first_slot_the_event_has(event_pages, N):
    for shift in range(31):
        pages = event_pages(N, shift)
        assert (pages - 1) << shift < N <= pages << shift
