"""The search for the key that bounds an active set (akv_active_set.cuh), compiled for the host: for any scores the set has
rows, never more than its size, and no key left out lies above the bound."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
HOST = r"""
#include "akv_active_set.cuh"
extern "C" void bound(const uint32_t* key, int n, uint32_t low, uint32_t kb, int cap, int enough, int least, uint32_t* out, int* ties) {
    auto count = [&](uint32_t v) { int c = 0; for (int i = 0; i < n; ++i) c += key[i] >= v; return c; };
    const akv::ActiveBound b = akv::active_bound(low, kb, cap, enough, least, [&](uint32_t v1, uint32_t v2, uint32_t v3, int& c1, int& c2, int& c3) {
        c1 = count(v1); c2 = count(v2); c3 = count(v3);
    });
    *out = b.key;
    *ties = b.ties;
}
"""


@pytest.fixture(scope="module")
def search(tmp_path_factory):
    d = tmp_path_factory.mktemp("active_set")
    src, so = d / "host.cpp", d / "host.so"
    src.write_text(HOST)
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", os.path.join(ROOT, "paper_2605_14292_b200", "csrc"),
                           "-o", str(so), str(src)])
    lib = C.CDLL(str(so))

    def run(keys, low, kb, cap, enough, least):
        out, ties = C.c_uint32(), C.c_int()
        lib.bound(np.ascontiguousarray(keys).ctypes.data_as(C.c_void_p), len(keys), C.c_uint32(low), C.c_uint32(kb), cap, enough, least,
                  C.byref(out), C.byref(ties))
        return out.value, ties.value
    return run


def orderable(x):
    u = np.asarray(x, dtype=np.float32).view(np.uint32)
    return np.where(u & 0x80000000, ~u, u | 0x80000000).astype(np.uint32)


def coarse_kth(keys, picks):
    """the picks-th largest key, its 14 low bits open (from below)"""
    return int(np.sort(keys)[::-1][picks - 1]) & ~0x3FFF


# (rows, budget, set size, enough, least): the small kernel, the 256 -> 128 kernel, the prefill kernel
SHAPES = [(192, 64, 127, 128, 112), (128, 128, 127, 128, 112), (256, 128, 180, 181, 158), (1000, 128, 192, 184, 160), (5000, 128, 192, 184, 160)]
SCORES = {
    "equal": lambda rng, n: np.full(n, 0.3),
    "zero": lambda rng, n: np.zeros(n),
    "close 1e-3": lambda rng, n: 0.3 + 1e-3 * rng.standard_normal(n),
    "close 3e-3": lambda rng, n: 0.3 + 3e-3 * rng.standard_normal(n),
    "one bucket": lambda rng, n: rng.uniform(0.25, 0.2578, n),
    "few values": lambda rng, n: rng.integers(0, 3, n) * 0.25,
    "non-finite": lambda rng, n: np.full(n, -np.inf),
    "mostly non-finite": lambda rng, n: np.where(np.arange(n) % 16 == 3, rng.standard_normal(n), -np.inf),
    "normal": lambda rng, n: rng.standard_normal(n),
    "negative": lambda rng, n: -5 + 0.1 * rng.standard_normal(n),
}


@pytest.mark.parametrize("lam", [0.25, 0.5, 1.0, 4.0])
@pytest.mark.parametrize("scores", list(SCORES))
@pytest.mark.parametrize("n,picks,cap,enough,least", SHAPES)
def test_active_set_is_filled_and_bounded(search, n, picks, cap, enough, least, scores, lam):
    rng = np.random.default_rng(n)
    s = SCORES[scores](rng, n).astype(np.float32)
    keys = orderable(s)
    kb = coarse_kth(keys, picks)
    sb = np.uint32(kb & 0x7FFFFFFF if kb & 0x80000000 else ~kb & 0xFFFFFFFF).view(np.float32)
    with np.errstate(invalid="ignore"):
        thr = np.float32(-np.inf) if kb < 0x00800000 else np.float32(np.float64(-1.001) * lam + sb) - np.float32(1e-6) * np.abs(sb)
    low = int(orderable(thr))
    pool = keys >= low
    assert pool.sum() >= picks
    if pool.sum() <= cap:
        return                      # the set is the whole pool, there is nothing to search
    bound, ties = search(keys, low, kb, cap, enough, least)
    above = pool & (keys > bound)
    equal = np.flatnonzero(keys == bound)
    assert ties == 0 or (bound >= low and ties < len(equal))
    chosen = np.flatnonzero(above).tolist() + equal[:ties].tolist()
    assert least <= len(chosen) <= cap
    left = np.setdiff1d(np.flatnonzero(pool), chosen)
    assert len(left) and np.all(keys[left] <= bound)
    assert ties == 0 or len(chosen) == cap
