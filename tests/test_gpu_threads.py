"""Calls from several host threads, a handle and a stream each: the library's kernels are shared by all of them."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest
import torch

import __graft_entry__ as entry
import paper_2605_14292_b200 as akv
from paper_2605_14292_b200 import synth

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
# two threads that call as fast as a host program can: the time between a call's preparation and its launch is a microsecond or two
HOST = r"""
#include <atomic>
#include <thread>
#include "alphakv.h"
typedef akv_status_t (*event_fn)(akv_handle_t*, const akv_layout_t*, void*, void*, int32_t*, int64_t, int64_t, int64_t, const int32_t*, const float*,
                                 const int32_t*, const float*, int32_t, const akv_options_t*, int32_t*, int32_t*, float*, float*, int32_t*, int32_t*, void*);
struct Side { akv_handle_t* h; const akv_layout_t* lay; void *K, *V; int32_t* pos; const float* q; const int32_t* p_ref; int32_t* idx; void* stream; };
extern "C" int hammer(event_fn event, const Side* side, int budget, const akv_options_t* opt, int calls) {
    std::atomic<int> refused{0}, ready{0};
    auto work = [&](const Side& s) {
        ++ready;
        while (ready < 2) {}
        for (int i = 0; i < calls; ++i)
            if (event(s.h, s.lay, s.K, s.V, s.pos, s.lay->N, s.lay->N, s.lay->N, nullptr, s.q, s.p_ref, nullptr, budget, opt, s.idx, nullptr, nullptr, nullptr, nullptr, nullptr, s.stream) != AKV_OK) ++refused;
    };
    std::thread a(work, side[0]), b(work, side[1]);
    a.join();
    b.join();
    return refused;
}
"""


class Side(C.Structure):
    _fields_ = [(n, C.c_void_p) for n in ("h", "lay", "K", "V", "pos", "q", "p_ref", "idx", "stream")]


@pytest.fixture(scope="module")
def hammer(tmp_path_factory):
    entry.build()
    d = tmp_path_factory.mktemp("threads")
    (d / "host.cpp").write_text(HOST)
    subprocess.check_call(["g++", "-std=c++17", "-O2", "-shared", "-fPIC", "-pthread", "-I", os.path.join(ROOT, "include"), "-o", str(d / "host.so"), str(d / "host.cpp")])
    return C.CDLL(str(d / "host.so")).hammer


# sizes of one kernel whose shared memory differs: the prefill kernel, the resident one
@pytest.mark.parametrize("dtype,sizes", [(synth.BF16, (300, 5000)), (synth.F32, (110, 190))])
def test_two_threads_with_different_sizes(hammer, dtype, sizes):
    """One thread's smaller call does not lower the shared memory that the other one's launch may take: no call is refused, and
    both threads' selections are those of a call alone."""
    lib, budget, opts = akv.load_library(), 16, akv.Options(lam=0.0).c()
    sides, keep = (Side * 2)(), []
    for side, N in zip(sides, sizes):
        ev = synth.make_plain(1, 1, 1, N, 128, budget, 0.0, dtype=dtype, seed=N)
        h, st = C.c_void_p(), torch.cuda.Stream()
        assert lib.akv_create(C.byref(h), 0) == 0
        K, V, pos, q, pref = (akv.to_device(x, "cuda") for x in (ev.K, ev.V, ev.pos, ev.qstat, ev.p_ref))
        alone = akv.alpha_compress_event(K, V, pos, q, budget, akv.Options(lam=0.0), p_ref=pref).idx_sorted.clone()
        after = [x.clone() for x in (K, V, pos)]
        again = akv.alpha_compress_event(K, V, pos, q, budget, akv.Options(lam=0.0), p_ref=pref).idx_sorted.clone()
        lay, idx = akv.Layout.dense(K).c(), torch.empty_like(alone)
        for x, y in zip((K, V, pos), after):
            x.copy_(y)
        keep.append((h, lay, K, V, pos, q, pref, idx, st, again))
        side.h, side.lay, side.stream = h, C.addressof(lay), st.cuda_stream
        side.K, side.V, side.pos, side.q, side.p_ref, side.idx = (x.data_ptr() for x in (K, V, pos, q, pref, idx))
    torch.cuda.synchronize()
    assert hammer(C.cast(lib.alpha_compress_event, C.c_void_p), sides, budget, C.byref(opts), 1) == 0
    torch.cuda.synchronize()
    for _, _, _, _, _, _, _, idx, _, again in keep:
        assert np.array_equal(idx.cpu().numpy(), again.cpu().numpy())
    refused = hammer(C.cast(lib.alpha_compress_event, C.c_void_p), sides, budget, C.byref(opts), 15000)
    torch.cuda.synchronize()
    for k in keep:
        lib.akv_destroy(k[0])
    assert refused == 0
