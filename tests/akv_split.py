"""The prefill kernel's rule for the number of CTAs that share an event's scoring (akv_split_rule.cuh), compiled for the host."""
import ctypes as C
import os
import subprocess
import tempfile

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
HOST = r"""
#include "akv_split_rule.cuh"
extern "C" int rule(long long events, int N, int sms, int topk, int ragged) { return akv::prefill_split(events, N, sms, topk, ragged); }
extern "C" long long tail(long long events, int N, int sms, int topk, int ragged) { return akv::prefill_tail(events, N, sms, topk, ragged); }
extern "C" int tail_split(long long tail, int sms) { return akv::prefill_tail_split(tail, sms); }
extern "C" int share(int stages, int split) { return akv::split_share(stages, split); }
"""
_lib = None


def _load():
    global _lib
    if _lib is None:
        with tempfile.TemporaryDirectory() as d:
            src, so = os.path.join(d, "host.cpp"), os.path.join(d, "host.so")
            with open(src, "w") as f:
                f.write(HOST)
            subprocess.check_call(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", os.path.join(ROOT, "paper_2605_14292_b200", "csrc"), "-o", so, src])
            _lib = C.CDLL(so)
        _lib.rule.argtypes = _lib.tail.argtypes = [C.c_longlong, C.c_int, C.c_int, C.c_int, C.c_int]
        _lib.tail.restype = C.c_longlong
        _lib.tail_split.argtypes = [C.c_longlong, C.c_int]
    return _lib


def prefill_split(events, N, sms=148, topk=False, ragged=False):
    return _load().rule(events, N, sms, topk, ragged)


def prefill_tail(events, N, sms=148, topk=False, ragged=False):
    return _load().tail(events, N, sms, topk, ragged)


def prefill_tail_split(tail, sms=148):
    return _load().tail_split(tail, sms)


def split_share(stages, split):
    return _load().share(stages, split)
