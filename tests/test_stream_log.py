"""What a kernel that begins early may read (csrc/segkv_stream_log.h), on the CPU: chains of launches on streams that share a
handle's value on two devices, appends that let their successors go at once, more streams than the log keeps."""
import ctypes
import os
import subprocess

import pytest

from paper_2401_05391_b200 import build as b

SOURCE = r"""
#include "segkv_stream_log.h"
using namespace segkv_impl;
static StreamLog* g;
static WriteMark marks[256];
extern "C" void fresh() { delete g; g = new StreamLog(); }
extern "C" int note(int dev, long st, long th, int rel) {
    static int n;
    n = (n + 1) % 256;
    StreamKey k{dev, (const void*)st, (const void*)th};
    marks[n] = WriteMark{k, g->note(k, (Release)rel)};
    return n;
}
extern "C" int complete(int dev, long st, long th, int m) {
    return g->complete_for_next(StreamKey{dev, (const void*)st, (const void*)th}, marks[m]);
}
"""
AFTER_WAIT, AT_ONCE, AT_ONCE_SERIALISED = 0, 1, 2


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    d = tmp_path_factory.mktemp("log")
    src, so = d / "log.cpp", d / "log.so"
    src.write_text(SOURCE)
    subprocess.check_call([os.environ.get("CXX", "g++"), "-std=c++17", "-O1", "-fPIC", "-shared", "-I", b.CSRC, str(src), "-o", str(so)])
    L = ctypes.CDLL(str(so))
    for f in (L.note, L.complete):
        f.argtypes = [ctypes.c_int, ctypes.c_long, ctypes.c_long, ctypes.c_int]
    return L


@pytest.fixture
def log(harness):
    harness.fresh()
    return harness


def test_default_streams_of_two_devices(log):
    # append on 0, append on 1, attention on 0: nothing of that says that device 1's append is complete
    a0 = log.note(0, 0, 0, AT_ONCE)
    a1 = log.note(1, 0, 0, AT_ONCE)
    log.note(0, 0, 0, AFTER_WAIT)
    assert log.complete(0, 0, 0, a0)
    assert not log.complete(1, 0, 0, a1)
    log.note(1, 0, 0, AFTER_WAIT)
    assert log.complete(1, 0, 0, a1)
    assert not log.complete(0, 0, 0, a1)          # another device's stream vouches for nothing


def test_per_thread_default_streams(log):
    a = log.note(0, 2, 100, AFTER_WAIT)
    log.note(0, 2, 200, AFTER_WAIT)
    assert not log.complete(0, 2, 100, a)
    log.note(0, 2, 100, AFTER_WAIT)
    assert log.complete(0, 2, 100, a) and not log.complete(0, 2, 200, a)


def test_chain_of_appends(log):
    first = log.note(0, 7, 0, AFTER_WAIT)
    marks = [log.note(0, 7, 0, AT_ONCE) for _ in range(3)]
    # what the first append's predecessor's successor could count on, and no more
    assert not log.complete(0, 7, 0, first)
    assert not any(log.complete(0, 7, 0, m) for m in marks)
    # an attention launch waits for all before it, and lets its successor go behind that wait
    att = log.note(0, 7, 0, AFTER_WAIT)
    assert all(log.complete(0, 7, 0, m) for m in [first] + marks) and not log.complete(0, 7, 0, att)


def test_append_behind_the_whole_kernel_before(log):
    first = log.note(0, 7, 0, AFTER_WAIT)
    a = log.note(0, 7, 0, AT_ONCE_SERIALISED)
    assert log.complete(0, 7, 0, first) and not log.complete(0, 7, 0, a)


def test_forgotten_streams_vouch_for_nothing(log):
    a = log.note(0, 1, 0, AFTER_WAIT)
    log.note(0, 1, 0, AFTER_WAIT)
    assert log.complete(0, 1, 0, a)
    for s in range(2, 40):
        log.note(0, s, 0, AFTER_WAIT)
    assert not log.complete(0, 1, 0, a)
    log.note(0, 1, 0, AT_ONCE)                    # its slot is new: nothing is known of its predecessor
    assert not log.complete(0, 1, 0, a)
    log.note(0, 1, 0, AFTER_WAIT)
    assert log.complete(0, 1, 0, a)
