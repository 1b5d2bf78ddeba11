"""What the library sets up once per device context (csrc/per_device.h), compiled for the
host: every device gets its own set-up, a failed one is tried again, a recreated context gets
a new one, and threads that arrive together make it once."""

import ctypes
import os
import re
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2607_28699_gb300", "csrc")
SOURCE = r"""
#include <atomic>
#include <thread>
#include <vector>
#include "per_device.h"

static wc::PerDevice<int> state;
static std::atomic<int> made{0};

extern "C" int get(int device, long context, int value, int fail, int* out) {
    return state.get(device, reinterpret_cast<void*>(context), *out, [&](int& v) {
        ++made;
        if (fail) return fail;
        v = value;
        return 0;
    });
}
extern "C" int times_made() { return made; }
extern "C" int together(int threads) {
    static wc::PerDevice<int> shared;
    std::atomic<int> runs{0}, wrong{0};
    std::vector<std::thread> all;
    for (int t = 0; t < threads; ++t)
        all.emplace_back([&] {
            int v = 0;
            if (shared.get(3, &shared, v, [&](int& x) { ++runs; x = 17; return 0; }) != 0 || v != 17) ++wrong;
        });
    for (auto& t : all) t.join();
    return wrong ? -1 : (int)runs;
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("per_device")
    (d / "t.cpp").write_text(SOURCE)
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-pthread", f"-I{CSRC}", "-o", str(d / "t.so"),
                    str(d / "t.cpp")], check=True)
    return ctypes.CDLL(str(d / "t.so"))


def _get(lib, device, context, value, fail=0):
    out = ctypes.c_int(0)
    st = lib.get(device, ctypes.c_long(context), value, fail, ctypes.byref(out))
    return st, out.value


def test_each_device_context_is_set_up_once(lib):
    n = lib.times_made()
    assert _get(lib, 0, 100, 5) == (0, 5) and _get(lib, 0, 100, 6) == (0, 5)     # the second finds the first
    assert _get(lib, 1, 200, 7) == (0, 7)                                        # another device: its own
    assert _get(lib, 2, 300, 8, fail=9)[0] == 9 and _get(lib, 2, 300, 8) == (0, 8)   # an error is tried again
    assert lib.times_made() == n + 4
    assert _get(lib, 0, 101, 10) == (0, 10) and _get(lib, 0, 101, 11) == (0, 10)     # a recreated context
    assert _get(lib, 64, 100, 12) == (0, 12) and _get(lib, 64, 100, 13) == (0, 13)   # past the table: each time
    assert _get(lib, 3, 0, 14) == (0, 14) and _get(lib, 3, 0, 15) == (0, 15)         # no context yet: each time
    assert lib.times_made() == n + 9


def test_threads_make_it_once(lib):
    assert lib.together(16) == 1


def test_no_launch_sets_attributes_once_per_process():
    for f in sorted(os.listdir(CSRC)):
        src = open(os.path.join(CSRC, f)).read()
        assert not re.search(r"static bool \w+ = false", src), f
