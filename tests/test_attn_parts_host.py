"""Into how many runs the attention products cut an item: the same as from trying every cut, in far fewer steps. On the CPU."""
import ctypes
import os
import subprocess

import pytest

HEADER = os.path.join(os.path.dirname(os.path.abspath(__file__)), "..", "paper_2312_05693_b200", "csrc", "aq_attn_parts.cuh")
SOURCE = """
#include "%s"
#include <chrono>
// every cut
static int all_cuts(long items, int tiles, int sms) {
    int best = 1;
    long least = (items + sms - 1) / sms * tiles;
    for (int p = 2; p <= tiles && items * p <= 0x7FFFFFFFl; ++p) {
        const int per = (tiles + p - 1) / p;
        if ((p - 1) * (long)per >= tiles) continue;          // the last run would be empty
        const long most = (items * p + sms - 1) / sms * per;
        if (most < least) { least = most; best = p; }
    }
    return best;
}
extern "C" int parts(long items, int tiles, int sms) { return aq::attn_parts(items, tiles, sms); }
extern "C" int every(long items, int tiles, int sms) { return all_cuts(items, tiles, sms); }
extern "C" double nanoseconds(int which, int tiles, int sms) {
    double best = 1e30;
    for (int rep = 0; rep < 20; ++rep) {
        const auto t = std::chrono::steady_clock::now();
        volatile int sum = 0;
        for (long items = 1; items <= 200; ++items) sum = sum + (which ? all_cuts(items, tiles, sms) : aq::attn_parts(items, tiles, sms));
        const double ns = std::chrono::duration<double, std::nano>(std::chrono::steady_clock::now() - t).count() / 200;
        if (ns < best) best = ns;
    }
    return best;
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("parts")
    src, out = d / "parts.cpp", d / "parts.so"
    src.write_text(SOURCE % os.path.abspath(HEADER))
    subprocess.check_call([os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-shared", "-fPIC", str(src), "-o", str(out)])
    lib = ctypes.CDLL(str(out))
    for f in (lib.parts, lib.every):
        f.argtypes = [ctypes.c_long, ctypes.c_int, ctypes.c_int]
    lib.nanoseconds.restype = ctypes.c_double
    return lib


def test_the_cuts_are_those_of_trying_all(lib):
    for sms in (1, 7, 132, 148, 160):
        for tiles in [*range(1, 40), 63, 64, 65, 127, 512, 1000]:
            for items in [*range(1, 30), 31, 32, 147, 148, 149, 256, 295, 297, 512, 4096, 65535]:
                assert lib.parts(items, tiles, sms) == lib.every(items, tiles, sms), (items, tiles, sms)
    for items, tiles in [(65535, 65535), (2**31 - 1, 2), (2**30, 3), (1, 65535), (16384, 65535)]:      # as far as the sizes go
        assert lib.parts(items, tiles, 148) == lib.every(items, tiles, 148)


def test_a_call_with_many_keys_does_not_pay_for_its_tiles(lib):
    assert lib.nanoseconds(0, 65535, 148) < lib.nanoseconds(1, 65535, 148) / 8
