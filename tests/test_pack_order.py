"""The rule that orders GEMM launches behind packs (csrc/pack_order.cuh: host code without CUDA calls), compiled with the host
compiler and driven through a small C interface."""
import ctypes
import os
import subprocess
import threading

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2601_16536_b200", "csrc")
DRIVER = r"""
#include "pack_order.cuh"
using w4a16::PackOrder;
extern "C" {
void* order_new() { return new PackOrder; }
void order_delete(void* o) { delete static_cast<PackOrder*>(o); }
void order_pack(void* o) { static_cast<PackOrder*>(o)->pack_issued(); }
int order_may_release(unsigned long long capture) { return PackOrder::may_release(capture); }
// returns whether the launch was allowed to overlap; `accepted`: whether it got onto the stream
int order_launch(void* o, unsigned long long stream, unsigned long long capture, int accepted) {
    bool overlapped = false;
    static_cast<PackOrder*>(o)->launch((uintptr_t)stream, [&] { return capture; }, [&](bool overlap) { overlapped = overlap; return accepted != 0; });
    return overlapped ? 1 : 0;
}
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("pack_order")
    src, so = str(d / "driver.cpp"), str(d / "driver.so")
    with open(src, "w") as f:
        f.write(DRIVER)
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-Wall", "-Werror", "-shared", "-fPIC", "-I", CSRC, "-o", so, src])
    L = ctypes.CDLL(so)
    L.order_new.restype = ctypes.c_void_p
    L.order_delete.argtypes = L.order_pack.argtypes = [ctypes.c_void_p]
    L.order_may_release.argtypes = [ctypes.c_ulonglong]
    L.order_launch.argtypes = [ctypes.c_void_p, ctypes.c_ulonglong, ctypes.c_ulonglong, ctypes.c_int]
    return L


class Order:
    def __init__(self, L):
        self.L, self.o = L, L.order_new()

    def __del__(self):
        self.L.order_delete(self.o)

    def pack(self):
        self.L.order_pack(self.o)

    def gemm(self, stream, accepted=True, capture=0):
        return "overlapped" if self.L.order_launch(self.o, stream, capture, int(accepted)) else "plain"


A, B = 0x5000, 0x6000


def test_the_first_gemm_of_every_stream_behind_a_pack_is_plain(lib):
    o = Order(lib)
    assert [o.gemm(A), o.gemm(A), o.gemm(0), o.gemm(0)] == ["plain", "overlapped"] * 2
    o.pack()
    assert [o.gemm(B), o.gemm(B), o.gemm(A), o.gemm(A), o.gemm(0), o.gemm(0)] == ["plain", "overlapped"] * 3


def test_streams_without_a_slot_are_plain(lib):
    o = Order(lib)
    for s in range(1, 41):                               # eight more than there are slots: the first eight are evicted
        assert o.gemm(s) == "plain"
    assert [o.gemm(40), o.gemm(9), o.gemm(1)] == ["overlapped", "overlapped", "plain"]


def test_a_refused_launch_orders_nothing(lib):
    """Pack, a launch that the device refuses (a cluster that it cannot place, say), and the retry: the retry stands directly
    behind the pack."""
    o = Order(lib)
    o.gemm(A)
    o.pack()
    assert [o.gemm(A, accepted=False), o.gemm(A, accepted=False), o.gemm(A), o.gemm(A)] == ["plain", "plain", "plain", "overlapped"]
    # one that is refused where overlap was allowed takes nothing away
    assert [o.gemm(A, accepted=False), o.gemm(A)] == ["overlapped", "overlapped"]


def test_the_per_thread_handle_is_a_stream_of_each_thread(lib):
    """A GEMM on another thread's stream of the same handle stands behind nothing of this thread's."""
    per_thread, o = 2, Order(lib)

    def on_another_thread(f):
        got = []
        t = threading.Thread(target=lambda: got.append(f()))
        t.start()
        t.join()
        return got[0]

    assert [o.gemm(per_thread), o.gemm(per_thread)] == ["plain", "overlapped"]
    o.pack()
    assert on_another_thread(lambda: [o.gemm(per_thread), o.gemm(per_thread)]) == ["plain", "overlapped"]
    assert [o.gemm(per_thread), o.gemm(per_thread)] == ["plain", "overlapped"]


def test_a_captured_gemm_orders_nothing_on_its_stream(lib):
    """Pack on a stream, a GEMM captured from that stream into a graph that is not replayed, then a GEMM on the stream: the
    last one stands directly behind the pack."""
    o = Order(lib)
    assert [o.gemm(A), o.gemm(A)] == ["plain", "overlapped"]
    o.pack()
    assert [o.gemm(A, capture=7), o.gemm(A, capture=7)] == ["plain", "overlapped"]
    assert [o.gemm(A, capture=8), o.gemm(A, capture=8)] == ["plain", "overlapped"]
    assert [o.gemm(A), o.gemm(A)] == ["plain", "overlapped"]
    assert o.gemm(A, capture=9) == "overlapped"          # no pack since the stream's last GEMM, hence none in this capture
    o.pack()                                             # captured or not
    assert [o.gemm(A, capture=8), o.gemm(A)] == ["plain", "plain"]


def test_a_pack_in_a_graph_releases_nothing(lib):
    """A replay is no call of the library: a GEMM behind one goes by what was launched before."""
    assert lib.order_may_release(0) and not lib.order_may_release(7)
    o = Order(lib)
    o.pack()                                             # captured
    assert [o.gemm(A), o.gemm(A)] == ["plain", "overlapped"]   # ... and the second may stand directly behind a replay
