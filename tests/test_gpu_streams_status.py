"""GPU: stream ordering of the packed weights, and the bounded-wait status path.

The GEMM kernels may prefetch packed weights before the previous kernel of their stream has
finished (programmatic dependent launch), so the library has to order the first GEMM of a stream
after a w4a16_pack enqueued on that stream.  The status path (a bounded wait that runs out) is
exercised with the library's diagnostic kernel: nothing faults, the context stays usable.
"""
import mmap
import threading

import numpy as np
import pytest
import torch

import oracle
from paper_2601_16536_b200 import binding as B
from paper_2601_16536_b200 import workloads as wl
from gpu_util import assert_close, c_bits, c_f64, ensure_ws, pack_problem, to_dev

pytestmark = pytest.mark.gpu


def test_pack_then_gemm_on_a_side_stream_with_another_stream_in_between():
    # pack on stream A, an unrelated GEMM on stream B, then the GEMM on stream A: the last one must
    # see the packed weights complete although a GEMM was launched elsewhere in between
    M, K, N = 4, 11008, 4096
    d = wl.make_problem(M, K, N, seed=3101)
    other = wl.make_problem(M, 1024, 256, seed=3102)
    ref = oracle.gemm(d["A"], d["Wq"], d["S"], d["Z"], M, N, K, 128)
    ws = ensure_ws(M, N, K, 0)
    pw_other = pack_problem(other, 256, 1024)
    A, A_other = to_dev(d["A"]), to_dev(other["A"])
    raw = [to_dev(d[k]) for k in ("Wq", "S", "Z")]
    torch.cuda.synchronize()
    sa, sb = torch.cuda.Stream(), torch.cuda.Stream()
    first = None
    for rep in range(4):
        with torch.cuda.stream(sa):
            # a long kernel in front so that the pack kernels are still pending when the GEMM is enqueued
            filler = torch.empty(64 << 20, dtype=torch.uint8, device="cuda")
            filler.fill_(rep)
            pw = B.w4a16_pack(raw[0], raw[1], raw[2], N, K)
        with torch.cuda.stream(sb):
            B.w4a16_gemm(A_other, pw_other, split_k=1)
        with torch.cuda.stream(sa):
            C = B.w4a16_gemm(A, pw)
            C2 = B.w4a16_gemm(A, pw)          # the second one may overlap its predecessor again
        torch.cuda.synchronize()
        assert B.w4a16_device_status() == 0
        assert_close(c_f64(C), ref, "first GEMM after pack, rep %d" % rep)
        assert np.array_equal(c_bits(C), c_bits(C2))
        if first is None:
            first = c_bits(C).copy()
        assert np.array_equal(c_bits(C), first)
        del pw, filler
    del ws


def test_pack_then_gemm_on_the_per_thread_stream_with_another_thread_in_between():
    """cudaStreamPerThread names a stream of each thread: a GEMM of another thread under the same handle, between this
    thread's pack and GEMM, must not count as the first one behind the pack."""
    M, K, N, per_thread = 4, 11008, 4096, 2
    probs = [wl.make_problem(M, K, N, seed=3110 + i) for i in range(3)]
    raw = [[to_dev(d[k]) for k in ("Wq", "S", "Z")] for d in probs]
    pw, ws = pack_problem(probs[0], N, K), ensure_ws(M, N, K, 0)
    other = wl.make_problem(M, 1024, 256, seed=3120)
    other_pw, A_other, A = pack_problem(other, 256, 1024), to_dev(other["A"]), [to_dev(d["A"]) for d in probs]
    C, C_other = [torch.empty((M, N), dtype=torch.float16, device="cuda") for _ in probs], torch.empty((M, 256), dtype=torch.float16, device="cuda")
    L, dev = B.load(), torch.cuda.current_device()
    torch.cuda.synchronize()

    def gemm(a, w, c, split_k):
        torch.cuda.set_device(dev)
        assert L.w4a16_gemm(a.data_ptr(), w.Wq.data_ptr(), w.S.data_ptr(), w.Z.data_ptr(), c.data_ptr(), M, w.N, w.K, 128, split_k, per_thread) == 0

    for r, a, c in zip(raw, A, C):
        for _ in range(4):                       # (several, so that the last is still to come when the GEMM is enqueued)
            assert L.w4a16_pack(r[0].data_ptr(), r[1].data_ptr(), r[2].data_ptr(), pw.Wq.data_ptr(), pw.S.data_ptr(), pw.Z.data_ptr(), N, K, 128, per_thread) == 0
        t = threading.Thread(target=gemm, args=(A_other, other_pw, C_other, 1))
        t.start()
        t.join()
        gemm(a, pw, c, 0)
    torch.cuda.synchronize()
    assert B.w4a16_device_status() == 0
    for d, c in zip(probs, C):
        assert_close(c_f64(c), oracle.gemm(d["A"], d["Wq"], d["S"], d["Z"], M, N, K, 128), "per-thread stream")
    del ws


@pytest.mark.parametrize("M", [1, 64, 300])
def test_pack_then_a_captured_gemm_then_gemm_on_the_same_stream(M):
    """The captured GEMM does not run on the stream, so the next one there still is the first behind the pack.  Replayed
    behind another pack, the graph has the new weights."""
    K, N = 4096, 2048
    probs = [wl.make_problem(M, K, N, seed=3130 + i) for i in range(3)]
    raw = [[to_dev(d[k]) for k in ("Wq", "S", "Z")] for d in probs]
    A = to_dev(probs[0]["A"])
    pw, ws, L = pack_problem(probs[0], N, K), ensure_ws(M, N, K, 0), B.load()
    want = []
    for r in raw:
        want.append(c_bits(B.w4a16_gemm(A, B.w4a16_pack(*r, N, K))).copy())
        torch.cuda.synchronize()
    side, graph = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    outs = [torch.empty((M, N), dtype=torch.float16, device="cuda") for _ in range(4)]
    captured = torch.empty((M, N), dtype=torch.float16, device="cuda")
    filler = torch.empty(256 << 20, dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()

    def pack(r):
        filler.fill_(1)                          # the pack is still to come when what is behind it is enqueued
        assert L.w4a16_pack(r[0].data_ptr(), r[1].data_ptr(), r[2].data_ptr(), pw.Wq.data_ptr(), pw.S.data_ptr(), pw.Z.data_ptr(), N, K, 128, side.cuda_stream) == 0

    with torch.cuda.stream(side):
        B.w4a16_gemm(A, pw, C=outs[3])
        pack(raw[1])
        graph.capture_begin()
        B.w4a16_gemm(A, pw, C=captured)
        graph.capture_end()
        B.w4a16_gemm(A, pw, C=outs[0])
        pack(raw[2])
        graph.replay()
        outs[1].copy_(captured)
        B.w4a16_gemm(A, pw, C=outs[2])
    torch.cuda.synchronize()
    assert B.w4a16_device_status() == 0
    for c, w in zip(outs, (want[1], want[2], want[2], want[0])):
        assert np.array_equal(c_bits(c), w)
    del ws


@pytest.mark.parametrize("M", [1, 64, 300])
@pytest.mark.parametrize("side", [False, True])
def test_pack_dequantize_gemm_rows_through_one_set_of_packed_buffers(M, side):
    """Per matrix: pack, dequantization, two GEMMs, and the quantizer on other weights in front of a third, all enqueued without
    a synchronisation into the same buffers.  Each of these lets the next launch start early, so that it is not the GEMM's
    direct predecessor alone that has to have ended before packed words are read."""
    K, N = 4096, 2048
    probs = [wl.make_problem(M, K, N, seed=3140 + i) for i in range(4)]
    raw = [[to_dev(d[k]) for k in ("Wq", "S", "Z")] for d in probs]
    A, W16 = to_dev(probs[0]["A"]), torch.randn(K, N, device="cuda").half()
    ws, want = ensure_ws(M, N, K, 0), []
    for r in raw:
        w = B.w4a16_pack(*r, N, K)
        torch.cuda.synchronize()
        want.append((B.w4a16_dequant(w), B.w4a16_gemm(A, w)))
        torch.cuda.synchronize()
    raw16 = B.w4a16_quantize(W16)
    pw, L = pack_problem(probs[0], N, K), B.load()
    outs = [(torch.empty((K, N), dtype=torch.float16, device="cuda"),
             [torch.empty((M, N), dtype=torch.float16, device="cuda") for _ in range(3)]) for _ in raw]
    torch.cuda.synchronize()
    stream = torch.cuda.Stream() if side else torch.cuda.current_stream()
    with torch.cuda.stream(stream):
        st = stream.cuda_stream
        for r, (w16, c) in zip(raw, outs):
            assert L.w4a16_pack(r[0].data_ptr(), r[1].data_ptr(), r[2].data_ptr(), pw.Wq.data_ptr(), pw.S.data_ptr(), pw.Z.data_ptr(), N, K, 128, st) == 0
            B.w4a16_dequant(pw, out=w16)
            B.w4a16_gemm(A, pw, C=c[0])
            B.w4a16_gemm(A, pw, C=c[1])
            assert L.w4a16_quantize(W16.data_ptr(), raw16[0].data_ptr(), raw16[1].data_ptr(), raw16[2].data_ptr(), N, K, 128, 0, st) == 0
            B.w4a16_gemm(A, pw, C=c[2])
    torch.cuda.synchronize()
    assert B.w4a16_device_status() == 0
    for (w16, c), (gw16, gc) in zip(want, outs):
        assert torch.equal(w16, gw16) and all(torch.equal(c, g) for g in gc)
    for a, b in zip(raw16, B.w4a16_quantize(W16)):
        assert torch.equal(a, b)
    del ws


@pytest.mark.parametrize("path,M", [(B.PATH_DECODE, 8), (B.PATH_TILE, 32)])
def test_gemm_on_a_non_default_stream_matches_the_default_stream(path, M):
    K, N = 2304, 512
    d = wl.make_problem(M, K, N, seed=3200 + M)
    pw = pack_problem(d, N, K)
    A = to_dev(d["A"])
    ws = ensure_ws(M, N, K, (0, 3))
    want = B.w4a16_gemm(A, pw, split_k=3, path=path)
    torch.cuda.synchronize()
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        got = [B.w4a16_gemm(A, pw, split_k=3, path=path) for _ in range(3)]
    torch.cuda.synchronize()
    assert B.w4a16_device_status() == 0
    for g in got:
        assert np.array_equal(c_bits(g), c_bits(want))
    assert_close(c_f64(want), oracle.gemm(d["A"], d["Wq"], d["S"], d["Z"], M, N, K, 128), "stream")
    del ws


@pytest.mark.parametrize("M,K,N", [(3, 256, 256), (16, 1152, 1152), (200, 11008, 256)])
def test_host_buffer_calls_are_ordered_on_their_stream(M, K, N):
    """Pinned activations staged by a kernel (up to 4 MiB) and by the copy engine: one staging buffer shared by calls that
    follow each other, and, where K = N, a result buffer that is the next call's activations."""
    d = wl.make_problem(M, K, N, seed=3400 + M)
    ws = ensure_ws(M, N, K, 0)
    raw = [to_dev(d[k]) for k in ("Wq", "S", "Z")]
    A2 = wl.draw_activations(M, K, 3401)
    hosts = [torch.from_numpy(a.view(np.float16)).pin_memory() for a in (d["A"], A2)]
    outs = [torch.zeros((M, N), dtype=torch.float16).pin_memory() for _ in range(3)]
    A_dev = torch.empty((M, K), dtype=torch.float16, device="cuda")
    C_dev = torch.empty((M, N), dtype=torch.float16, device="cuda")
    torch.cuda.synchronize()
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        for _ in range(3):
            pw = B.w4a16_pack(raw[0], raw[1], raw[2], N, K)       # the first call behind a pack must see it complete
            B.w4a16_gemm_host(hosts[0], A_dev, pw, C_dev, outs[0])
            B.w4a16_gemm_host(hosts[1], A_dev, pw, C_dev, outs[1])
            if K == N:
                B.w4a16_gemm_host(outs[1], A_dev, pw, C_dev, outs[2])
    torch.cuda.synchronize()
    assert B.w4a16_device_status() == 0
    for host, out in zip(hosts, outs):
        assert np.array_equal(out.numpy().view(np.uint16), c_bits(B.w4a16_gemm(host.cuda(), pw)))
    if K == N:
        assert np.array_equal(outs[2].numpy().view(np.uint16), c_bits(B.w4a16_gemm(outs[1].cuda(), pw)))
    del ws


@pytest.mark.parametrize("which", ["A", "C"])
def test_host_buffer_that_is_page_locked_in_part_is_refused(which):
    """Only the first page of the buffer is registered: no kernel may touch it by its address.  The copy engine refuses such
    a buffer; with its second part registered too, every byte is reachable and the call works."""
    M, K, N = 4, 1152, 1088                      # 9,216 and 8,704 bytes: three pages each
    d = wl.make_problem(M, K, N, seed=3400)
    pw = pack_problem(d, N, K)
    A = to_dev(d["A"])
    ws = ensure_ws(M, N, K, 0)
    want = c_bits(B.w4a16_gemm(A, pw)).copy()
    page = mmap.PAGESIZE
    memory = mmap.mmap(-1, 3 * page)
    cols, bits = (K, d["A"]) if which == "A" else (N, None)
    buf = torch.frombuffer(memory, dtype=torch.float16)[:M * cols].view(M, cols)
    A_host = torch.from_numpy(d["A"].view(np.float16)).pin_memory()
    C_host = torch.zeros((M, N), dtype=torch.float16).pin_memory()
    if bits is not None:
        buf.copy_(A_host)
        A_host = buf
    else:
        C_host = buf
    A_dev, C_dev = torch.empty((M, K), dtype=torch.float16, device="cuda"), torch.empty((M, N), dtype=torch.float16, device="cuda")
    rt, base = torch.cuda.cudart(), buf.data_ptr()
    assert base % page == 0
    assert int(rt.cudaHostRegister(base, page, 0)) == 0
    try:
        with pytest.raises(B.W4A16Error) as e:
            B.w4a16_gemm_host(A_host, A_dev, pw, C_dev, C_host)
        assert e.value.code == -6
        torch.cuda.synchronize()
        assert int(rt.cudaHostRegister(base + page, 2 * page, 0)) == 0
        try:
            B.w4a16_gemm_host(A_host, A_dev, pw, C_dev, C_host)
            torch.cuda.synchronize()
            assert B.w4a16_device_status() == 0
            assert np.array_equal(C_host.numpy().view(np.uint16), want)
        finally:
            rt.cudaHostUnregister(base + page)
    finally:
        rt.cudaHostUnregister(base)
    del ws


def test_a_wait_that_runs_out_is_reported_and_the_library_keeps_working():
    M, K, N = 8, 1152, 256
    d = wl.make_problem(M, K, N, seed=3300)
    pw = pack_problem(d, N, K)
    A = to_dev(d["A"])
    ws = ensure_ws(M, N, K, 3)
    before = c_bits(B.w4a16_gemm(A, pw, split_k=3, path=B.PATH_DECODE)).copy()
    torch.cuda.synchronize()
    assert B.w4a16_device_status() == 0
    B.w4a16_selftest_wait_timeout(1000)          # a barrier nobody arrives on, 1 ms limit
    torch.cuda.synchronize()                     # the kernel returned by itself
    assert B.w4a16_device_status() == 1          # bit 0: a barrier wait ran out ...
    assert B.w4a16_device_status() == 0          # ... and reading the word cleared it
    # the workspace (whose ticket counters the status call re-zeroed) and both kernels still work
    after = c_bits(B.w4a16_gemm(A, pw, split_k=3, path=B.PATH_DECODE))
    assert np.array_equal(before, after)
    tile = B.w4a16_gemm(A, pw, split_k=3, path=B.PATH_TILE)
    torch.cuda.synchronize()
    assert B.w4a16_device_status() == 0
    assert_close(c_f64(tile), oracle.gemm(d["A"], d["Wq"], d["S"], d["Z"], M, N, K, 128), "after timeout")
    with pytest.raises(B.W4A16Error):
        B.w4a16_selftest_wait_timeout(0)
    del ws
