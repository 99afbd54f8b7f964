"""GPU: the quantizer of Eq. 1 through the C ABI, bit for bit against the oracle (codes, scales and zero
points are integers / bit patterns decided in binary32 on both sides), and the whole chain
quantize -> pack -> GEMM against the oracle's product of the weights it quantized."""
import numpy as np
import pytest
import torch

import oracle
from paper_2601_16536_b200 import binding as B
from paper_2601_16536_b200 import workloads as wl
from gpu_util import assert_close, ensure_ws

pytestmark = pytest.mark.gpu


def _weights(K, N, seed, bf16):
    r = np.random.Generator(np.random.PCG64([seed, 9]))
    x = (r.standard_normal((K, N)) * 0.04).astype(np.float32)
    x[::97, ::5] *= 6.0                                   # a few outliers per group
    x[128:256, 3] = 0.0                                   # a group of zeros
    x[256:384, 4] = 0.0123                                # a constant group
    return wl._bits16(x, bf16)


@pytest.mark.parametrize("group", [32, 64, 128])
@pytest.mark.parametrize("symmetric", [False, True])
@pytest.mark.parametrize("bf16", [False, True])
def test_quantize_is_bit_exact(group, symmetric, bf16):
    K, N = 512, 192
    bits = _weights(K, N, group + symmetric, bf16)
    flags = (B.FLAG_SYMMETRIC if symmetric else 0) | (B.FLAG_BF16 if bf16 else 0)
    W = torch.from_numpy(bits.view(np.int16)).cuda().view(torch.bfloat16 if bf16 else torch.float16)
    Wq, S, Z = B.w4a16_quantize(W, group, flags)
    torch.cuda.synchronize()
    wq, s, z = oracle.quantize(bits, K, N, group, symmetric=symmetric, bf16=bf16)
    assert np.array_equal(Wq.cpu().numpy().view(np.uint32), wq)
    assert np.array_equal(S.view(torch.int16).cpu().numpy().view(np.uint16), s)
    if symmetric:
        assert Z is None and np.all(z == 8)
    else:
        assert np.array_equal(Z.cpu().numpy(), z)


@pytest.mark.parametrize("group", [32, 128])
@pytest.mark.parametrize("symmetric", [False, True])
@pytest.mark.parametrize("bf16", [False, True])
def test_quantize_is_bit_exact_on_ties_and_extreme_scales(group, symmetric, bf16):
    """Quotients that are exact half-integers (weights k/2 times a short scale), groups far from zero (every quotient
    large), and column magnitudes from the format's subnormals to its largest numbers: the integers still are the ones
    of the definition's binary32 division."""
    K, N = 256, 128
    r = np.random.Generator(np.random.PCG64([group, 21]))
    x = (r.integers(-15, 16, size=(K, N)) * 0.5 * 2.0 ** r.integers(-6, 3, size=(1, N))).astype(np.float64)
    x[:, 1::4] = r.standard_normal((K, N // 4)) * 1e-3 + 100.0
    x[:, 2::4] = r.standard_normal((K, N // 4)) * 2.0 ** np.linspace(-120 if bf16 else -23, 100 if bf16 else 11, N // 4)
    x[:, 3::4] = r.integers(-255, 256, size=(K, N // 4)) * 0.125
    bits = wl._bits16(x.astype(np.float32), bf16)
    flags = (B.FLAG_SYMMETRIC if symmetric else 0) | (B.FLAG_BF16 if bf16 else 0)
    W = torch.from_numpy(bits.view(np.int16)).cuda().view(torch.bfloat16 if bf16 else torch.float16)
    Wq, S, Z = B.w4a16_quantize(W, group, flags)
    torch.cuda.synchronize()
    wq, s, z = oracle.quantize(bits, K, N, group, symmetric=symmetric, bf16=bf16)
    assert np.array_equal(Wq.cpu().numpy().view(np.uint32), wq)
    assert np.array_equal(S.view(torch.int16).cpu().numpy().view(np.uint16), s)
    assert symmetric or np.array_equal(Z.cpu().numpy(), z)


@pytest.mark.parametrize("group", [32, 64, 128])
@pytest.mark.parametrize("symmetric", [False, True])
@pytest.mark.parametrize("bf16", [False, True])
def test_quantize_infinities_and_nans(group, symmetric, bf16):
    """A group with an infinity has scale 1 (the definition's rule for a scale that is not finite), the infinities codes 15 and
    0.  A NaN takes no part in a group's minimum and maximum and gets code 0; what is beside it has the codes it would have
    without it (the oracle, whose conversion of a NaN to an integer is not defined, gets another number of the group in its
    place)."""
    K, N = 256, 128
    r = np.random.Generator(np.random.PCG64([group, 31]))
    x = (r.standard_normal((K, N)) * 2.0 ** r.integers(-9, 3, size=(1, N))).astype(np.float32)
    x[r.random((K, N)) < 0.02] = np.inf
    x[r.random((K, N)) < 0.02] = -np.inf
    x[:, 5] = np.inf
    x[:, 6] = -np.inf
    x[:, 7] = np.where(r.random(K) < 0.5, np.inf, -np.inf)
    x[:, 64:] = np.where(np.isinf(x[:, 64:]), np.float32(0.5), x[:, 64:])          # the second tile: NaN only
    bits = wl._bits16(x, bf16)
    exp = 0x7F80 if bf16 else 0x7C00
    nan = r.random((K, N)) < 0.05
    nan[:group, 9] = True                                                          # a group of nothing else
    nan[:, 10] = np.arange(K) % group != 3                                         # one number a group
    poisoned = bits.copy()
    poisoned[nan] = r.choice(np.array([exp | 1, exp | 0x40, exp | 0x8001, 0xFFFF], dtype=np.uint16), size=int(nan.sum()))
    # oracle's weights: in place of a NaN a number that its group has anyway, or, in a group of NaN alone, 0: there scale 1 and
    # zero point 0 are what the definition gives for the empty minimum and maximum (+inf, -inf) and for zeros alike
    clean = bits.copy()
    for g in range(K // group):
        rows = slice(g * group, (g + 1) * group)
        for n in range(N):
            bad = nan[rows, n]
            clean[rows, n][bad] = 0 if bad.all() else bits[rows, n][~bad][0]
    flags = (B.FLAG_SYMMETRIC if symmetric else 0) | (B.FLAG_BF16 if bf16 else 0)
    W = torch.from_numpy(poisoned.view(np.int16)).cuda().view(torch.bfloat16 if bf16 else torch.float16)
    Wq, S, Z = B.w4a16_quantize(W, group, flags)
    torch.cuda.synchronize()
    wq, s, z = oracle.quantize(clean, K, N, group, symmetric=symmetric, bf16=bf16)
    assert np.array_equal(S.view(torch.int16).cpu().numpy().view(np.uint16), s)
    assert symmetric or np.array_equal(Z.cpu().numpy(), z)
    want = oracle.unpack(wq, K, N)
    want[nan] = 0
    assert np.array_equal(oracle.unpack(Wq.cpu().numpy().view(np.uint32), K, N), want)


@pytest.mark.parametrize("M,symmetric", [(4, False), (4, True), (48, False)])
def test_quantize_pack_gemm_chain(M, symmetric):
    K, N, group = 2048, 512, 128
    bits = _weights(K, N, 5, False)
    flags = B.FLAG_SYMMETRIC if symmetric else 0
    W = torch.from_numpy(bits.view(np.float16)).cuda()
    Wq, S, Z = B.w4a16_quantize(W, group, flags)
    pw = B.w4a16_pack(Wq, S, Z, N, K, group, flags)
    A_bits = wl.draw_activations(M, K, 17)
    ws = ensure_ws(M, N, K, 0)
    C = B.w4a16_gemm(torch.from_numpy(A_bits.view(np.float16)).cuda(), pw)
    torch.cuda.synchronize()
    assert B.w4a16_device_status() == 0
    wq, s, z = oracle.quantize(bits, K, N, group, symmetric=symmetric)
    ref = oracle.gemm(A_bits, wq, s, z, M, N, K, group)
    assert_close(C.cpu().numpy().astype(np.float64), ref, "chain M%d sym%d" % (M, symmetric))
    # and the quantized product stays close to the product with the original FP16 weights (4-bit error)
    full = A_bits.view(np.float16).astype(np.float64) @ bits.view(np.float16).astype(np.float64)
    assert np.linalg.norm(ref - full) / np.linalg.norm(full) < 0.2
    del ws


@pytest.mark.parametrize("K,N", [(128, 64), (1024, 960), (4096, 4096)])
def test_a_row_of_quantize_and_pack_calls_is_ordered(K, N):
    """Eight matrices through one set of raw buffers without a synchronisation in between: each launch is set up while the
    one in front of it runs, so a pack that read too early, or a quantizer that wrote too early, would mix two matrices."""
    Ws = [(torch.randn(K, N, device="cuda") * 0.04 * (1 + i)).half() for i in range(8)]
    Wq = torch.empty((K // 8, N), dtype=torch.int32, device="cuda")
    S = torch.empty((K // 128, N), dtype=torch.float16, device="cuda")
    Z = torch.empty((K // 128, N), dtype=torch.uint8, device="cuda")
    L, st = B.load(), torch.cuda.current_stream().cuda_stream
    packed = []
    for W in Ws:
        assert L.w4a16_quantize(W.data_ptr(), Wq.data_ptr(), S.data_ptr(), Z.data_ptr(), N, K, 128, 0, st) == 0
        packed.append(B.w4a16_pack(Wq, S, Z, N, K))
    torch.cuda.synchronize()
    for W, pw in zip(Ws, packed):
        q, s, z = B.w4a16_quantize(W)
        torch.cuda.synchronize()
        one = B.w4a16_pack(q, s, z, N, K)
        torch.cuda.synchronize()
        assert torch.equal(pw.Wq, one.Wq) and torch.equal(pw.S, one.S) and torch.equal(pw.Z, one.Z)


@pytest.mark.parametrize("M", [1, 64, 300])
def test_quantize_pack_dequantize_in_a_graph_in_front_of_gemms(M):
    """The three kernels captured and replayed on new weights, with two GEMMs on the stream behind every replay: what they
    request early is what the replay has packed."""
    K, N = 2048, 1024
    Ws = [(torch.randn(K, N, device="cuda") * 0.04 * (1 + i)).half() for i in range(4)]
    W, A = Ws[0].clone(), torch.randn(M, K, device="cuda").half()
    ws, want = ensure_ws(M, N, K, 0), []
    for w in Ws:
        pw = B.w4a16_pack(*B.w4a16_quantize(w), N, K)
        torch.cuda.synchronize()
        want.append((B.w4a16_dequant(pw), B.w4a16_gemm(A, pw)))
        torch.cuda.synchronize()
    L, side, graph = B.load(), torch.cuda.Stream(), torch.cuda.CUDAGraph()
    Wq, S, Z = B.w4a16_quantize(W)
    pw = B.w4a16_pack(Wq, S, Z, N, K)
    W16 = torch.empty((K, N), dtype=torch.float16, device="cuda")
    got = [(torch.empty_like(W16), *(torch.empty((M, N), dtype=torch.float16, device="cuda") for _ in range(2))) for _ in Ws]
    torch.cuda.synchronize()
    with torch.cuda.stream(side):
        graph.capture_begin()
        st = side.cuda_stream
        assert L.w4a16_quantize(W.data_ptr(), Wq.data_ptr(), S.data_ptr(), Z.data_ptr(), N, K, 128, 0, st) == 0
        assert L.w4a16_pack(Wq.data_ptr(), S.data_ptr(), Z.data_ptr(), pw.Wq.data_ptr(), pw.S.data_ptr(), pw.Z.data_ptr(), N, K, 128, st) == 0
        B.w4a16_dequant(pw, out=W16)
        graph.capture_end()
        for w, (d, c0, c1) in zip(Ws, got):
            W.copy_(w)
            graph.replay()
            B.w4a16_gemm(A, pw, C=c0)
            B.w4a16_gemm(A, pw, C=c1)
            d.copy_(W16)
    torch.cuda.synchronize()
    assert B.w4a16_device_status() == 0
    for (d, c), (gd, g0, g1) in zip(want, got):
        assert torch.equal(d, gd) and torch.equal(c, g0) and torch.equal(c, g1)
    del ws
