"""GPU: every build of the tcgen05 kernels that a batch of more than 64 rows runs (format, group, epilogue), each way of
summing slices, on shapes for which the plan of the call says that the build is the one that runs.  (Kernel and schedule are
chosen by cost, so a shape alone does not tell.)  Sampled columns, a 64-column tail tile among them, against the oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_2601_16536_b200 import binding as B
from paper_2601_16536_b200 import workloads as wl
from gpu_util import assert_close, ensure_ws
from test_gpu_formats import _assert_close_bf16, _dev16, _f64, _pack

pytestmark = pytest.mark.gpu

WINDOW = 192      # sampled columns at the end: one whole 128-column tile and the tail


def _bias(N, bf16):
    bias32 = np.random.Generator(np.random.PCG64(N)).standard_normal(N).astype(np.float32)
    if bf16:
        bits = (bias32.view(np.uint32) >> 16).astype(np.uint16)
        return bits, (bits.astype(np.uint32) << 16).view(np.float32).astype(np.float64)
    bits = bias32.astype(np.float16).view(np.uint16)
    return bits, bits.view(np.float16).astype(np.float64)


def _check(M, K, N, group, symmetric, bf16, calls):
    """calls: (split_k, bias and SiLU, expected kernel, expected slices, expected cluster)"""
    d = wl.make_problem(M, K, N, seed=M + K + N + group, group=group, symmetric=symmetric, bf16=bf16)
    pw = _pack(d, N, K, group, symmetric, bf16)
    n0 = N - WINDOW
    ref = oracle.gemm(d["A"], d["Wq"][:, n0:].copy(), d["S"][:, n0:].copy(), d["Z"][:, n0:].copy(), M, WINDOW, K, group, bf16=bf16)
    bias_bits, bias = _bias(N, bf16)
    A, bias_dev = _dev16(d["A"], bf16), _dev16(bias_bits, bf16)
    ws = ensure_ws(M, N, K, tuple({c[0] for c in calls}), group)
    for split_k, epi, kernel, slices, cluster in calls:
        plan = B.w4a16_gemm_plan(M, N, K, group, split_k, B.PATH_TILE, epi)
        assert (plan.kernel, plan.split_k, plan.cluster) == (kernel, slices, cluster)
        C = B.w4a16_gemm(A, pw, split_k=split_k, path=B.PATH_TILE, bias=bias_dev if epi else None, act=B.ACT_SILU if epi else B.ACT_NONE)
        torch.cuda.synchronize()
        assert B.w4a16_device_status() == 0
        want = oracle.epilogue(ref, bias[n0:], "silu") if epi else ref
        (_assert_close_bf16 if bf16 else assert_close)(_f64(C)[:, n0:], want, "g%d sym%d bf%d split %d epi%d" % (group, symmetric, bf16, split_k, epi))
    del ws


FORMATS = [(g, s, b) for g in (32, 64, 128) for s in (False, True) for b in (False, True)]


@pytest.mark.parametrize("group,symmetric,bf16", FORMATS)
def test_wide_tiles(group, symmetric, bf16):
    # whole tiles, whose epilogue is the kernel's own, and three slices, whose sum and epilogue are the second kernel's
    T = B.KERNEL_TILE
    _check(777, 1536, 6848, group, symmetric, bf16, [(1, False, T, 1, 0), (1, True, T, 1, 0), (3, False, T, 3, 0), (3, True, T, 3, 0)])


@pytest.mark.parametrize("group,symmetric,bf16", FORMATS)
def test_two_ctas_per_sm_above_64_rows(group, symmetric, bf16):
    # whole tiles, slices in a cluster (exchange on top of the rings), slices beyond one (second kernel)
    D = B.KERNEL_MID128
    _check(96, 1152, 19776, group, symmetric, bf16, [(1, False, D, 1, 0), (1, True, D, 1, 0), (3, True, D, 3, 1), (9, True, D, 9, 0)])


@pytest.mark.parametrize("bf16", [False, True])
def test_balanced_chunks(bf16):
    # chunks of 2.07 tiles of 47 blocks: every tile is shared, the last one by a chunk that ends with the matrix
    T = B.KERNEL_TILE
    _check(129, 6016, 6336, 128, False, bf16, [(0, False, T, 0, 0), (0, True, T, 0, 0)])


@pytest.mark.parametrize("bf16", [False, True])
def test_slices_beyond_a_cluster_with_bias_and_activation(bf16):
    M64 = B.KERNEL_MID64
    _check(40, 1280, 320, 128, False, bf16, [(9, False, M64, 9, 0), (9, True, M64, 9, 0), (1, True, M64, 1, 0)])
