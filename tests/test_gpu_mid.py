"""GPU: the tcgen05 kernel with two CTAs per SM at the sizes where it can go wrong: batch rows at the
edges of its 16-row steps, slices that share a tile's rows unevenly or outnumber them, slices inside a cluster (up to
eight) and beyond one (summed by a second kernel), odd unit counts per slice, a 64-column tail tile, several chunks per
CTA, several batch tiles.  Inputs are exactly representable, so every schedule has to give the closed form's bits."""
import numpy as np
import pytest
import torch

import oracle
from paper_2601_16536_b200 import binding as B
from paper_2601_16536_b200 import workloads as wl
from gpu_util import c_bits, ensure_ws, pack_problem, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,K,N,splits", [
    (1, 128, 64, (0, 1)), (16, 1152, 192, (0, 1, 3, 8, 9)), (17, 1408, 128, (0, 2, 5, 8, 11)), (32, 640, 320, (0, 1, 4, 5)),
    (33, 2304, 256, (0, 5, 7, 8)), (48, 1280, 192, (0, 3, 5, 6)), (49, 1024, 448, (0, 4, 8)), (64, 2176, 128, (0, 2, 8, 17)),
    (64, 256, 128 * 300, (0, 1, 2)), (65, 1152, 576, (0, 1, 4, 9)), (300, 512, 128, (0, 3))])
def test_exact_inputs_bit_equal_for_every_schedule(M, K, N, splits):
    d = wl.make_exact_problem(M, K, N, seed=8000 + M)
    want = oracle.gemm_int(d["A_int"], d["Wq"], d["E"], d["Z"], M, N, K, 128)
    pw = pack_problem(d, N, K)
    A = to_dev(d["A"])
    ws = ensure_ws(M, N, K, splits)
    for split_k in splits:
        C = torch.full((M, N), float("nan"), dtype=torch.float16, device="cuda")
        B.w4a16_gemm(A, pw, C=C, split_k=split_k, path=B.PATH_TILE)
        torch.cuda.synchronize()
        assert B.w4a16_device_status() == 0
        assert np.array_equal(c_bits(C), want), "split_k=%d" % split_k
    del ws


@pytest.mark.parametrize("M,K,N,splits,kernel,rows", [
    # batch tiles of 96, 112, 128 rows in the two-CTA kernel (exchange on top of its rings), several of them, a ragged last one
    (96, 640, 21952, (0, 1, 2), B.KERNEL_MID128, 96), (300, 1024, 12288, (0, 2), B.KERNEL_MID128, 112),
    (128, 384, 22016, (0, 3), B.KERNEL_MID128, 128),
    # several batch tiles of the 64-row build
    (128, 1152, 11072, (0, 3), B.KERNEL_MID64, 64), (176, 2048, 3200, (0, 1, 3), B.KERNEL_MID64, 64), (777, 512, 5696, (0, 1, 2), B.KERNEL_MID64, 64),
    # batch tiles of the wide-tile kernel: ragged last ones, whole tiles and slices (balanced chunks: test_gpu_builds.py)
    (470, 1536, 8256, (0, 1, 4), B.KERNEL_TILE, 240), (600, 1024, 8192, (0, 1), B.KERNEL_TILE, 160), (200, 2048, 4224, (0, 1, 3), B.KERNEL_TILE, 208)])
def test_batch_tiles_above_64_rows_bit_equal(M, K, N, splits, kernel, rows):
    for split_k in splits:
        plan = B.w4a16_gemm_plan(M, N, K, split_k=split_k, path=B.PATH_TILE)
        assert (plan.kernel, plan.tile_rows) == (kernel, rows)
    d = wl.make_exact_problem(M, K, N, seed=8100 + M)
    n0 = N - 192        # the last columns: a 64-column tail tile where there is one
    want = oracle.gemm_int(d["A_int"], d["Wq"][:, n0:].copy(), d["E"][:, n0:].copy(), d["Z"][:, n0:].copy(), M, 192, K, 128)
    pw = pack_problem(d, N, K)
    A = to_dev(d["A"])
    ws = ensure_ws(M, N, K, splits)
    first = None
    for split_k in splits:
        C = torch.full((M, N), float("nan"), dtype=torch.float16, device="cuda")
        B.w4a16_gemm(A, pw, C=C, split_k=split_k, path=B.PATH_TILE)
        torch.cuda.synchronize()
        assert B.w4a16_device_status() == 0
        assert np.array_equal(c_bits(C)[:, n0:], want), "split_k=%d" % split_k
        first = C if first is None else first
        assert torch.equal(first, C), "split_k=%d" % split_k
    del ws
