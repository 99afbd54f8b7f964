"""GPU: the tcgen05 kernel for 17 to 64 batch rows (two CTAs per SM) at the sizes where it can go wrong: batch rows at the
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
