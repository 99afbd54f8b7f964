"""The C-ABI library loads, exports every symbol include/w4a16.h declares, and validates
arguments on the host before touching a device (no compute calls here)."""
import ctypes
import os
import random
import re

import pytest

from paper_2601_16536_b200 import binding as B
from paper_2601_16536_b200 import build as libbuild

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def lib():
    libbuild.build_library()
    return B.load()


def _declared():
    text = open(os.path.join(ROOT, "include", "w4a16.h")).read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    return sorted(set(re.findall(r"\b(w4a16_[a-z0-9_]+)\s*\(", text)))


def test_every_declared_symbol_is_exported(lib):
    names = _declared()
    assert len(names) >= 12
    for n in names:
        assert hasattr(lib, n), n
    assert set(names) == set(B.EXPORTS)


def test_packed_sizes_hold_exactly_the_raw_information(lib):
    for N, K in [(64, 128), (4096, 4096), (4096, 11008), (8192, 28672), (22016, 4096)]:
        assert lib.w4a16_packed_wq_bytes(N, K, 128) == K * N // 2
        assert lib.w4a16_packed_s_bytes(N, K, 128) == (K // 128) * N * 2
        assert lib.w4a16_packed_z_bytes(N, K, 128) == (K // 128) * N // 2
    # unsupported shapes report size 0
    assert lib.w4a16_packed_wq_bytes(100, 4096, 128) == 0
    assert lib.w4a16_packed_wq_bytes(4096, 4000, 128) == 0
    assert lib.w4a16_packed_wq_bytes(4096, 4096, 48) == 0
    # smaller quantization groups: the same nibbles, proportionally more scales and zero points
    for group in (32, 64):
        assert lib.w4a16_packed_wq_bytes(4096, 4096, group) == 4096 * 4096 // 2
        assert lib.w4a16_packed_s_bytes(4096, 4096, group) == (4096 // group) * 4096 * 2
        assert lib.w4a16_packed_z_bytes(4096, 4096, group) == (4096 // group) * 4096 // 2


def test_choose_split_k_is_always_acceptable(lib):
    for M in (1, 2, 4, 8, 16, 32, 64, 256, 1024, 4096):
        for N, K in [(4096, 4096), (4096, 11008), (8192, 28672), (12288, 4096), (22016, 4096),
                     (8192, 8192), (64, 128), (64, 256)]:
            s = lib.w4a16_choose_split_k(M, N, K, 128)
            assert 1 <= s <= K // 128
            for path in (1, 2, 3):
                s = lib.w4a16_choose_split_k_ex(M, N, K, 128, path)
                assert 1 <= s <= K // 128
            # automatic scheduling shares column tiles between CTAs, so it needs partial-tile slots
            assert lib.w4a16_workspace_bytes(M, N, K, 128, 0) >= 16384
            assert lib.w4a16_workspace_bytes(M, N, K, 128, 1) == 0
    assert lib.w4a16_workspace_bytes(4, 4096, 4096, 128, 1) == 0
    assert lib.w4a16_workspace_bytes(4, 4096, 4096, 128, 4) >= 4 * 4 * 4096 * 4


def test_schedule_queries_are_consistent_on_a_grid_of_shapes(lib):
    """Host logic over 675 (M, N, K, group) combinations, none of them tuned for: the path is one of the two
    GEMM kernels, the reported split is one w4a16_gemm accepts (1 .. K/128 for every group size), a split of
    1 needs no workspace, any other split needs at least the ticket header, and the size is bounded by the
    partial tiles the schedule can produce (two per CTA slot of a 148-SM device, per batch chunk)."""
    header = 16384 + 131072
    n = 0
    for group in (32, 64, 128):
        for M in (1, 3, 8, 9, 16, 17, 64, 300, 4096):
            for N in (64, 1536, 4096, 4608, 22016):
                for K in (128, 1024, 4096, 11008, 28672):
                    n += 1
                    blocks = K // 128
                    assert lib.w4a16_choose_path(M, N, K, group) in (2, 3)
                    s = lib.w4a16_choose_split_k(M, N, K, group)
                    assert 1 <= s <= blocks, (M, N, K, group, s)
                    for path in (1, 2, 3):
                        assert 1 <= lib.w4a16_choose_split_k_ex(M, N, K, group, path) <= blocks
                    assert lib.w4a16_workspace_bytes(M, N, K, group, 1) == 0
                    assert lib.w4a16_workspace_bytes(M, N, K, group, blocks + 1) == 0      # not a valid split
                    for split in {0, s, min(2, blocks), blocks}:
                        if split == 1:
                            continue
                        need = lib.w4a16_workspace_bytes(M, N, K, group, split)
                        assert need == 0 or need >= header
                        # plain path: split x M x N floats; warp-MMA path: two 16 x 64 tiles per chunk and batch
                        # chunk; tcgen05 path: two MT x 128 tiles per chunk
                        sp = split if split else max(s, 1)
                        bound = header + 256 + max(4 * sp * M * N,
                                                   2 * max(296, (N // 64) * sp) * ((M + 15) // 16) * 16 * 64 * 4,
                                                   2 * max(148, ((M + 15) // 16) * ((N + 127) // 128) * sp) * 256 * 128 * 4)
                        assert need <= bound, (M, N, K, group, split, need, bound)
    assert n == 675


def test_path_and_schedule_rules_at_the_benchmark_shapes(lib):
    """Host logic only (148 SMs assumed without a device, which is also what a B200 reports): the
    path and the split the library reports for a shape are the ones it runs (w4a16_gemm asks the same
    functions).  Values are the measured optima recorded beside the rules in the sources."""
    DECODE, TILE = 2, 3
    path = lambda M, N, K: lib.w4a16_choose_path(M, N, K, 128)
    split = lambda M, N, K: lib.w4a16_choose_split_k(M, N, K, 128)
    # up to 16 rows (one pass of the warp-MMA kernel over the weights): that kernel, but for long shapes from 9 rows on
    for N, K in [(4096, 4096), (4096, 11008), (8192, 28672), (22016, 4096), (1536, 6144), (12288, 4096)]:
        for M in (1, 4, 8, 9, 16):
            assert path(M, N, K) == (TILE if M > 8 and (N, K) in [(8192, 28672), (22016, 4096), (12288, 4096)] else DECODE)
    assert split(16, 4096, 11008) == 4
    # path and split are those of the plan that the call itself makes, and forcing them gives the same plan
    for M, N, K in [(9, 22016, 4096), (16, 12288, 4096), (16, 4096, 11008), (8, 8192, 28672), (32, 4096, 4096), (600, 8192, 8192)]:
        plan = B.w4a16_gemm_plan(M, N, K)
        assert path(M, N, K) == (DECODE if plan.kernel == B.KERNEL_DECODE else TILE)
        forced = B.w4a16_gemm_plan(M, N, K, path=path(M, N, K))
        assert (forced.kernel, forced.tile_rows, forced.split_k) == (plan.kernel, plan.tile_rows, plan.split_k)
    # above 16 rows: tcgen05
    for M in (17, 32, 64, 256, 4096):
        assert path(M, 4096, 11008) == TILE
    # slices per tile of the warp-MMA kernel: four (one cluster per tile) at config 2, whole tiles
    # for the wide gate/up layer, at most six per cluster for narrow matrices
    assert split(1, 4096, 11008) == 4
    assert split(1, 4096, 4096) == 4
    assert split(1, 22016, 4096) == 1
    assert split(1, 12288, 4096) == 1
    assert split(1, 1536, 6144) == 6
    assert split(1, 2048, 8192) == 6
    # wide batch tiles: whole tiles at M = 4096 (no partial tiles at all)
    assert split(4096, 8192, 8192) == 1
    # unsupported shapes are refused, not guessed
    assert lib.w4a16_choose_path(1, 100, 4096, 128) < 0


def test_workspace_query_covers_what_every_call_asks_for(lib):
    """Host logic, sizes drawn over the supported range: the size that w4a16_workspace_bytes reports is enough for the
    call on every path, whatever the group, and w4a16_choose_split_k reports the split that runs.  (The exchange buffer of a
    cluster shares its room with scale rows, so the number of slices depends on the group.)"""
    rng = random.Random(20)
    shapes = [(64, 2560, 5120), (64, 3008, 5120), (51, 1024, 1536), (50, 3072, 19200), (9, 22016, 4096)]
    for _ in range(1500):
        shapes.append((rng.choice([1, 8, 16, 32, rng.randint(1, 64), rng.randint(49, 64), rng.randint(65, 256), rng.randint(257, 4096)]),
                       64 * rng.randint(1, 448), 128 * rng.randint(1, 224)))
    for M, N, K in shapes:
        for group in (32, 64, 128):
            for split in {0, min(2, K // 128), min(rng.randint(2, 12), K // 128), K // 128}:
                size = lib.w4a16_workspace_bytes(M, N, K, group, split)
                for path in (0, 1, 2, 3):
                    try:
                        p = B.w4a16_gemm_plan(M, N, K, group, split, path)
                    except B.W4A16Error as e:
                        assert e.code == -9 and path == B.PATH_DECODE and M > 16     # more batch chunks than tickets
                        continue
                    assert p.workspace_bytes <= size, (M, N, K, group, split, path)
                    assert B.w4a16_gemm_plan(M, N, K, group, split, path, True).workspace_bytes <= size, (M, N, K, group, split, path)
                    if split != 0:
                        assert p.split_k == split
                    elif path != B.PATH_SIMPLE and p.split_k != 0:
                        assert lib.w4a16_choose_split_k_ex(M, N, K, group, path) == p.split_k, (M, N, K, group, path)


def test_slices_of_few_column_tiles_meet_in_a_cluster(lib):
    """Up to 16 rows and few column tiles: the sum through the workspace costs time for every slice and every row, so many
    slices are not taken because each is short (us, six in a cluster / the slices named): M = 10, K = 4480 4.6 / 35 14.1;
    M = 11, K = 6016 5.4 / 18 10.7; M = 16, K = 5632 6.2 / 15 11.6.  With one row and a long K they are ahead."""
    for M, N, K, group in [(10, 384, 4480, 32), (10, 384, 4224, 64), (11, 896, 6016, 128), (9, 768, 5888, 32), (16, 1088, 5632, 32)]:
        p = B.w4a16_gemm_plan(M, N, K, group, 0, B.PATH_DECODE)
        assert (p.split_k, p.cluster) == (6, 1), (M, N, K, group)
    assert B.w4a16_gemm_plan(2, 640, 19072, 64).split_k == 25        # 7.9 us; six in a cluster 9.3
    # pairs of CTAs up to the last two places (147 tiles 10.3 us, balanced 14.4; 148 10.3 and 12.4), but one tile per SM
    # of a short K stays whole (K = 2048: 5.9, pairs 6.2)
    for M, N, K, split in [(4, 64 * 147, 7168, 2), (16, 64 * 148, 7168, 2), (16, 64 * 147, 2048, 2), (16, 64 * 148, 2048, 1)]:
        assert B.w4a16_gemm_plan(M, N, K, 128, 0, B.PATH_DECODE).split_k == split, (M, N, K)


def test_schedules_of_few_or_whole_column_tiles_above_16_rows(lib):
    """tcgen05 path, us of the schedule taken once / of the one asked for here.  Few column tiles and a long K: as many slices
    as pay for being added, more than a cluster holds for the two-CTA kernel and not one per SM for the wide one (M = 51,
    K = 19712, N = 128: 8 slices 11.9 / 25 9.1; M = 240, K = 21760, N = 128: 74 slices 25.6 / 24 11.0).  One wave of whole tiles
    where slices do not fit well (M = 45, K = 1408, N = 11904: three slices 9.6 / 8.0)."""
    p = B.w4a16_gemm_plan(51, 128, 19712)
    assert (p.kernel, p.cluster) == (B.KERNEL_MID64, 0) and 16 <= p.split_k <= 32
    for M, N, K in [(240, 128, 21760), (89, 128, 22784), (256, 128, 17152), (177, 64, 13312), (71, 320, 6016)]:
        p = B.w4a16_gemm_plan(M, N, K)
        assert 2 <= p.split_k <= 30, (M, N, K, p.split_k)
    assert B.w4a16_gemm_plan(45, 11904, 1408, 64).split_k <= 2
    # 9 to 16 rows: long shapes of few tiles go to the tcgen05 kernel, groups of 32 and more tiles than CTA slots do not
    assert B.w4a16_gemm_plan(16, 1024, 27648).kernel == B.KERNEL_MID64
    assert B.w4a16_gemm_plan(16, 22016, 4096).kernel == B.KERNEL_MID64
    assert B.w4a16_gemm_plan(16, 22016, 4096, 32).kernel == B.KERNEL_DECODE
    assert B.w4a16_gemm_plan(16, 20224, 8192).kernel == B.KERNEL_DECODE


def test_sizes_beyond_32_bit_arithmetic_are_refused(lib):
    """The GEMM kernels number their units and chunks in 32 bits, the kernel that sums slices the rows of all tiles, which
    are the bound for a short K."""
    def code(*args):
        try:
            B.w4a16_gemm_plan(*args)
        except B.W4A16Error as e:
            return e.code
        return 0
    assert code(1 << 25, 4096, 256, 128, 2, B.PATH_TILE) == 0           # 2^30 rows
    assert code(1 << 26, 8192, 256, 128, 2, B.PATH_TILE) == -2          # 2^32 rows, 2^25 units
    assert code(1 << 26, 8192, 256, 128, 1, B.PATH_TILE) == 0           # whole tiles: nothing is summed
    assert code(1 << 30, 8192, 256, 128, 1, B.PATH_TILE) == 0           # 2^29 units
    assert code(1 << 30, 65536, 256, 128, 1, B.PATH_TILE) == -2         # 2^32 units
    assert code(1 << 24, 64, 128, 128, 1, B.PATH_SIMPLE) == -9


def test_argument_errors_are_reported_before_any_device_work(lib):
    buf = (ctypes.c_uint8 * 4096)()
    p = ctypes.addressof(buf)
    p = (p + 15) // 16 * 16
    assert lib.w4a16_gemm(None, p, p, p, p, 1, 64, 128, 128, 1, None) == -1
    assert lib.w4a16_gemm(p, p, p, p, None, 1, 64, 128, 128, 1, None) == -1
    assert lib.w4a16_gemm(p, p, p, p, p, 1, 64, 128, 48, 1, None) == -2      # group
    assert lib.w4a16_gemm(p, p, p, p, p, 1, 60, 128, 128, 1, None) == -2     # N % 64
    assert lib.w4a16_gemm(p, p, p, p, p, 1, 64, 100, 128, 1, None) == -2     # K % 128
    assert lib.w4a16_gemm(p, p, p, p, p, 0, 64, 128, 128, 1, None) == -2     # M
    assert lib.w4a16_gemm(p + 2, p, p, p, p, 1, 64, 128, 128, 1, None) == -3  # alignment
    assert lib.w4a16_gemm(p, p, p, p, p, 1, 64, 128, 128, 2, None) == -4     # split_k > K/group
    assert lib.w4a16_gemm(p, p, p, p, p, 1, 64, 128, 128, -1, None) == -4
    assert lib.w4a16_gemm_ex(p, p, p, p, p, 1, 64, 128, 128, 1, 9, None) == -9
    assert lib.w4a16_pack(None, p, p, p, p, p, 64, 128, 128, None) == -1
    assert lib.w4a16_pack(p, p, p, p, p, p, 64, 128, 16, None) == -2
    assert lib.w4a16_pack(p, p, None, p, p, p, 64, 128, 128, None) == -1      # the plain entry points need Z
    assert lib.w4a16_gemm(p, p, p, None, p, 1, 64, 128, 128, 1, None) == -1
    assert lib.w4a16_pack_fmt(p, p, None, p, p, None, 64, 128, 128, 0, None) == -1   # asymmetric: Z required
    assert lib.w4a16_pack_fmt(p, p, None, p, p, None, 64, 128, 128, 8, None) == -2   # unknown flag
    assert lib.w4a16_gemm_fmt(p, p, p, None, None, p, 1, 64, 128, 128, 1, 0, 0, 0, None) == -1
    assert lib.w4a16_gemm_fmt(p, p, p, p, None, p, 1, 64, 128, 128, 1, 0, 0, 7, None) == -2   # unknown activation
    assert lib.w4a16_gemm_fmt(p, p, p, p, p + 1, p, 1, 64, 128, 128, 1, 0, 0, 0, None) == -3  # odd bias address
    assert lib.w4a16_dequant_fmt(p, p, None, p, 64, 128, 128, 0, None) == -1
    assert lib.w4a16_dequant(p, p, p, None, 64, 128, 128, None) == -1
    assert lib.w4a16_dequant(p, p, p, p + 4, 64, 128, 128, None) == -3
    assert lib.w4a16_gemm_host(None, p, p, p, p, p, p, 1, 64, 128, 128, 1, None) == -1
    assert lib.w4a16_device_status(None) == -1
    for code in range(-9, 1):
        assert len(B.strerror(code)) > 1


def test_binding_refuses_to_run_without_the_library(monkeypatch, tmp_path):
    monkeypatch.setattr(B, "_lib", None)
    monkeypatch.setattr(B, "LIB_PATH", str(tmp_path / "missing.so"))
    with pytest.raises(RuntimeError, match="no CPU or PyTorch fallback"):
        B.load()
