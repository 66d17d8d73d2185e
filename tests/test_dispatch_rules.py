"""The rules that choose between the forms of a kernel, by the library's test-only build, without a device."""
import ctypes

from paper_2606_26453_b200 import build
from tests.test_gpu_mxfp8_pair_tiles import CASES
from tests.test_gpu_tile_edges import SWAPPED_SWIGLU


def test_mxfp8_gemm():
    """Which kernel a shape goes to: single CTAs, pairs with the weights on the M side, pairs with the rows there."""
    lib = ctypes.CDLL(build.build_library(waittest=True))
    lib.moe_test_mx_form.argtypes = [ctypes.c_longlong] + [ctypes.c_int] * 3
    forms = {name: lib.moe_test_mx_form(sum(c), len(c), H, I) for name, (H, I, c) in CASES.items()}
    assert forms == {"one_tile_half_wide": 0, "row_edges": 2, "last_tile_half_wide": 1, "low_box_edges": 1, "empty_and_last": 0, "many_slices": 1,
                     "rows_m_edges": 2, "rows_m_halves": 2, "rows_m_empty": 2, "rows_m_many_slices": 2, "rows_m_narrow_last": 2, "96_rows": 1,
                     "96_rows_too_few_tiles": 0, "96_rows_short": 0, "96_rows_uneven": 0}
    # sizes at which each was found the better one: many rows of 128 and of 384 features, row tiles of 208 that are just exceeded, few rows
    for R, E, n, k, form in ((893 * 110, 110, 128, 2688, 0), (5263 * 9, 9, 384, 8064, 2), (733 * 10, 10, 384, 2432, 2), (481 * 85, 85, 1664, 768, 2),
                             (419 * 152, 152, 3328, 640, 2), (110 * 129, 129, 384, 1024, 0), (106 * 15, 15, 2432, 896, 0), (96 * 130, 130, 640, 3456, 0), (128 * 128, 128, 1536, 2048, 1), (384 * 64, 64, 2816, 2048, 1),
                             (1024 * 128, 128, 2048, 768, 1), (2048 * 8, 8, 28672, 4096, 1), (2048 * 8, 8, 4096, 14336, 1), (25 * 8, 8, 4096, 14336, 0)):
        assert lib.moe_test_mx_form(R, E, n, k) == form, (R, E, n, k)


def test_threads_per_token_of_the_combine_backward():
    """Narrow rows share a block; not of so few tokens that the chip is not full, nor long rows."""
    lanes = ctypes.CDLL(build.build_library(waittest=True)).moe_test_combine_bwd_lanes
    for T, H, want in ((20000, 256, 32), (20000, 512, 32), (20000, 832, 32), (20000, 1024, 64), (10000, 1280, 32), (16384, 2048, 128), (8192, 4096, 256),
                       (14442, 2880, 128), (27, 2304, 256), (12, 7744, 256), (515, 3776, 256), (41, 2624, 256), (3593, 5696, 256), (4736, 1152, 32),
                       (2367, 1152, 64), (1, 64, 256), (148, 256, 256), (149, 256, 32), (444, 320, 256), (445, 320, 64), (445, 512, 64), (445, 1088, 256), (2368, 3072, 128), (2368, 3328, 32), (2367, 3328, 64), (2368, 3584, 128), (6681, 4352, 128), (9000, 3520, 64)):
        assert lanes(T, H, 2, 1) == want, (T, H, lanes(T, H, 2, 1))
    for T, H, want in ((148, 256, 256), (149, 256, 32), (592, 320, 256), (593, 320, 64), (593, 1088, 256), (4735, 1152, 64), (4736, 1152, 32), (20000, 1024, 64), (20000, 1536, 64), (20000, 1600, 128), (4279, 2304, 128), (2433, 3200, 128), (27, 2304, 256), (8192, 4096, 256)):
        assert lanes(T, H, 2, 0) == want, (T, H, lanes(T, H, 2, 0))   # without dtopk_w
    assert lanes(296, 320, 9, 1) == lanes(296, 320, 9, 0) == 256 and lanes(297, 320, 9, 1) == 64   # fewer blocks at once of the run-time K
    # the form that leaves its successor to the end exists for 32 threads per token only: others are small grids or blocks of 1024 pieces and more
    for T in (*range(1, 3000, 61), 592, 593, 1184, 1185, 2367, 2368, 4735, 4736, 100000):
        for H in range(64, 8192, 64):
            for with_dw in (0, 1):
                n = lanes(T, H, 1, with_dw)
                assert n == 32 or T <= (1 if with_dw else 2) * 592 * (256 // n) or 3 * (H // 8) * (256 // n) >= 1024, (T, H, with_dw, n)


def test_launches_of_a_permute():
    """A scan goes in between where the blocks' sums are worth a launch; the benchmark's count of launches follows the library's."""
    import bench
    from paper_2606_26453_b200 import workloads as W
    launches = ctypes.CDLL(build.build_library(waittest=True)).moe_test_permute_launches
    for T, K, E, want in ((2048, 1, 128, 1), (2049, 1, 128, 2), (32768, 8, 128, 3), (36485, 7, 8, 3), (5118, 5, 95, 3), (2354, 3, 552, 2), (536, 5, 999, 2),
                          (4096, 6, 64, 2), (1420, 7, 236, 2), (14336, 1, 128, 3), (6250, 4, 73, 2), (6250, 4, 74, 3),
                          (8192, 1, 183, 2), (8192, 1, 184, 3)):
        assert launches(T, K, E) == want, (T, K, E)
    for T, K, E in [(c.T, c.K, c.E) for c in W.CONFIGS.values()] + [(T, K, E) for T in (1, 2047, 2048, 3000, 8192, 60000) for K in (1, 2, 8) for E in (8, 183, 184, 1000)]:
        assert bench.permute_launches(W.MoeConfig("x", T=T, H=64, I=64, E=E, K=K, cfg_id=0)) == launches(T, K, E), (T, K, E)


def test_weight_gradient_beside_a_data_gradient():
    """Beside a short data gradient, not one that fills the chip, nor where hardly an expert has a row."""
    beside = ctypes.CDLL(build.build_library(waittest=True)).moe_test_weight_gradient_beside
    for rows, E, n, want in ((512, 8, 512, 1), (512, 8, 256, 1), (10500, 2, 512, 1), (16384, 64, 2048, 0), (10, 67, 256, 0), (10, 69, 320, 0), (8, 32, 256, 0),
                             (9, 32, 256, 1), (1, 1, 64, 1), (18944 - 256, 1, 255, 1), (147 * 256 + 255, 1, 64, 1), (148 * 256, 1, 64, 0)):
        assert beside(rows, E, n) == want, (rows, E, n)


def test_swapped_swiglu_forward():
    """From 96 rows per expert and widths of 1536 on, but below 320 rows not where single CTAs take one round; from 320 rows on with eight
    tiles and more per pair; not from 1600 on."""
    swapped = ctypes.CDLL(build.build_library(waittest=True)).moe_test_use_swapped_swiglu
    for H, I, counts in SWAPPED_SWIGLU:
        assert swapped(sum(counts), H, I, len(counts), 1), (H, I, counts)
    for R, E, H, I, want in ((95, 1, 1536, 128, 0), (96, 1, 1472, 128, 0), (177, 1, 1536, 128, 0), (315 * 4, 4, 2560, 1216, 0), (294 * 22, 22, 1920, 256, 0),
                             (236 * 5, 5, 3840, 1408, 0), (162 * 19, 19, 3584, 512, 0), (107 * 5, 5, 2944, 896, 1), (107 * 43, 43, 1792, 640, 1),
                             (250 * 8, 8, 4096, 14336, 1), (320 * 80, 80, 1536, 64, 0), (384 * 64, 64, 2048, 1408, 1), (1024 * 128, 128, 2048, 768, 1),
                             (1599 * 8, 8, 4096, 14336, 1), (1600 * 8, 8, 4096, 14336, 0), (1000 * 8, 8, 2048, 192, 0)):
        assert swapped(R, H, I, E, 1) == want, (R, E, H, I)
