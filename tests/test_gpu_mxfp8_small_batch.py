"""The single-CTA block-scaled FP8 GEMM at the edges of its two forms: fewer rows than a tile, experts at and around a tile's
64 and 128 rows, and both sides of 64 rows per expert on average, where one form hands over to the other.

Tolerance: the per-call bound of the other FP8 GEMM tests (exact products of the dequantised operands, fp32 accumulation,
one rounding to bf16)."""
import ctypes

import numpy as np
import pytest
import torch

from oracle import moe_oracle as O
from paper_2606_26453_b200 import build, workloads as W
from tests import helpers as Hh

pytestmark = pytest.mark.gpu

CASES = {
    "one_row": [1],
    "fewer_rows_than_a_tile": [0, 7, 1, 0, 31],
    "tile_edges": [64, 63, 1, 65, 0, 32, 33, 128, 97],                 # 53 rows per expert: swapped, one to three tiles
    "a_long_expert": [300] + [0] * 11,                                 # swapped, five tiles of one expert
    "at_the_border": [64, 60, 68],                                     # 64 rows per expert: the last of the swapped form
    "past_the_border": [64, 60, 69],                                   # the first of the other
    "unswapped_edges": [128, 127, 129, 31, 255, 1],
    "most_experts_of_the_swapped_form": [1] * 450 + [0] * 35 + [70],
    "more_experts": [1] * 450 + [0] * 36 + [70],                       # unswapped from here on
    "most_experts": [1] * 1000 + [0] * 23 + [70],
}


@pytest.mark.parametrize("name", list(CASES))
def test_small_batches(name):
    from paper_2606_26453_b200 import binding as B
    counts = CASES[name]
    H, I = (384, 640) if len(counts) < 100 else (128, 128)
    rng = np.random.default_rng(len(name))
    offsets = np.concatenate([[0], np.cumsum(counts)]).astype(np.int32)
    R, E = int(offsets[-1]), len(counts)
    h = W.round_to_bf16(rng.standard_normal((R, I)).astype(np.float32))
    w = W.round_to_bf16((0.02 * rng.standard_normal((E, I, H))).astype(np.float32))
    d = B.dims(R, H, I, E, 1)
    u8 = lambda n: torch.full((n,), 0xFF, dtype=torch.uint8, device="cuda")
    hc, hs = u8(R * I), u8(B.moe_mxfp8_act_scale_bytes(d))
    wc, ws = u8(E * H * I), u8(B.moe_mxfp8_w_down_scale_bytes(d))
    B.moe_mxfp8_quantize_h_act(d, Hh.to_dev_bf16(h), hc, hs)
    B.moe_mxfp8_quantize_w_down(d, Hh.to_dev_bf16(w), wc, ws)
    guard = 4                                                          # rows behind the output that nobody may touch
    out = torch.full((R + guard, H), float("nan"), dtype=torch.bfloat16, device="cuda")
    B.moe_grouped_gemm_down_mxfp8(d, hc, hs, wc, ws, torch.from_numpy(offsets).cuda(), out[:R])
    torch.cuda.synchronize()
    assert B.moe_device_status() == 0
    assert bool(torch.isnan(out[R:]).all())
    Hh.assert_close(Hh.to_np64(out[:R]), O.down_mxfp8(h, w, offsets), name, rel_fro=Hh.PER_CALL_FROBENIUS)


@pytest.mark.parametrize("E", [1, 8, 486, 487, 512, 1024])
@pytest.mark.parametrize("rows", [1, 64, 100])
def test_every_launched_cta_fits_its_sm(E, rows):
    """The kernel runs over a tile list that is dealt out by CTA: a CTA that had to wait for another one's SM would double the
    duration.  The tables grow with the experts, so the form with two CTAs per SM has a largest expert count."""
    lib = ctypes.CDLL(build.build_library(waittest=True))
    ctas, smem = ctypes.c_int(), ctypes.c_int()
    lib.moe_test_mx_single_ctas(rows * E, E, ctypes.byref(ctas), ctypes.byref(smem))
    per_sm = torch.cuda.get_device_properties(0).shared_memory_per_multiprocessor
    assert ctas.value * (smem.value + 1024) <= per_sm                  # 1 KB of every CTA is the system's
    assert ctas.value == (2 if rows <= 64 and E <= 486 else 1)
