"""The CTA-pair block-scaled FP8 GEMM at the edges of its tiles (256 output features and equal tiles of at most 208 rows, or 256 rows
and 208 features) and at the lines where it takes over from the single-CTA kernel, through the down projection, against the exact products of the dequantised
operands with the tolerance of the other FP8 GEMM tests."""
import numpy as np
import pytest
import torch

from oracle import moe_oracle as O
from paper_2606_26453_b200 import workloads as W
from tests import helpers as Hh

pytestmark = pytest.mark.gpu

CASES = {   # output features, contraction, rows of each expert
    "one_tile_half_wide": (128, 128, [256]),                       # one block of features: a single CTA's
    "row_edges": (384, 256, [207, 208, 209, 415, 416, 417]),       # 256 rows a tile; one and two row tiles
    # 256 features a tile:
    "last_tile_half_wide": (640, 256, [207, 208, 209, 415, 416, 417]),   # the second CTA has no features; one, two and three row tiles
    "low_box_edges": (256, 640, [128, 129, 1, 16, 17, 1040, 624]), # 64 rows per CTA and more; five tiles of 208
    "empty_and_last": (640, 384, [0, 900, 0, 33, 0]),
    "many_slices": (256, 1152, [300, 250]),                        # more slices than scale words in flight
    # 256 rows a tile:
    "rows_m_edges": (384, 256, [255, 256, 257, 511, 512, 513]),    # columns 208 and 176; one, two and three row tiles
    "rows_m_halves": (384, 640, [127, 128, 129, 1, 33, 1040, 624]),  # the second CTA's rows: none, one; five tiles
    "rows_m_empty": (384, 128, [0, 900, 0, 33, 0, 700]),
    "rows_m_many_slices": (384, 1152, [300, 250]),
    "rows_m_narrow_last": (1664, 128, [431] * 8),                  # eight tiles of 208 against six and a half of 256
    "96_rows": (256, 512, [96] * 74),                              # the first sizes of the pair form with few rows ...
    "96_rows_too_few_tiles": (256, 512, [96] * 73),                # ... and the last of the other:
    "96_rows_short": (256, 384, [96] * 74),                        # too few tiles, too short a contraction
    "96_rows_uneven": (384, 512, [1, 0, 31, 33, 352] + [99] * 42),
}


@pytest.mark.parametrize("name", list(CASES))
def test_pair_tiles(name):
    from paper_2606_26453_b200 import binding as B
    H, I, counts = CASES[name]
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
    guard = 40                                                     # rows behind the output that nobody may touch
    out = torch.full((R + guard, H), float("nan"), dtype=torch.bfloat16, device="cuda")
    B.moe_grouped_gemm_down_mxfp8(d, hc, hs, wc, ws, torch.from_numpy(offsets).cuda(), out[:R])
    torch.cuda.synchronize()
    assert B.moe_device_status() == 0
    assert bool(torch.isnan(out[R:]).all())
    Hh.assert_close(Hh.to_np64(out[:R]), O.down_mxfp8(h, w, offsets), name, rel_fro=Hh.PER_CALL_FROBENIUS)
