"""Widths that are no multiple of a tile's features or columns, and experts at the edges of the tiles, through every bf16 grouped GEMM of
a step, against the oracle with the tolerance of the other parity tests: the first cases with the SwiGLU forward unswapped (its swapped
form needs widths of 1536 and more), the others with all row-ragged GEMMs swapped."""
import pytest
import torch

from oracle import moe_oracle as O
from tests import helpers as Hh
from tests.test_gpu_fuzz import FLOAT_OUTPUTS

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,I,counts", [
    # fewer than 256 rows per expert
    (64, 64, [1]),                                       # one K block, 64 of a tile's features
    (64, 192, [1, 15, 16, 17, 0, 31, 32, 33, 63, 65]),   # rows around the MMA's steps of 16 and a block's 32
    (320, 448, [64, 127, 128, 129, 5]),
    (384, 576, [255, 256, 257, 48, 80]),                 # an expert's second tile
    # 256 and more: several tiles of at most 256 rows
    (64, 128, [300, 0, 490]),
    (128, 64, [511, 257, 16]),                           # two tiles less a row; a tile and a row
    (192, 320, [512, 700, 0, 100]),                      # two full tiles; three; none; one
    (320, 384, [513, 288, 289]),                         # two full tiles and a row
    (640, 576, [272, 1025, 129]),                        # five tiles
    # 1600 and more
    (320, 576, [1700, 1500]),
    (640, 704, [3300, 0]),
    (576, 896, [1601]),
])
def test_widths_and_rows_at_tile_edges(H, I, counts):
    cfg, host = Hh.ragged_workload(counts, K=1, H=H, I=I, seed=23)
    ref = O.layer_fwd_bwd(host["X"], host["topk_idx"], host["topk_w"], host["W_gate"], host["W_up"], host["W_down"], host["dY"])
    for fused in (False, True):
        b = Hh.run_cuda_layer(Hh.device_workload(host), cfg.E, fused_swiglu_bwd=fused)
        for attr, key in FLOAT_OUTPUTS:
            if not (fused and attr == "dh_act"):
                Hh.assert_close(Hh.to_np64(getattr(b, attr)), ref[key], f"{key} H={H} I={I} counts={counts} fused={fused}")


SWAPPED_SWIGLU = [   # H, I, rows of each expert
    (1536, 64, [255, 256, 257, 15, 16, 17, 31, 32, 33, 0, 300, 129]),   # the second CTA has no features; a tile and a row; blocks of 32 rows
    (1600, 192, [1, 0, 200, 176, 100, 127, 128]),                       # the last tile's second CTA has no features
    (1536, 448, [96, 97, 400, 0, 63, 65, 47, 49]),
    (1536, 128, [96]),                                                  # the fewest rows
    (1664, 320, [176, 176]),                                            # the most while one round of single CTAs would do
    (1536, 64, [200] * 100),                                            # more tiles than that
    (1536, 64, [319] * 80),
]


@pytest.mark.parametrize("H,I,counts", SWAPPED_SWIGLU)
def test_swapped_swiglu_forward(H, I, counts):
    """With and without saved pre-activations, nothing written behind the last row; then a whole step."""
    from paper_2606_26453_b200 import binding as B
    cfg, host = Hh.ragged_workload(counts, K=1, H=H, I=I, seed=31)
    ref = O.layer_fwd_bwd(host["X"], host["topk_idx"], host["topk_w"], host["W_gate"], host["W_up"], host["W_down"], host["dY"])
    dev = Hh.device_workload(host)
    b = Hh.run_cuda_layer(dev, cfg.E)
    for attr, key in FLOAT_OUTPUTS:
        Hh.assert_close(Hh.to_np64(getattr(b, attr)), ref[key], f"{key} H={H} I={I} counts={counts}")
    guarded = lambda n: torch.full((cfg.R + 32, n), float("nan"), dtype=torch.bfloat16, device="cuda")
    h, h_only, gu = guarded(I), guarded(I), guarded(2 * I)
    B.moe_grouped_gemm_gateup_swiglu(b.d, b.x_perm, dev["W_gate"], dev["W_up"], b.offsets, h[:cfg.R], gu[:cfg.R])
    B.moe_grouped_gemm_gateup_swiglu(b.d, b.x_perm, dev["W_gate"], dev["W_up"], b.offsets, h_only[:cfg.R], None)
    torch.cuda.synchronize()
    assert B.moe_device_status() == 0
    assert torch.equal(h[:cfg.R], b.h_act) and torch.equal(h_only[:cfg.R], b.h_act) and torch.equal(gu[:cfg.R], b.gu)
    assert all(bool(torch.isnan(t[cfg.R:]).all()) for t in (h, h_only, gu))


@pytest.mark.parametrize("counts", [[40, 250, 0, 33], [700, 333], [1600, 1650]])
def test_forward_without_saved_pre_activations(counts):
    """The activations do not depend on whether the pre-activations are kept, and nothing behind the last row is written."""
    from paper_2606_26453_b200 import binding as B
    H, I = 320, 448
    cfg, host = Hh.ragged_workload(counts, K=1, H=H, I=I, seed=29)
    dev = Hh.device_workload(host)
    b = Hh.run_cuda_layer(dev, cfg.E)
    h = torch.full((cfg.R + 32, I), float("nan"), dtype=torch.bfloat16, device="cuda")
    B.moe_grouped_gemm_gateup_swiglu(b.d, b.x_perm, dev["W_gate"], dev["W_up"], b.offsets, h[:cfg.R], None)
    torch.cuda.synchronize()
    assert B.moe_device_status() == 0
    assert torch.equal(h[:cfg.R], b.h_act) and bool(torch.isnan(h[cfg.R:]).all())
