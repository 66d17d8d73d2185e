"""Both sides of the row count at which the plain grouped GEMMs change from swapped to fixed-height tiles (1600 rows per expert
on average, 512 for contractions of fewer than 512 elements), at the heights where either form has a remainder, against
the oracle."""
import numpy as np
import pytest

from oracle import moe_oracle as O
from tests import helpers as Hh
from tests.test_gpu_fuzz import FLOAT_OUTPUTS

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,I,counts", [
    (576, 512, [1599]),                       # swapped: seven tiles of 240 rows, the last one shorter
    (576, 512, [1600]),                       # fixed: six tiles and a quarter
    (512, 576, [257, 1, 2941, 3200]),         # swapped, tiles of 256 and 128 + 1 rows
    (512, 576, [3072, 127, 1601]),            # fixed, one row in the last tile
    # a contraction of fewer than 512 elements (down, down dgrad; the gate/up dgrad contracts 2I): fixed from 512 rows on
    (320, 192, [1599]),
    (192, 320, [257, 1, 2941, 3200]),
    (448, 448, [600, 0, 425]),                # 342 rows per expert: swapped
    (448, 448, [600, 0, 936]),                # 512: fixed but for the gate/up dgrad, with an expert without rows
    (512, 448, [600, 0, 936]),                # and the down dgrad
])
def test_tile_forms_at_their_border(H, I, counts):
    cfg, host = Hh.ragged_workload(counts, K=1, H=H, I=I, seed=11)
    ref = O.layer_fwd_bwd(host["X"], host["topk_idx"], host["topk_w"], host["W_gate"], host["W_up"], host["W_down"], host["dY"])
    for fused in (False, True):
        b = Hh.run_cuda_layer(Hh.device_workload(host), cfg.E, fused_swiglu_bwd=fused)
        assert np.array_equal(b.offsets.cpu().numpy(), ref["offsets"])
        for attr, key in FLOAT_OUTPUTS:
            if not (fused and attr == "dh_act"):
                Hh.assert_close(Hh.to_np64(getattr(b, attr)), ref[key], f"{key} counts={counts} fused={fused}")
