"""Edges of the block-scaled FP8 quantisers that the layer's own values do not reach: infinities, NaN, subnormals and signed
zeros, and the token-axis quantiser's scan over the experts at its smallest and largest expert counts.  Codes and scale
bytes are whole numbers and compared bit for bit."""
import numpy as np
import pytest
import torch

from oracle import moe_oracle as O
from paper_2606_26453_b200 import workloads as W
from tests import helpers as Hh
from tests.test_gpu_mxfp8 import _act_scales_from_layout, _oracle_tokens_layout

pytestmark = pytest.mark.gpu


def _u8(n):
    return torch.full((n,), 0xFF, dtype=torch.uint8, device="cuda")


@pytest.mark.parametrize("rows", [1, 127, 129])
def test_special_values(rows):
    """A NaN takes no part in its block's scale and keeps a NaN code; an infinity gives the largest scale and saturates."""
    from paper_2606_26453_b200 import binding as B
    n, r = 256, rows - 1
    x = W.round_to_bf16(np.random.default_rng(rows).standard_normal((rows, n)).astype(np.float32))
    x[r, 0:32] = -0.0
    x[r, 32:64] = np.linspace(-31, 31, 32, dtype=np.float32) * 2.0 ** -133       # subnormal bf16 values
    finite = x.copy()
    x[r, 70] = np.nan                                                           # one NaN among numbers
    x[r, 96:128] = np.nan                                                       # nothing but NaN
    x[r, 130], x[r, 131] = np.inf, -np.inf
    finite[r, 70], finite[r, 96:128], finite[r, 128:160] = 0.0, 0.0, 0.0
    codes, scales, _ = O.mxfp8_quantize(finite)
    codes[r, 70], codes[r, 96:128] = 0x7F, 0x7F
    codes[r, 128:160] = np.where(np.signbit(x[r, 128:160]), 0x80, 0)            # any finite value over 2^120
    codes[r, 130], codes[r, 131] = 0x7E, 0xFE
    scales[r, 4] = 120 + 127
    d = B.dims(rows, 128, n, 1, 1)
    c, s = _u8(rows * n), _u8(B.moe_mxfp8_act_scale_bytes(d))
    B.moe_mxfp8_quantize_h_act(d, Hh.to_dev_bf16(x), c, s)
    torch.cuda.synchronize()
    got = c.cpu().numpy().reshape(rows, n)
    nan = np.isnan(x)
    assert np.array_equal(np.where(nan, got & 0x7F, got), codes)                # the sign of a NaN is nobody's
    assert np.array_equal(_act_scales_from_layout(s.cpu().numpy(), rows, n), scales)


def _mixed_counts(E):
    rng = np.random.default_rng(E)
    counts = rng.integers(0, 3, size=E)
    counts[rng.integers(0, E)] = 129
    counts[-1] = 31
    return counts


# ... and rows that need as many slices as there are rows, the most there can be: one row per expert, one row in all
@pytest.mark.parametrize("counts", [_mixed_counts(E) for E in (1, 2, 127, 1023, 1024)] +
                         [np.ones(130, int), np.ones(1024, int), np.eye(1, 300, 299, dtype=int)[0], np.eye(1, 1024, 0, dtype=int)[0]],
                         ids=["E1", "E2", "E127", "E1023", "E1024", "one_each", "one_each_of_1024", "last_only", "first_only"])
def test_token_quantiser_expert_scan(counts):
    from paper_2606_26453_b200 import binding as B
    E = counts.size
    rng = np.random.default_rng(E)
    offsets = np.concatenate([[0], np.cumsum(counts)]).astype(np.int32)
    R, ld, col0, n = int(offsets[-1]), 384, 8, 256
    x = W.round_to_bf16(rng.standard_normal((R, ld)).astype(np.float32))
    d = B.dims(R, 128, 128, E, 1)
    P = ((R + 127) // 128) * 128 + 128 * E
    codes, scales = _u8(B.moe_mxfp8_tokens_codes_bytes(d, n)), _u8(B.moe_mxfp8_tokens_scale_bytes(d, n))
    B.moe_mxfp8_quantize_tokens(d, Hh.to_dev_bf16(x), ld, col0, n, torch.from_numpy(offsets).cuda(), codes, scales)
    torch.cuda.synchronize()
    want_codes, want_scales, sp = _oracle_tokens_layout(x[:, col0:col0 + n], offsets)
    n_sl = int(sp[-1])
    assert np.array_equal(scales[:4 * (E + 1)].cpu().numpy().view(np.int32), sp.astype(np.int32))
    assert np.array_equal(codes.view(n, P)[:, :n_sl * 128].cpu().numpy(), want_codes)
    words = scales[8192: 8192 + (P // 128) * n * 4].view(P // 128, n, 4)[:n_sl].cpu().numpy()
    assert np.array_equal(words, want_scales)


@pytest.mark.parametrize("shift", [16, 32])
def test_transposing_quantisers_take_any_16_byte_alignment(shift):
    from paper_2606_26453_b200 import binding as B
    E, H, I = 3, 256, 384
    rng = np.random.default_rng(shift)
    w = W.round_to_bf16(rng.standard_normal((E, I, H)).astype(np.float32))
    d = B.dims(40, H, I, E, 1)
    out = []
    for s in (0, shift):
        room, scales = _u8(E * H * I + 64), _u8(B.moe_mxfp8_w_down_scale_bytes(d))
        codes = room[s:s + E * H * I]
        B.moe_mxfp8_quantize_w_down(d, Hh.to_dev_bf16(w), codes, scales)
        torch.cuda.synchronize()
        assert bool((room[s + E * H * I:] == 0xFF).all()) and bool((room[:s] == 0xFF).all())
        out.append((codes.clone(), scales))
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])
    want = np.stack([O.mxfp8_quantize(w[e].T)[0] for e in range(E)])               # [E, H, I]
    assert np.array_equal(out[0][0].cpu().numpy().reshape(E, H, I), want)


@pytest.mark.parametrize("rows", [1, 33, 130])
def test_row_quantisers_take_any_16_byte_alignment(rows):
    from paper_2606_26453_b200 import binding as B
    n, E = 384, 2
    rng = np.random.default_rng(rows)
    x = W.round_to_bf16(rng.standard_normal((rows, n)).astype(np.float32))
    w = W.round_to_bf16(rng.standard_normal((E, n, 128)).astype(np.float32))      # W_down [E, I, H]
    d = B.dims(rows, 128, n, E, 1)
    for shift in (8, 16):                                                         # elements: 16 and 32 bytes into the buffer
        def shifted(a):
            room = torch.zeros(a.size + 32, dtype=torch.bfloat16, device="cuda")
            room[shift:shift + a.size] = Hh.to_dev_bf16(a).flatten()
            return room[shift:shift + a.size].view(a.shape)
        c, s = _u8(rows * n + 16)[16:], _u8(B.moe_mxfp8_act_scale_bytes(d))
        B.moe_mxfp8_quantize_h_act(d, shifted(x), c, s)
        wc, ws = _u8(E * n * 128 + 16)[16:], _u8(B.moe_mxfp8_w_down_dgrad_scale_bytes(d))
        B.moe_mxfp8_quantize_w_down_dgrad(d, shifted(w), wc, ws)
        torch.cuda.synchronize()
        codes, scales, _ = O.mxfp8_quantize(x)
        assert np.array_equal(c.cpu().numpy().reshape(rows, n), codes)
        assert np.array_equal(_act_scales_from_layout(s.cpu().numpy(), rows, n), scales)
        assert np.array_equal(wc.cpu().numpy().reshape(E, n, 128), O.mxfp8_quantize(w)[0])
