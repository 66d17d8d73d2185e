"""When the kernel behind a GEMM may start.  Kernels are launched as programmatic dependents; a GEMM lets its successor in
from its teardown, not while it runs (streaming blocks beside a running GEMM slow both down).  A probe launched behind the
GEMM records when it started and when the GEMM had completed."""
import ctypes

import numpy as np
import pytest
import torch

from paper_2606_26453_b200 import build

pytestmark = pytest.mark.gpu


class Dims(ctypes.Structure):
    _fields_ = [(n, ctypes.c_int32) for n in "THIEK"]


# kernel, rows per expert of 8 experts: swapped and fixed-height pairs, single-CTA tiles, the weight gradients, the three FP8
# kernels and the FP8 weight gradient
CASES = [("down", 1024), ("down", 2048), ("gateup", 128), ("down_wgrad", 2048), ("down_mxfp8", 32), ("down_mxfp8", 128),
         ("down_mxfp8", 2048), ("down_wgrad_mxfp8", 2048)]


@pytest.mark.parametrize("kernel,rows", CASES)
def test_a_gemm_lets_its_successor_in_at_its_end(kernel, rows):
    from paper_2606_26453_b200 import binding as B
    B.load_library()
    lib = ctypes.CDLL(build.build_library(waittest=True))
    E, H, I = 8, 2048, 2048
    R = rows * E
    d, bd = Dims(R, H, I, E, 1), B.dims(R, H, I, E, 1)
    off = torch.arange(0, R + 1, rows, dtype=torch.int32, device="cuda")
    bf = lambda *s: torch.zeros(s, dtype=torch.bfloat16, device="cuda")
    u8 = lambda n: torch.zeros(n, dtype=torch.uint8, device="cuda")
    act = (u8(R * I), u8(B.moe_mxfp8_act_scale_bytes(bd)))
    wts = (u8(E * H * I), u8(B.moe_mxfp8_w_down_scale_bytes(bd)))
    tok = lambda n: (u8(B.moe_mxfp8_tokens_codes_bytes(bd, n)), u8(B.moe_mxfp8_tokens_scale_bytes(bd, n)))
    htok, dtok = tok(I), tok(H)
    for t, n in ((htok, I), (dtok, H)):
        B.moe_mxfp8_quantize_tokens(bd, bf(R, n), n, 0, n, off, *t)
    fn, tensors = {
        "down": ("moe_grouped_gemm_down", (bf(R, I), bf(E, I, H), off, bf(R, H))),
        "gateup": ("moe_grouped_gemm_gateup_swiglu", (bf(R, H), bf(E, H, I), bf(E, H, I), off, bf(R, I), bf(R, 2 * I))),
        "down_wgrad": ("moe_grouped_gemm_down_wgrad", (bf(R, I), bf(R, H), off, bf(E, I, H))),
        "down_mxfp8": ("moe_grouped_gemm_down_mxfp8", (*act, *wts, off, bf(R, H))),
        "down_wgrad_mxfp8": ("moe_grouped_gemm_down_wgrad_mxfp8", (*htok, *dtok, bf(E, I, H))),
    }[kernel]
    stamps = torch.zeros(2, dtype=torch.int64, device="cuda")
    begin, end = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    p, stream = ctypes.c_void_p, ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    early, total = [], []
    for _ in range(7):
        torch.cuda.synchronize()
        begin.record()
        assert getattr(lib, fn)(ctypes.byref(d), *(p(t.data_ptr()) for t in tensors), stream) == 0
        assert lib.moe_test_dependent_start(p(stamps.data_ptr()), stream) == 0
        end.record()
        torch.cuda.synchronize()
        early.append(int(stamps[1] - stamps[0]) / 1e3)
        total.append(begin.elapsed_time(end) * 1e3)
    print(kernel, rows, "started", early, "us ahead of the end of", total)
    # let in at the start it would be nearly the whole duration (tens to hundreds of us) ahead of the end
    assert np.median(early) < max(0.3 * np.median(total), 8.0), (early, total)
