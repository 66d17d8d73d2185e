"""The kernels of one stream start before their predecessors have finished (programmatic dependent launch).  Back to back
without any synchronisation, and replayed from a CUDA graph, a step has to give bit for bit what it gives when the
device is idle before every call; every buffer is reused from step to step, so that a kernel which read too early or
wrote too early would meet the other step's values."""
import pytest
import torch

pytestmark = pytest.mark.gpu

SHAPES = [(64, 128, 256, 8, 2), (300, 384, 256, 16, 3), (2048, 512, 768, 8, 2)]   # T, H, I, E, K


def _inputs(B, T, H, I, E, K, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    n = lambda *s: torch.randn(s, generator=g, device="cuda")
    return dict(logits=n(T, E), x=n(T, H).bfloat16(), dy=n(T, H).bfloat16(), wg=(0.1 * n(E, H, I)).bfloat16(),
                wu=(0.1 * n(E, H, I)).bfloat16(), wd=(0.1 * n(E, I, H)).bfloat16())


class _Step:
    """Router, bf16 layer forward and backward, router backward, then the FP8 forward on the same routing."""

    def __init__(self, B, T, H, I, E, K):
        self.B, self.b = B, B.alloc_layer_buffers(T, H, I, E, K)
        self.d, R = self.b.d, T * K
        u8 = lambda n: torch.zeros(n, dtype=torch.uint8, device="cuda")
        d = self.d
        self.idx = torch.empty((T, K), dtype=torch.int32, device="cuda")
        self.w = torch.empty((T, K), dtype=torch.float32, device="cuda")
        self.dlogits = torch.empty((T, E), dtype=torch.float32, device="cuda")
        self.xq = u8(R * H), u8(B.moe_mxfp8_x_scale_bytes(d))
        self.hq = u8(R * I), u8(B.moe_mxfp8_act_scale_bytes(d))
        self.gq = u8(E * 2 * I * H), u8(B.moe_mxfp8_w_gateup_scale_bytes(d))
        self.dq = u8(E * H * I), u8(B.moe_mxfp8_w_down_scale_bytes(d))
        self.gu8 = torch.empty((R, 2 * I), dtype=torch.bfloat16, device="cuda")
        self.h8 = torch.empty((R, I), dtype=torch.bfloat16, device="cuda")
        self.y8 = torch.empty((R, H), dtype=torch.bfloat16, device="cuda")

    def calls(self, v):
        B, b, d = self.B, self.b, self.d
        return [
            lambda: B.moe_router_topk(d, v["logits"], self.idx, self.w),
            lambda: B.moe_permute(d, v["x"], self.idx, b.x_perm, b.counts, b.offsets, b.row_to_pair, b.pair_to_row, b.workspace),
            lambda: B.moe_grouped_gemm_gateup_swiglu(d, b.x_perm, v["wg"], v["wu"], b.offsets, b.h_act, b.gu),
            lambda: B.moe_grouped_gemm_down(d, b.h_act, v["wd"], b.offsets, b.y_perm),
            lambda: B.moe_unpermute_combine(d, b.y_perm, self.w, b.pair_to_row, b.y),
            lambda: B.layer_backward(b, v["dy"], self.w, v["wg"], v["wu"], v["wd"]),
            lambda: B.moe_router_topk_bwd(d, self.idx, self.w, b.dtopk_w, self.dlogits),
            lambda: B.moe_mxfp8_quantize_w_gateup(d, v["wg"], v["wu"], *self.gq),
            lambda: B.moe_mxfp8_quantize_w_down(d, v["wd"], *self.dq),
            lambda: B.moe_mxfp8_quantize_x_perm(d, b.x_perm, *self.xq),
            lambda: B.moe_grouped_gemm_gateup_mxfp8(d, *self.xq, *self.gq, b.offsets, self.gu8),
            lambda: B.moe_swiglu_mxfp8(d, self.gu8, self.h8, *self.hq),
            lambda: B.moe_grouped_gemm_down_mxfp8(d, *self.hq, *self.dq, b.offsets, self.y8),
        ]

    def results(self):
        b = self.b
        return [t.clone() for t in (self.idx, self.w, b.offsets, b.pair_to_row, b.y, b.dx, b.dtopk_w, self.dlogits, b.dw_gate,
                                    b.dw_up, b.dw_down, self.h8, self.y8)]


@pytest.mark.parametrize("shape", SHAPES)
def test_back_to_back_and_replayed_steps_equal_synchronised_ones(shape):
    from paper_2606_26453_b200 import binding as B
    B.load_library()
    step = _Step(B, *shape)
    sets = [_inputs(B, *shape, seed) for seed in (1, 2)]
    want = []
    for v in sets:
        for call in step.calls(v):
            call()
            torch.cuda.synchronize()
        want.append(step.results())
    for i in range(12):                                   # no synchronisation between calls or steps
        for call in step.calls(sets[i % 2]):
            call()
        got = step.results()
        for a, b in zip(got, want[i % 2]):
            assert torch.equal(a, b)
    fixed = {k: t.clone() for k, t in sets[0].items()}    # the captured step reads these
    stream = torch.cuda.Stream()
    stream.wait_stream(torch.cuda.current_stream())
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        for call in step.calls(fixed):
            call()
    for i in range(4):
        for k, t in sets[i % 2].items():
            fixed[k].copy_(t)
        graph.replay()
        got = step.results()
        for a, b in zip(got, want[i % 2]):
            assert torch.equal(a, b)
    assert B.moe_device_status() == 0
