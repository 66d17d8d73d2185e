"""The kernels of one stream start before their predecessors have finished (programmatic dependent launch).  Back to back
without any synchronisation, and replayed from a CUDA graph, a step has to give bit for bit what it gives when the
device is idle before every call; every buffer is reused from step to step, so that a kernel which read too early or
wrote too early would meet the other step's values.  The first test looks at the results of every step, with plain copies
that then stand between the steps; the second one has nothing between them and every call of the library in them."""
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


class _EveryCall(_Step):
    """The whole of the library's calls on one routing: the layer with the fused down dgrad, a second route-permute that takes
    the layer's own output (the combine writes it right ahead of the permute), and the FP8 training step with both kinds of
    weight gradients.  Nothing but these calls runs between one step and the next."""

    def __init__(self, B, T, H, I, E, K):
        super().__init__(B, T, H, I, E, K)
        R, d = T * K, self.d
        u8 = lambda n: torch.zeros(n, dtype=torch.uint8, device="cuda")
        bf = lambda *s: torch.zeros(s, dtype=torch.bfloat16, device="cuda")
        i32 = lambda n: torch.zeros(n, dtype=torch.int32, device="cuda")
        self.again = [bf(R, H), i32(E), i32(E + 1), i32(R), i32(R)]     # x_perm, counts, offsets, row_to_pair, pair_to_row
        self.static = [torch.zeros_like(t) for t in self.again]
        self.dyq = u8(R * H), u8(B.moe_mxfp8_dy_scale_bytes(d))
        self.dguq = u8(R * 2 * I), u8(B.moe_mxfp8_dgu_scale_bytes(d))
        self.ddq = u8(E * I * H), u8(B.moe_mxfp8_w_down_dgrad_scale_bytes(d))
        self.gdq = u8(E * H * 2 * I), u8(B.moe_mxfp8_w_gateup_dgrad_scale_bytes(d))
        tok = lambda n: (u8(B.moe_mxfp8_tokens_codes_bytes(d, n)), u8(B.moe_mxfp8_tokens_scale_bytes(d, n)))
        self.h_tok, self.dy_tok, self.x_tok, self.dg_tok, self.du_tok = tok(I), tok(H), tok(H), tok(I), tok(I)
        self.dh8, self.dgu8, self.dx8, self.dgu_fused = bf(R, I), bf(R, 2 * I), bf(R, H), bf(R, 2 * I)
        self.dw8 = bf(E, I, H), bf(E, H, I), bf(E, H, I)

    def calls(self, v):
        B, b, d, H, I = self.B, self.b, self.d, self.d.H, self.d.I
        forward = super().calls(v)
        return forward[:5] + [
            lambda: B.moe_permute(d, b.y, self.idx, *self.again, b.workspace),
            lambda: B.moe_permute_static_scratch(d, b.y, self.idx, *self.static)] + forward[5:7] + [
            lambda: B.moe_grouped_gemm_down_dgrad_swiglu_bwd(d, b.dy_perm, v["wd"], b.gu, b.offsets, self.dgu_fused)] + forward[7:] + [
            lambda: B.moe_mxfp8_quantize_w_down_dgrad(d, v["wd"], *self.ddq),
            lambda: B.moe_mxfp8_quantize_w_gateup_dgrad(d, v["wg"], v["wu"], *self.gdq),
            lambda: B.moe_mxfp8_quantize_dy_perm(d, b.dy_perm, *self.dyq),
            lambda: B.moe_grouped_gemm_down_dgrad_mxfp8(d, *self.dyq, *self.ddq, b.offsets, self.dh8),
            lambda: B.moe_swiglu_bwd_mxfp8(d, self.dh8, self.gu8, self.dgu8, *self.dguq),
            lambda: B.moe_grouped_gemm_gateup_dgrad_mxfp8(d, *self.dguq, *self.gdq, b.offsets, self.dx8),
            lambda: B.moe_mxfp8_quantize_tokens(d, self.h8, I, 0, I, b.offsets, *self.h_tok),
            lambda: B.moe_mxfp8_quantize_tokens(d, b.dy_perm, H, 0, H, b.offsets, *self.dy_tok),
            lambda: B.moe_grouped_gemm_down_wgrad_mxfp8(d, *self.h_tok, *self.dy_tok, self.dw8[0]),
            lambda: B.moe_mxfp8_quantize_tokens(d, b.x_perm, H, 0, H, b.offsets, *self.x_tok),
            lambda: B.moe_mxfp8_quantize_tokens(d, self.dgu8, 2 * I, 0, I, b.offsets, *self.dg_tok),
            lambda: B.moe_mxfp8_quantize_tokens(d, self.dgu8, 2 * I, I, I, b.offsets, *self.du_tok),
            lambda: B.moe_grouped_gemm_gateup_wgrad_mxfp8(d, *self.x_tok, *self.dg_tok, *self.du_tok, self.dw8[1], self.dw8[2]),
        ]

    def results(self):
        return super().results() + [t.clone() for t in (*self.again, *self.static, self.dgu_fused, self.dh8, self.dgu8, self.dx8,
                                                        *self.dw8)]


# the last one: 2000 rows per expert, where the plain GEMMs run fixed-height tiles; the one before: the fused call swapped
@pytest.mark.parametrize("shape", SHAPES + [(1000, 256, 128, 8, 2), (4000, 128, 256, 4, 2)])
def test_steps_that_follow_one_another_directly(shape):
    from paper_2606_26453_b200 import binding as B
    B.load_library()
    step = _EveryCall(B, *shape)
    sets = [_inputs(B, *shape, seed) for seed in (1, 2)]
    want = []
    for v in sets:
        for call in step.calls(v):
            call()
            torch.cuda.synchronize()
        want.append(step.results())
    assert all(torch.equal(a, b) for a, b in zip(want[0][13:18], want[0][18:23]))   # the two route-permutes agree
    for last in range(2, 8):                              # steps of alternating inputs, then a look at the last one's results
        for i in range(last + 1):
            for call in step.calls(sets[i % 2]):
                call()
        for k, (a, b) in enumerate(zip(step.results(), want[last % 2])):
            assert torch.equal(a, b), (last, k)
    stream = torch.cuda.Stream()
    stream.wait_stream(torch.cuda.current_stream())
    graphs = []
    for first in (0, 1):                                  # two steps per graph
        graphs.append(torch.cuda.CUDAGraph())
        with torch.cuda.graph(graphs[-1], stream=stream):
            for v in (sets[first], sets[1 - first]):
                for call in step.calls(v):
                    call()
    for first in (0, 1, 1, 0):
        graphs[first].replay()
        graphs[first].replay()
        for k, (a, b) in enumerate(zip(step.results(), want[1 - first])):
            assert torch.equal(a, b), ("graph", first, k)
    assert B.moe_device_status() == 0
