"""The combined backward calls, in which the weight gradient may run beside the data gradient before it, against the separate calls:
the same bits, also where the weight gradient goes over the data gradient's own weights (then one after the other)."""
import pytest
import torch

from tests import helpers as Hh

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("in_place", [False, True])
@pytest.mark.parametrize("counts,H,I", [([64] * 8, 256, 512), ([1], 64, 64), ([3, 0, 130], 192, 320),
                                        ([5200, 5300], 256, 512)])      # more tiles than the chip takes at once: always one after the other
def test_combined_calls(counts, H, I, in_place):
    from paper_2606_26453_b200 import binding as B
    cfg, host = Hh.ragged_workload(counts, K=1, H=H, I=I, seed=3)
    dev = Hh.device_workload(host)
    b = Hh.run_cuda_layer(dev, cfg.E)
    B.moe_grouped_gemm_down_dgrad(b.d, b.dy_perm, dev["W_down"], b.offsets, b.dh_act)
    B.moe_grouped_gemm_down_wgrad(b.d, b.h_act, b.dy_perm, b.offsets, b.dw_down)
    B.moe_swiglu_bwd(b.d, b.dh_act, b.gu, b.dgu)
    B.moe_grouped_gemm_gateup_dgrad(b.d, b.dgu, dev["W_gate"], dev["W_up"], b.offsets, b.dx_perm)
    B.moe_grouped_gemm_gateup_wgrad(b.d, b.x_perm, b.dgu, b.offsets, b.dw_gate, b.dw_up)
    torch.cuda.synchronize()
    outs = ("dh_act", "dgu", "dx_perm", "dw_down", "dw_gate", "dw_up")
    want = {k: getattr(b, k).clone() for k in outs}
    for _ in range(10):
        w = {k: dev[k].clone() for k in ("W_gate", "W_up", "W_down")}
        got = {k: torch.full_like(want[k], float("nan")) for k in outs}
        if in_place:
            got["dw_down"], got["dw_gate"], got["dw_up"] = w["W_down"], w["W_gate"], w["W_up"]
        B.moe_grouped_gemm_down_bwd(b.d, b.dy_perm, b.h_act, w["W_down"], b.offsets, got["dh_act"], got["dw_down"])
        B.moe_grouped_gemm_gateup_swiglu_bwd(b.d, got["dh_act"], b.gu, b.x_perm, w["W_gate"], w["W_up"], b.offsets, got["dgu"],
                                             got["dx_perm"], got["dw_gate"], got["dw_up"])
        copies = [got[k].clone() for k in outs]        # a kernel of another kind right behind
        torch.cuda.synchronize()
        for k, c in zip(outs, copies):
            assert torch.equal(c, want[k]), k
    assert B.moe_device_status() == 0


def test_inputs_that_change_from_call_to_call():
    """Steps of two workloads by turns through the same buffers, nothing waited for in between: the routing, the packed rows and the
    gradients that a weight gradient reads without waiting for the kernel before it are those of its own step."""
    from paper_2606_26453_b200 import binding as B
    H, I = 256, 512
    hosts = [Hh.ragged_workload(c, K=1, H=H, I=I, seed=s) for c, s in (([64] * 8, 41), ([130, 0, 3, 200, 64, 17, 97, 1], 43))]
    (cfg, _), E = hosts[0], 8
    devs = [Hh.device_workload(h) for _, h in hosts]
    outs = ("y", "dx", "dtopk_w", "dw_gate", "dw_up", "dw_down")
    b = B.alloc_layer_buffers(cfg.T, H, I, E, 1)

    def step(w):
        B.layer_forward(b, w["X"], w["topk_idx"], w["topk_w"], w["W_gate"], w["W_up"], w["W_down"])
        B.layer_backward(b, w["dY"], w["topk_w"], w["W_gate"], w["W_up"], w["W_down"])
        return {k: getattr(b, k).clone() for k in outs}

    want = []
    for w in devs:
        Hb = Hh.run_cuda_layer(w, E)      # buffers of its own
        B.moe_grouped_gemm_down_wgrad(Hb.d, Hb.h_act, Hb.dy_perm, Hb.offsets, Hb.dw_down)
        B.moe_grouped_gemm_gateup_wgrad(Hb.d, Hb.x_perm, Hb.dgu, Hb.offsets, Hb.dw_gate, Hb.dw_up)
        torch.cuda.synchronize()
        want.append({k: getattr(Hb, k).clone() for k in outs})
    live = {k: torch.empty_like(v) for k, v in devs[0].items()}
    got = []
    for i in range(40):
        for k, v in live.items():
            v.copy_(devs[i % 2][k])
        got.append(step(live))
    torch.cuda.synchronize()
    assert B.moe_device_status() == 0
    for i, g in enumerate(got):
        for k in outs:
            assert torch.equal(g[k], want[i % 2][k]), (i, k)
