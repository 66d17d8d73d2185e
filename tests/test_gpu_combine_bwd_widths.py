"""Combine backward over the widths at which the number of threads per token changes (32, 64, 128, 256), with last blocks that are not
full, against the oracle; dtopk_w is a sum in fp32, held to what that gives (1e-5 of its norm)."""
import numpy as np
import pytest
import torch

from oracle import moe_oracle as O
from paper_2606_26453_b200 import workloads as W
from tests import helpers as Hh

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H", [64, 256, 320, 1024, 1280, 2048, 2880, 3520, 4096, 4160])
@pytest.mark.parametrize("T,K", [(1, 1), (7, 3), (13, 8), (5, 20), (451, 20), (601, 8), (2373, 2), (4745, 1)])   # from 451 on several tokens to a block
def test_widths(H, T, K):
    from paper_2606_26453_b200 import binding as B
    E, R = max(K, 4), T * K
    rng = np.random.default_rng(H + T)
    idx = np.stack([rng.permutation(E)[:K] for _ in range(T)]).astype(np.int32)
    p2r = O.permute_indices(idx, E)[3].astype(np.int32)
    dy, yp = (W.round_to_bf16(rng.standard_normal((n, H)).astype(np.float32)) for n in (T, R))
    w = rng.random((T, K), dtype=np.float32)
    d = B.dims(T, H, 64, E, K)
    dyp = torch.full((R + 1, H), float("nan"), dtype=torch.bfloat16, device="cuda")
    dw = torch.full((T + 1, K), float("nan"), dtype=torch.float32, device="cuda")
    B.moe_unpermute_combine_bwd(d, Hh.to_dev_bf16(dy), Hh.to_dev_bf16(yp), torch.from_numpy(w).cuda(), torch.from_numpy(p2r).cuda(), dyp[:R], dw[:T])
    only = torch.full((R, H), float("nan"), dtype=torch.bfloat16, device="cuda")
    B.moe_unpermute_combine_bwd(d, Hh.to_dev_bf16(dy), None, torch.from_numpy(w).cuda(), torch.from_numpy(p2r).cuda(), only, None)
    torch.cuda.synchronize()
    want, want_dw = O.unpermute_combine_bwd(dy, yp, w, p2r)
    Hh.assert_close(Hh.to_np64(dyp[:R]), want, "dY_perm", rel_fro=Hh.PER_CALL_FROBENIUS)
    Hh.assert_close(dw[:T].cpu().numpy().astype(np.float64), want_dw, "dtopk_w", rel_fro=1e-5, max_abs=1e-4)
    assert torch.equal(only, dyp[:R]) and bool(torch.isnan(dyp[R:]).all()) and bool(torch.isnan(dw[T:]).all())
