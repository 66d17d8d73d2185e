"""Route-permute on both sides of the number of pairs (2048) from which a histogram launch goes before the ranking, and of the number of
sums over all blocks (1.5 million) from which a scan launch goes in between: indices, offsets, counts and rows against the oracle, bit for
bit, with expert ids outside [0, E) among them."""
import numpy as np
import pytest
import torch

from oracle import moe_oracle as O
from paper_2606_26453_b200 import workloads as W
from tests import helpers as Hh

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,K,E", [(1, 1, 1), (5, 3, 1024), (2047, 1, 3), (2048, 1, 128), (2049, 1, 128), (64, 32, 40), (65, 32, 40), (682, 3, 7),
                                   (683, 3, 7), (14336, 1, 128), (14337, 1, 128), (4099, 8, 1000), (1024, 10, 300), (33000, 1, 64)])
@pytest.mark.parametrize("invalid", [False, True])
def test_few_pairs(T, K, E, invalid):
    check(T, K, E, invalid)


@pytest.mark.parametrize("T,K,E", [(8192, 1, 183), (8192, 1, 184), (36485, 7, 8)])
@pytest.mark.parametrize("invalid", [False, True])
def test_many_pairs(T, K, E, invalid):
    check(T, K, E, invalid)


@pytest.mark.parametrize("T,K,E", [(3000, 2, 40), (32768, 8, 128)])   # two launches, three
def test_inputs_that_change_from_call_to_call(T, K, E):
    """Two routings and inputs by turns through the same buffers, nothing waited for in between: the ranking kernel, which reads both
    before it waits for the kernel before it, sees those of its own call."""
    from paper_2606_26453_b200 import binding as B
    H, rng = 64, np.random.default_rng(T)
    idx = [torch.from_numpy(rng.integers(0, n, size=(T, K)).astype(np.int32)).cuda() for n in (E, E // 2)]
    X = [Hh.to_dev_bf16(W.round_to_bf16(rng.standard_normal((T, H), dtype=np.float32))) for _ in idx]
    d, i32 = B.dims(T, H, 64, E, K), dict(dtype=torch.int32, device="cuda")
    ws = torch.empty(B.moe_permute_workspace_bytes(d), dtype=torch.uint8, device="cuda")
    xp, counts, offsets, r2p, p2r = torch.empty((T * K, H), dtype=torch.bfloat16, device="cuda"), *(torch.empty(n, **i32) for n in (E, E + 1, T * K, T * K))
    live_x, live_idx, got = torch.empty_like(X[0]), torch.empty_like(idx[0]), []
    for i in range(40):
        live_x.copy_(X[i % 2])
        live_idx.copy_(idx[i % 2])
        B.moe_permute(d, live_x, live_idx, xp, counts, offsets, r2p, p2r, ws)
        got.append([t.clone() for t in (xp, r2p, offsets)])
    torch.cuda.synchronize()
    assert B.moe_device_status() == 0
    for i, (xp_i, r2p_i, offsets_i) in enumerate(got):
        flat = idx[i % 2].flatten().long()
        order = torch.argsort(flat, stable=True)
        assert torch.equal(r2p_i.long(), order), i
        assert torch.equal(offsets_i[1:].long(), torch.bincount(flat, minlength=E).cumsum(0)), i
        assert torch.equal(xp_i, X[i % 2][order // K]), i


def check(T, K, E, invalid):
    from paper_2606_26453_b200 import binding as B
    H, R, guard = 192, T * K, 16
    rng = np.random.default_rng(R + E)
    idx = rng.integers(0, E, size=(T, K)).astype(np.int32)
    flat = idx.reshape(-1)
    if invalid:
        flat[rng.choice(R, size=max(1, R // 50), replace=False)] = rng.choice(np.array([-1, E, 2 ** 30], dtype=np.int32))
    X = W.round_to_bf16(rng.standard_normal((T, H), dtype=np.float32))
    i32 = lambda n: torch.full((n + guard,), -7, dtype=torch.int32, device="cuda")
    counts, offsets, r2p, p2r = i32(E), i32(E + 1), i32(R), i32(R)
    xp = torch.full((R + guard, H), float("nan"), dtype=torch.bfloat16, device="cuda")
    d = B.dims(T, H, 128, E, K)
    ws = torch.empty(max(B.moe_permute_workspace_bytes(d), 16), dtype=torch.uint8, device="cuda")
    B.moe_permute(d, Hh.to_dev_bf16(X), torch.from_numpy(idx).cuda(), xp[:R], counts[:E], offsets[:E + 1], r2p[:R], p2r[:R], ws)
    torch.cuda.synchronize()
    assert B.moe_device_status() == (7 if invalid else 0)
    good = np.flatnonzero((flat >= 0) & (flat < E))
    order = good[np.argsort(flat[good], kind="stable")]              # the stable sort of the valid pairs
    n = order.size
    want_counts = np.bincount(flat[good], minlength=E)
    assert np.array_equal(counts[:E].cpu().numpy(), want_counts)
    assert np.array_equal(offsets[:E + 1].cpu().numpy(), np.concatenate([[0], np.cumsum(want_counts)]))
    assert np.array_equal(r2p[:n].cpu().numpy(), order)
    assert np.array_equal(p2r[:R].cpu().numpy()[order], np.arange(n))
    assert np.array_equal(Hh.to_np64(xp[:n]), X[order // K].astype(np.float64))
    if not invalid:
        assert all(np.array_equal(a, b) for a, b in zip((r2p[:R].cpu().numpy(), p2r[:R].cpu().numpy()), O.permute_indices(idx, E)[2:4]))
    for t in (counts[E:], offsets[E + 1:], r2p[n:], p2r[R:]):
        assert bool((t == -7).all())
    assert bool(torch.isnan(xp[n:]).all())
