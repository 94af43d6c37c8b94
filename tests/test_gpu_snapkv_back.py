"""Importance of prompts that take two passes, the second from the last head, run and tile to the first: numbers of tiles that do
not fill the last run, heads and runs in one round of CTAs and (the last case: 1920) in several, a window of fewer than 64
queries, pages of both sizes; against softmax in fp64. The bound is that of the short prompts: a score of D terms carries at
most D 2^-24 of its terms' absolute values, ex2 2^-22, the sums less; 2e-5 of the largest importance."""
import pytest
import torch

import paper_2605_28640_b200 as rq

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("BH,T,W,S,D", [(1, 4097, 64, 16, 128), (5, 4225, 17, 64, 128), (2, 50001, 64, 16, 128), (127, 6001, 64, 64, 128),
                                        (9, 20000, 1, 16, 128), (5, 9001, 64, 16, 64), (320, 13000, 64, 16, 128)])
def test_importance(BH, T, W, S, D):
    g = torch.Generator(device=DEV)
    g.manual_seed(T + W)
    cache = rq.Cache(1, BH, D, S, T, torch.bfloat16)
    k = torch.randn(1, T, BH, D, generator=g, device=DEV, dtype=torch.bfloat16)
    k[:, T // 2] = k[:, 0]                                        # equal keys in different runs
    z = torch.zeros_like(k)
    rq.rq_build_cache(cache.handle, k, z, z)                      # zero gates: the cache holds the keys themselves
    qw = torch.randn(1, W, BH, D, generator=g, device=DEV, dtype=torch.bfloat16)
    scratch = torch.empty(rq.rq_snapkv_scratch_bytes(cache.handle), dtype=torch.uint8, device=DEV)
    idx = torch.empty(1, BH, W, dtype=torch.int32, device=DEV)
    imp = torch.full((1, BH, T), float("nan"), dtype=torch.float32, device=DEV)
    rq.rq_snapkv_select(cache.handle, qw, W, W, 0.0, idx, imp, scratch)
    torch.cuda.synchronize()
    assert rq.rq_device_status(cache.handle) == rq.RQ_OK
    assert not imp.isnan().any()                                  # every tile of every head was written
    for h in sorted({0, BH // 3, BH // 2, max(0, BH - 2), BH - 1}):
        s = qw[0, :, h].double() @ k[0, :, h].double().T * D ** -0.5
        pos = torch.arange(T, device=DEV)
        s[pos[None, :] > (T - W + torch.arange(W, device=DEV))[:, None]] = float("-inf")
        want = torch.softmax(s, -1).sum(0)
        err = (imp[0, h].double() - want).abs().max().item()
        assert err <= 2e-5 * want.max().item(), f"head {h}: {err} of {want.max().item()}"
    assert torch.equal(imp[0, :, 0], imp[0, :, T // 2])           # equal keys before the window: the same bits
