"""Importance of short prompts, whose scores stay in tensor memory between the passes (one launch, a cluster of CTAs per
head), at the edges of its tiles, of its two sizes and of the range it serves, against softmax in fp64.  Products of bf16 are
exact in fp32; a score of D terms carries at most D 2^-24 of the sum of its terms' absolute values, which for these unit
normal inputs moves an exponent by less than 2e-6; ex2 adds 2^-22 and the sums over 64 queries less: 2e-5 of the largest
importance covers all of it by a factor of five."""
import pytest
import torch

import paper_2605_28640_b200 as rq

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("D,S", [(64, 64), (128, 16)])
@pytest.mark.parametrize("BH,T,W", [(1, 64, 64), (3, 65, 64), (1, 128, 1), (2, 129, 33), (1, 511, 64), (75, 513, 64), (2, 1000, 7), (40, 2048, 64),
                                    (300, 640, 64), (3, 4095, 64), (75, 4096, 64), (2, 4097, 64), (3, 5000, 40), (150, 5121, 64), (2, 8192, 64),
                                    (2, 8193, 64)])
def test_importance(BH, T, W, D, S):
    g = torch.Generator(device=DEV)
    g.manual_seed(T + W)
    cache = rq.Cache(1, BH, D, S, T, torch.bfloat16)
    k = torch.randn(1, T, BH, D, generator=g, device=DEV, dtype=torch.bfloat16)
    k[:, T // 2] = k[:, 0]                                        # equal keys in different tiles
    z = torch.zeros_like(k)
    rq.rq_build_cache(cache.handle, k, z, z)                      # zero gates: the cache holds the keys themselves
    qw = torch.randn(1, W, BH, D, generator=g, device=DEV, dtype=torch.bfloat16)
    scratch = torch.empty(rq.rq_snapkv_scratch_bytes(cache.handle), dtype=torch.uint8, device=DEV)
    idx = torch.empty(1, BH, W, dtype=torch.int32, device=DEV)
    imp = torch.full((1, BH, T), float("nan"), dtype=torch.float32, device=DEV)
    rq.rq_snapkv_select(cache.handle, qw, W, W, 0.0, idx, imp, scratch)
    torch.cuda.synchronize()
    assert rq.rq_device_status(cache.handle) == rq.RQ_OK
    for h in range(0, BH, max(1, BH // 6)):
        s = qw[0, :, h].double() @ k[0, :, h].double().T * D ** -0.5
        pos = torch.arange(T, device=DEV)
        s[pos[None, :] > (T - W + torch.arange(W, device=DEV))[:, None]] = float("-inf")
        want = torch.softmax(s, -1).sum(0)
        err = (imp[0, h].double() - want).abs().max().item()
        assert err <= 2e-5 * want.max().item(), f"head {h}: {err} of {want.max().item()}"
    if T // 2 < T - W:
        assert torch.equal(imp[0, :, 0], imp[0, :, T // 2])       # equal keys before the window: the same bits
