"""MoBA where the representatives' bf16 terms, and what any of 128 queries chose, do and do not find room in the scratch (behind the
masks, in what the lists would take: the first three budgets have room for neither, for the second only, for both): the lists are those of
a sort by (score, lower block first) either way, the attention is the same, and nothing behind the scratch is written."""
import numpy as np
import pytest
import torch

import paper_2605_28640_b200 as rq
from test_gpu_moba_route import expected

pytestmark = pytest.mark.gpu
DEV = "cuda"
BLOCK, S = 64, 16


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("T,K", [(64 * 64, 2), (64 * 64, 5), (64 * 64, 6), (64 * 130 + 1, 9), (64 * 130 + 1, 10), (64 * 513 + 7, 18), (64 * 513 + 7, 21)])
def test_room_for_the_terms(T, K, D, H=2):
    nb = -(-T // BLOCK)
    r = np.random.default_rng(T + K)
    levels = [r.permutation(np.arange(nb)) / 8.0 - 30.0, r.integers(-3, 4, nb) / 2.0]          # all different; runs of equal ones
    cache = rq.Cache(1, H, D, S, T, torch.bfloat16)
    k = torch.zeros(1, T, H, D, dtype=torch.bfloat16, device=DEV)
    for h in range(H):
        k[0, :, h, 0] = torch.tensor(np.repeat(levels[h], BLOCK)[:T], dtype=torch.bfloat16, device=DEV)
    levels = [k[0, ::BLOCK, h, 0].double().cpu().numpy() for h in range(H)]                     # as rounded
    rq.rq_build_cache(cache.handle, k, k, torch.zeros_like(k))    # zero gates: the cache holds the keys themselves
    q = torch.zeros(1, T, H, D, dtype=torch.bfloat16, device=DEV)
    q[..., 0] = 1.0
    n = rq.rq_moba_scratch_bytes(cache.handle, BLOCK, K)
    scratch = torch.full((n + 4096,), 0x5A, dtype=torch.uint8, device=DEV)
    o, o2 = torch.empty_like(q), torch.empty_like(q)
    lists = torch.full((1, H, T, K), -7, dtype=torch.int32, device=DEV)
    rq.rq_moba_prefill(cache.handle, q, BLOCK, K, 0.0, o, lists, None, scratch)
    rq.rq_moba_prefill(cache.handle, q, BLOCK, K, 0.0, o2, None, None, scratch)
    torch.cuda.synchronize()
    assert rq.rq_device_status(cache.handle) == rq.RQ_OK
    assert (scratch[n:] == 0x5A).all()
    assert torch.equal(o, o2)
    got = lists[0].cpu().numpy()
    for h in range(H):
        for own in range(nb):
            t0, t1 = own * BLOCK, min(T, (own + 1) * BLOCK)
            assert (got[h, t0:t1] == expected(levels[h], own, K)).all(), f"head {h}, block {own}"
