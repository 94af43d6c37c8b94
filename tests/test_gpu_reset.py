"""Emptying a cache: the recurrence state is zero and the same prompt gives the same bits again, for the smallest state, for
one whose 16-byte pieces are no multiple of the clearing kernel's share, and for a large one."""
import pytest
import torch

import paper_2605_28640_b200 as rq

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("B,H,D,T", [(1, 1, 64, 17), (1, 3, 64, 300), (5, 7, 128, 65), (16, 32, 128, 40)])
def test_reset(B, H, D, T):
    g = torch.Generator(device=DEV)
    g.manual_seed(T)
    cache = rq.Cache(B, H, D, 16, T, torch.bfloat16)
    k, v, gate = (torch.rand(B, T, H, D, generator=g, device=DEV).to(torch.bfloat16) for _ in range(3))
    rq.rq_build_cache(cache.handle, k, v, gate)
    torch.cuda.synchronize()
    kv, state = cache.kv.clone(), cache.state.clone()
    rq.rq_cache_reset(cache.handle)
    torch.cuda.synchronize()
    assert not cache.state.any()
    rq.rq_build_cache(cache.handle, k, v, gate)
    torch.cuda.synchronize()
    assert rq.rq_device_status(cache.handle) == rq.RQ_OK
    assert torch.equal(cache.state, state) and torch.equal(cache.kv, kv)
