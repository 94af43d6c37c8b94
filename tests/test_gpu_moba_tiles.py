"""MoBA attention where a CTA takes several tiles of queries one after the other (more tiles than SMs): prompts whose last tile has one
accumulator only, a ragged end, choices that come as unions, as masks and as lists, blocks of one chunk and of two; against softmax in fp64
at sampled queries of every head.  Weights and output are rounded to bf16: 2^-8 of the largest value, a tenth on top for the rest."""
import pytest
import torch

import paper_2605_28640_b200 as rq

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("H,T,block,K", [(40, 1100, 64, 4), (10, 4225, 64, 2), (300, 257, 64, 3), (60, 900, 128, 2), (160, 128, 64, 2)])
def test_several_tiles_to_a_cta(H, T, block, K, D):
    g = torch.Generator(device=DEV)
    g.manual_seed(T)
    k, v, q = (torch.randn(1, T, H, D, generator=g, device=DEV, dtype=torch.bfloat16) for _ in range(3))
    cache = rq.Cache(1, H, D, 16, T, torch.bfloat16)
    rq.rq_build_cache(cache.handle, k, v, torch.zeros_like(k))    # zero gates: the cache holds k and v themselves
    scratch = torch.empty(rq.rq_moba_scratch_bytes(cache.handle, block, K), dtype=torch.uint8, device=DEV)
    o, o2 = torch.full_like(q, float("nan")), torch.full_like(q, float("nan"))
    lists = torch.empty(1, H, T, K, dtype=torch.int32, device=DEV)
    rq.rq_moba_prefill(cache.handle, q, block, K, 0.0, o, None, None, scratch)
    rq.rq_moba_prefill(cache.handle, q, block, K, 0.0, o2, lists, None, scratch)
    torch.cuda.synchronize()
    assert rq.rq_device_status(cache.handle) == rq.RQ_OK
    assert torch.equal(o.view(torch.int16), o2.view(torch.int16)) and not o.isnan().any()
    top = v.abs().max().item()
    pos = torch.arange(T, device=DEV)
    for t in sorted({0, 63, 64, min(T - 1, 127), min(T - 1, 128), T // 2, T - 2, T - 1}):
        own = lists[0, :, t].long()                               # [H][K]
        seen = ((pos // block)[None, :, None] == own[:, None, :]).any(-1) & (pos <= t)
        s = torch.einsum("hd,thd->ht", q[0, t].double(), k[0].double()) * D ** -0.5
        want = torch.einsum("ht,thd->hd", torch.softmax(s.masked_fill(~seen, float("-inf")), -1), v[0].double())
        assert (o[0, t].double() - want).abs().max().item() <= 1.1 * 2 ** -8 * top, t
