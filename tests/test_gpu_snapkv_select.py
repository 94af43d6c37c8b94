"""Selection of the retained positions over the sizes that take its different forms (one to eight CTAs per head, keys in
registers or read again), with many equal importances (keys from a handful of vectors) and with all different ones: index
for index the sort of the importances that the same call returns, equal importance to the lower position."""
import numpy as np
import pytest
import torch

import paper_2605_28640_b200 as rq

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("kinds", [1, 3, 0])
@pytest.mark.parametrize("BH,T,keeps", [(1, 100, (64, 65, 99)), (2, 1063, (64, 700)), (2, 1089, (65, 70)), (40, 2112, (130,)),
                                        (3, 4096, (66, 1024)), (3, 16449, (300, 16448)), (160, 5000, (1000,)),
                                        (2, 131136, (8192,)), (1, 140001, (70, 9000)), (310, 9000, (64, 2000))])
def test_index_for_index(BH, T, keeps, kinds, D=64):
    W = 64
    g = torch.Generator(device=DEV)
    g.manual_seed(T + kinds)
    cache = rq.Cache(1, BH, D, 64, T, torch.bfloat16)
    if kinds:
        table = torch.randn(kinds, D, generator=g, device=DEV, dtype=torch.bfloat16)
        k = table[torch.randint(kinds, (1, T, BH), generator=g, device=DEV)]
    else:
        k = torch.randn(1, T, BH, D, generator=g, device=DEV, dtype=torch.bfloat16)
    z = torch.zeros_like(k)
    rq.rq_build_cache(cache.handle, k, z, z)                      # zero gates: the cache holds the keys themselves
    del z
    qw = torch.randn(1, W, BH, D, generator=g, device=DEV, dtype=torch.bfloat16)
    scratch = torch.empty(rq.rq_snapkv_scratch_bytes(cache.handle), dtype=torch.uint8, device=DEV)
    for keep in keeps:
        idx = torch.full((1, BH, keep), -7, dtype=torch.int32, device=DEV)
        imp = torch.empty(1, BH, T, dtype=torch.float32, device=DEV)
        rq.rq_snapkv_select(cache.handle, qw, W, keep, 0.0, idx, imp, scratch)
        torch.cuda.synchronize()
        assert rq.rq_device_status(cache.handle) == rq.RQ_OK
        for h in range(0, BH, max(1, BH // 8)):
            x = imp[0, h, :T - W].cpu().numpy()
            best = np.lexsort((np.arange(T - W), -x))[:keep - W]
            want = np.concatenate([np.sort(best), np.arange(T - W, T)])
            assert np.array_equal(idx[0, h].cpu().numpy(), want), f"head {h}, keep {keep}"


@pytest.mark.parametrize("kinds", [3, 0])
@pytest.mark.parametrize("BH,T,keeps", [(9, 66000, (4000,)), (10, 66000, (64, 66000 - 1)), (32, 16449, (900,)), (32, 33000, (2000,)),
                                        (33, 8257, (900,)), (64, 16449, (1500,)), (64, 70000, (3000,)), (65, 8256, (700,)),
                                        (65, 8257, (64, 65, 700, 8257))])
def test_forms_by_heads(BH, T, keeps, kinds):
    """At the edges of the rule that gives a head one CTA, a cluster of two, four or eight, or the one-CTA form by digits."""
    test_index_for_index(BH, T, keeps, kinds)


@pytest.mark.parametrize("BH,T,keeps", [(5, 32833, (1000,)), (13, 65600, (64, 5000)), (14, 40000, (2000,))])
def test_clusters_of_eight(BH, T, keeps):
    """128 channels, few heads, keys that fill four to eight CTAs of 512 threads."""
    test_index_for_index(BH, T, keeps, 0, D=128)
