"""The decode step as one launch of a cluster per head (rq_cache.reserved[2] = 16) where it can go wrong: page counts at the
edges of its selection (pages ranked against each other up to 96, buckets beyond, rows of 256 pages, 2048 at most), runs of
equal scores with the cut inside, forced pages that fill the budget, budgets that keep everything, one head and more heads
than clusters of eight find room for, a first token, a token that opens a page; the staged comparison with the oracle on
drawn inputs, and index for index on planted page bounds, whose scores are exact."""
import numpy as np
import pytest
import torch

import paper_2605_28640_b200 as rq
from paper_2605_28640_b200 import workloads as wl

from test_gpu_parity import run_case

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("B,H,D,S,T,K,dtype", [
    (1, 1, 128, 16, 1, 1, torch.bfloat16), (1, 3, 64, 16, 17, 1, torch.float32), (2, 2, 128, 64, 65, 2, torch.bfloat16),
    (1, 4, 64, 16, 1000, 16, torch.float32), (1, 5, 128, 16, 1536, 12, torch.bfloat16), (1, 2, 128, 16, 1553, 97, torch.bfloat16),
    (1, 2, 128, 16, 1600, 200, torch.float32), (1, 2, 64, 64, 16500, 40, torch.bfloat16), (1, 1, 128, 16, 32766, 128, torch.bfloat16),
    (3, 50, 64, 16, 700, 9, torch.bfloat16), (9, 33, 64, 64, 400, 3, torch.bfloat16), (1, 32, 128, 64, 4090, 16, torch.bfloat16)])
def test_against_the_oracle(B, H, D, S, T, K, dtype):
    w = wl.Workload("cluster", B=B, H=H, D=D, T=T, S=S, dtype=dtype, seed=T + K)
    heads = sorted({(0, 0), (B - 1, H - 1), (B // 2, H // 2)})
    run_case(w, T - 1, steps=3, heads=heads, budget=K, path=16, want_launches=1)


def levels_of(kind, P, r):
    if kind == "distinct":
        x = r.permutation(np.concatenate([s * (128 + np.arange(128)) * 2.0 ** e for e in range(8) for s in (-1, 1)]))[:P]
    elif kind == "runs":
        x = r.integers(-2, 3, P).astype(np.float64)
    elif kind == "equal":
        x = np.full(P, 0.5)
    else:                                                        # one far outlier: everything else lands in one bucket
        x = 1.0 + r.integers(0, 100, P) / 128.0
        x[P // 2] = -20000.0
    return x


@pytest.mark.parametrize("kind", ["distinct", "runs", "equal", "outlier"])
@pytest.mark.parametrize("P,K", [(1, 1), (2, 1), (33, 5), (96, 40), (97, 40), (128, 3), (257, 100), (1000, 62), (2048, 2), (2048, 500)])
@pytest.mark.parametrize("ns,nl", [(1, 1), (0, 0), (3, 2)])
def test_lists_on_planted_bounds(P, K, ns, nl, kind):
    S, D, H = 16, 64, 3
    c = rq.Cache(1, H, D, S, P * S, torch.bfloat16, n_sink_pages=ns, n_local_pages=nl, max_budget_pages=K)
    c.handle.reserved[2] = 16
    c.kv.zero_()
    c.meta.zero_()
    r = np.random.default_rng(P * 7 + K)
    lv = np.stack([levels_of(kind, P, r) for _ in range(H)])
    c.meta_view()[0, :, :, 1, 0] = torch.tensor(lv, dtype=torch.bfloat16, device=DEV)       # channel 0's maximum; the minimum likewise
    c.meta_view()[0, :, :, 0, 0] = torch.tensor(lv, dtype=torch.bfloat16, device=DEV)
    c.handle.len = P * S - 1                                      # the last page lacks one slot, which the step fills
    q = torch.zeros(1, H, D, dtype=torch.bfloat16, device=DEV)
    q[..., 0] = 1.0
    z = torch.zeros_like(q)
    o = torch.empty_like(q)
    idx = torch.full((1, H, K), -7, dtype=torch.int32, device=DEV)
    assert rq.rq_decode_step_launches(c.handle, K) == 1
    rq.rq_decode_step(c.handle, q, z, z, z, K, 0.0, o, idx)
    torch.cuda.synchronize()
    score = c.meta_view()[0, :, :, 1, 0].double().cpu().numpy()   # (the newest page's maximum has met the new key, a zero)
    n = min(K, P)
    s = min(ns, n)
    loc = min(nl, n - s, P - s)
    for h in range(H):
        cand = np.arange(s, P - loc)
        best = cand[np.lexsort((cand, -score[h, cand]))][:n - s - loc]
        want = np.sort(np.concatenate([np.arange(s), best, np.arange(P - loc, P)]))
        got = idx[0, h].cpu().numpy()
        assert np.array_equal(got[:n], want) and (got[n:] == -1).all(), f"head {h}: {got} instead of {want}"
