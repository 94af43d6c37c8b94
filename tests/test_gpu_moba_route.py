"""MoBA routing on the tensor cores where it can go wrong: block counts at the edges of a product (64 blocks), of what
tensor memory holds at once (512 blocks: one panel, two panels), runs of equal scores longer than what is ranked
directly with the cut inside and at the end of a run, a bucket that needs finer cuts, and the smallest budget.

Keys are planted so that the block means are exactly representable and two blocks' scores are either equal or far
apart; the expected list is then a plain sort by (score, lower block first), index for index, for every query."""
import numpy as np
import pytest
import torch

import paper_2605_28640_b200 as rq

pytestmark = pytest.mark.gpu
DEV = "cuda"


def route(levels, T, D, block, K):
    """levels: the value of channel 0 of every block's keys; queries have 1 in channel 0 and nothing else.  Also that the
    attention is the same whether the caller asks for the lists or not (bit masks then, where they fit)."""
    nb = -(-T // block)
    cache = rq.Cache(1, 1, D, 16, T, torch.bfloat16)
    k = torch.zeros(1, T, 1, D, dtype=torch.bfloat16, device=DEV)
    k[0, :, 0, 0] = torch.tensor(np.repeat(levels, block)[:T], dtype=torch.bfloat16, device=DEV)
    z = torch.zeros_like(k)
    v = torch.randn(1, T, 1, D, device=DEV, dtype=torch.bfloat16)
    rq.rq_build_cache(cache.handle, k, v, z)                      # zero gates: the cache holds the keys themselves
    q = torch.zeros(1, T, 1, D, dtype=torch.bfloat16, device=DEV)
    q[..., 0] = 1.0
    o = torch.empty_like(q)
    blocks = torch.full((1, 1, T, K), -7, dtype=torch.int32, device=DEV)
    scratch = torch.empty(rq.rq_moba_scratch_bytes(cache.handle, block, K), dtype=torch.uint8, device=DEV)
    rq.rq_moba_prefill(cache.handle, q, block, K, 0.0, o, blocks, None, scratch)
    torch.cuda.synchronize()
    assert rq.rq_device_status(cache.handle) == rq.RQ_OK
    o2 = torch.empty_like(q)
    rq.rq_moba_prefill(cache.handle, q, block, K, 0.0, o2, None, None, scratch)
    assert torch.equal(o, o2)
    return blocks[0, 0].cpu().numpy(), nb


def expected(levels, own, K):
    if K >= own + 1:
        want = np.arange(own + 1)
    else:
        cand = np.arange(1, own)
        best = cand[np.lexsort((cand, -levels[cand]))][: K - 2]
        want = np.sort(np.concatenate([[0], best, [own]]))
    return np.concatenate([want, np.full(K - len(want), -1)]).astype(np.int64)


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("T,K", [(64 * 64, 16), (64 * 17, 4), (64 * 33 + 5, 6), (64 * 48 + 1, 47), (64 * 65 + 1, 9), (64 * 257, 40), (64 * 512, 100), (64 * 513 + 7, 33), (64 * 130, 2)])
@pytest.mark.parametrize("kind", ["distinct", "runs", "equal", "clustered"])
def test_lists_at_the_edges(kind, T, K, D):
    block = 64
    nb = -(-T // block)
    r = np.random.default_rng(T + K)
    if kind == "distinct":                                        # bf16 values of one sign change, all different for < 1000 blocks
        levels = r.permutation(np.concatenate([-(128 + np.arange(128)) * 2.0 ** e for e in range(4)] +
                                              [(128 + np.arange(128)) * 2.0 ** e for e in range(4)]))[:nb]
    elif kind == "runs":                                          # five values: runs of a fifth of the blocks
        levels = r.integers(-2, 3, nb).astype(np.float64)
    elif kind == "equal":
        levels = np.full(nb, 0.5)
    else:                                                         # one far outlier: everything else lands in one bucket
        levels = 1.0 + r.integers(0, 100, nb) / 128.0
        levels[1] = -20000.0
    got, _ = route(levels, T, D, block, K)
    for own in range(nb):
        want = expected(levels, own, K)
        t0, t1 = own * block, min(T, (own + 1) * block)
        bad = np.nonzero((got[t0:t1] != want).any(axis=1))[0]
        assert len(bad) == 0, f"block {own}: query {t0 + bad[0]}: {got[t0 + bad[0]]} instead of {want}"
