"""MoBA on bf16 caches with keys whose scores overflow or are infinite: a query that did not choose their block does not
notice, in the routing (an infinite mean scores +inf or -inf by the sign of the query) and in the attention."""
import numpy as np
import pytest
import torch

import paper_2605_28640_b200 as rq

pytestmark = pytest.mark.gpu
DEV = "cuda"
BLOCK, H = 64, 1


def run(k, v, q, K):
    T, D = k.shape[1], k.shape[3]
    cache = rq.Cache(1, H, D, 16, T, torch.bfloat16)
    rq.rq_build_cache(cache.handle, k, v, torch.zeros_like(k))    # zero gates: the cache holds k and v themselves
    o = torch.empty_like(q)
    blocks = torch.empty(1, H, T, K, dtype=torch.int32, device=DEV)
    scratch = torch.empty(rq.rq_moba_scratch_bytes(cache.handle, BLOCK, K), dtype=torch.uint8, device=DEV)
    rq.rq_moba_prefill(cache.handle, q, BLOCK, K, 0.0, o, blocks, None, scratch)
    o2 = torch.empty_like(q)
    rq.rq_moba_prefill(cache.handle, q, BLOCK, K, 0.0, o2, None, None, scratch)
    torch.cuda.synchronize()
    assert rq.rq_device_status(cache.handle) == rq.RQ_OK
    assert torch.equal(o.view(torch.int16), o2.view(torch.int16))
    return o[0, :, 0], blocks[0, 0]


def reference(k, v, q, blocks, t):
    """Softmax in fp64 of query t over the positions up to t of its blocks."""
    pos = torch.cat([torch.arange(int(b) * BLOCK, int(b) * BLOCK + BLOCK, device=DEV) for b in blocks[t] if b >= 0])
    pos = pos[pos <= t]
    s = (k[0, pos, 0].double() @ q[0, t, 0].double()) * q.shape[-1] ** -0.5
    return torch.softmax(s, 0) @ v[0, pos, 0].double()


def inputs(T, D, seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return [torch.randn(1, T, H, D, generator=g, device=DEV, dtype=torch.bfloat16) for _ in range(3)]


@pytest.mark.parametrize("D", [64, 128])
def test_scores_that_overflow_stay_with_those_who_chose_them(D):
    """Block 1 holds a pair of keys whose scores are +inf and -inf and whose mean is not large; of neighbouring queries, lanes
    of one warp, every other one chooses block 1 and the rest block 2."""
    T, K = 8 * BLOCK, 3
    k, v, q = inputs(T, D, D)
    k[..., :2] = 0
    k[0, 70, 0, 0], k[0, 71, 0, 0] = 2e38, -2e38
    k[0, BLOCK:2 * BLOCK, 0, 1], k[0, 2 * BLOCK:3 * BLOCK, 0, 1] = 4.0, -4.0
    q[..., 0] = 4.0
    q[0, ::2, 0, 1], q[0, 1::2, 0, 1] = 8.0, -8.0
    o, blocks = run(k, v, q, K)
    for t in range(4 * BLOCK, T):
        assert int(blocks[t, 1]) == (1 if t % 2 == 0 else 2)
    top = v.abs().max().item()
    for t in range(4 * BLOCK + 1, T, 2):
        # weights and output rounded to bf16, as everywhere: 2^-8 of the largest value, a tenth on top for the rest
        assert (o[t].double() - reference(k, v, q, blocks, t)).abs().max().item() <= 1.1 * 2 ** -8 * top, t


@pytest.mark.parametrize("D", [64, 128])
def test_scores_of_minus_infinity_first(D):
    """Every score of the first block is -inf: it weighs nothing, and the output is that of the blocks behind it."""
    T, K = 4 * BLOCK, 4
    k, v, q = inputs(T, D, D + 1)
    k[0, :BLOCK, 0, 0] = -3e38
    k[0, BLOCK:, 0, 0] = 0
    q[..., 0] = 8.0
    o, blocks = run(k, v, q, K)
    top = v.abs().max().item()
    for t in range(BLOCK, T):
        assert (o[t].double() - reference(k, v, q, blocks, t)).abs().max().item() <= 1.1 * 2 ** -8 * top, t


@pytest.mark.parametrize("D,T,K", [(64, 12 * BLOCK, 4), (128, 12 * BLOCK, 4), (64, 70 * BLOCK, 12)])
def test_infinite_means(D, T, K):
    """A block whose mean is infinite in channel 0 scores +inf or -inf by the sign of the query's channel 0; the others as
    planted."""
    nb = T // BLOCK
    r = np.random.default_rng(T)
    levels = r.permutation(np.arange(nb)) / 4.0                   # exact in bf16 and so are the means
    k, v, q = (torch.zeros(1, T, H, D, dtype=torch.bfloat16, device=DEV) for _ in range(3))
    k[0, :, 0, 1] = torch.tensor(np.repeat(levels, BLOCK), dtype=torch.bfloat16, device=DEV)
    inf_block = 3
    k[0, inf_block * BLOCK + 5:inf_block * BLOCK + 7, 0, 0] = 3e38    # the sum of the two overflows
    q[0, ::2, 0, 0], q[0, 1::2, 0, 0] = 0.5, -0.5
    q[..., 1] = 1.0
    for c in range(2, D):
        q[..., c] = 0.25
    _, blocks = run(k, v, q, K)
    got = blocks.cpu().numpy()
    for t in range(T):
        own = t // BLOCK
        if K >= own + 1:
            want = np.arange(own + 1)
        else:
            sc = levels.copy()
            sc[inf_block] = np.inf if t % 2 == 0 else -np.inf
            cand = np.arange(1, own)
            best = cand[np.lexsort((cand, -sc[cand]))][:K - 2]
            want = np.sort(np.concatenate([[0], best, [own]]))
        want = np.concatenate([want, np.full(K - len(want), -1)])
        assert np.array_equal(got[t], want), f"query {t}: {got[t]} instead of {want}"
