"""MoBA attention of prompts whose keys and values are worked on in sets of heads (more than 96 MB of them): a first set that is
not full, full sets only, one head more than a set holds, a last tile of queries that is not full; every tile of every head is
looked at.  And of scores that exceed those of the chunks before by tens and hundreds of powers of two: in one block only, far from
the query, chosen by some queries of a warp and not by others.

Bound: the weights are rounded to bf16 (2^-9 of each) and so is the output (2^-9 of it), together at most 2^-8 of the
largest value; a tenth on top for the fp32 sums and the scores."""
import pytest
import torch

import paper_2605_28640_b200 as rq

pytestmark = pytest.mark.gpu
DEV = "cuda"
BLOCK = 64


def attend(k, v, q, K):
    _, T, H, D = k.shape
    cache = rq.Cache(1, H, D, 16, T, torch.bfloat16)
    rq.rq_build_cache(cache.handle, k, v, torch.zeros_like(k))    # zero gates: the cache holds k and v themselves
    o = torch.full_like(q, float("nan"))                         # what no CTA writes stays NaN
    blocks = torch.empty(1, H, T, K, dtype=torch.int32, device=DEV)
    scratch = torch.empty(rq.rq_moba_scratch_bytes(cache.handle, BLOCK, K), dtype=torch.uint8, device=DEV)
    rq.rq_moba_prefill(cache.handle, q, BLOCK, K, 0.0, o, blocks, None, scratch)
    torch.cuda.synchronize()
    assert rq.rq_device_status(cache.handle) == rq.RQ_OK
    return o, blocks


def check(k, v, q, o, blocks, h, t):
    pos = torch.cat([torch.arange(int(b) * BLOCK, int(b) * BLOCK + BLOCK, device=DEV) for b in blocks[0, h, t] if b >= 0])
    pos = pos[pos <= t]
    s = (k[0, pos, h].double() @ q[0, t, h].double()) * q.shape[-1] ** -0.5
    want = torch.softmax(s, 0) @ v[0, pos, h].double()
    err = (o[0, t, h].double() - want).abs().max().item()
    assert err <= 1.1 * 2 ** -8 * v[0, pos, h].abs().max().item(), (h, t, err)


def check_rows(k, v, q, o, blocks, h, t):
    """The positions `t` (a tensor) of a head at once."""
    pos = (blocks[0, h, t].long()[:, :, None] * BLOCK + torch.arange(BLOCK, device=DEV)).flatten(1)
    hidden = (blocks[0, h, t] < 0).repeat_interleave(BLOCK, 1) | (pos > t[:, None])
    pos = pos.clamp(0, k.shape[1] - 1)
    s = torch.einsum("npd,nd->np", k[0, :, h][pos].double(), q[0, t, h].double()) * q.shape[-1] ** -0.5
    vs = v[0, :, h][pos].double()
    want = torch.einsum("np,npd->nd", torch.softmax(s.masked_fill(hidden, float("-inf")), 1), vs)
    err = (o[0, t, h].double() - want).abs().amax(1)
    top = vs.masked_fill(hidden[:, :, None], 0).abs().amax((1, 2))
    assert (err <= 1.1 * 2 ** -8 * top).all(), (h, t[err > 1.1 * 2 ** -8 * top].tolist())


@pytest.mark.parametrize("H,T,D,K", [(40, 14001, 128, 12), (28, 14001, 128, 8), (14, 14001, 128, 8), (15, 13700, 128, 8), (33, 40961, 64, 20)])
def test_sets_of_heads(H, T, D, K):
    g = torch.Generator(device=DEV)
    g.manual_seed(T)
    k, v, q = (torch.randn(1, T, H, D, generator=g, device=DEV, dtype=torch.bfloat16) for _ in range(3))
    q *= 2
    o, blocks = attend(k, v, q, K)
    assert not torch.isnan(o).any()
    for h in range(H):
        t = torch.arange(0, T, 256, device=DEV)                   # a position of every tile of 256
        t = torch.cat([(t + (h * 37 + t // 256 * 101) % 256).clamp(max=T - 1), torch.tensor([63, 64, T // 2, T - 2, T - 1], device=DEV)])
        check_rows(k, v, q, o, blocks, h, t)


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("height", [30.0, 34.0, 120.0, 300.0])
def test_one_block_far_above_the_own_chunk(height, D):
    """Scores of about `height` powers of two in a block that every other query chooses, those of the other blocks around zero."""
    T, K, H = 10 * BLOCK, 3, 1
    g = torch.Generator(device=DEV)
    g.manual_seed(D)
    k, v, q = (torch.randn(1, T, H, D, generator=g, device=DEV, dtype=torch.bfloat16) for _ in range(3))
    k[..., :2] = 0
    k[0, 2 * BLOCK:3 * BLOCK, 0, 1], k[0, 3 * BLOCK:4 * BLOCK, 0, 1] = 4.0, -4.0      # the routing: block 2 or block 3
    q[0, ::2, 0, 1], q[0, 1::2, 0, 1] = 8.0, -8.0
    k[0, 2 * BLOCK + 5, 0, 0], k[0, 2 * BLOCK + 6, 0, 0] = 4.0, -4.0                  # one key far above, one far below
    q[..., 0] = height / 1.4427 * D ** 0.5 / 4.0
    o, blocks = attend(k, v, q, K)
    for t in range(5 * BLOCK, T):
        assert int(blocks[0, 0, t, 1]) == (2 if t % 2 == 0 else 3)
        check(k, v, q, o, blocks, 0, t)
