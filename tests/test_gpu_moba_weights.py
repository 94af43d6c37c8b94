"""What the weights of MoBA's attention are relative to, where the scores of a chunk of 64 positions exceed all before it: the
largest score so far, at most 8 powers of two behind.  The error of the output hangs on it (the rounding of the largest weight to
bf16 is none where the weight is 1), and so does the range of values that stay finite."""
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
    o = torch.full_like(q, float("nan"))
    blocks = torch.empty(1, H, T, K, dtype=torch.int32, device=DEV)
    scratch = torch.empty(rq.rq_moba_scratch_bytes(cache.handle, BLOCK, K), dtype=torch.uint8, device=DEV)
    rq.rq_moba_prefill(cache.handle, q, BLOCK, K, 0.0, o, blocks, None, scratch)
    torch.cuda.synchronize()
    assert rq.rq_device_status(cache.handle) == rq.RQ_OK
    return o[0, :, 0], blocks[0, 0].long()


def scores(k, q, blocks):
    """In fp64, as powers of two; -inf where a query does not attend."""
    T, D = k.shape[1], k.shape[3]
    nb = T // BLOCK
    chosen = torch.zeros(T, nb + 1, dtype=torch.bool, device=DEV)
    chosen.scatter_(1, torch.where(blocks < 0, nb, blocks), True)
    keep = chosen[:, :nb].repeat_interleave(BLOCK, 1) & torch.ones(T, T, dtype=torch.bool, device=DEV).tril()
    s = q[0, :, 0].double() @ k[0, :, 0].double().T * (D ** -0.5 * 1.4426950408889634)
    return s.masked_fill(~keep, float("-inf"))


@pytest.mark.parametrize("D,T,K,gain", [(64, 2048, 32, 8.0), (128, 1024, 16, 5.0), (128, 2048, 16, 5.0), (128, 1536, 8, 15.0)])
def test_relative_to_the_largest_score(D, T, K, gain):
    """The same in fp64 with weights rounded to bf16.  The fp32 sums are good to 2^-18 of the output, and outputs that lie closer than
    that to a boundary between two bf16 values, 2^-8 apart, may be rounded the other way: one in 2^9; as many again for weights
    that are rounded the other way.  (With the first chunk's maximum kept longer 91 to 97 of 100 outputs are the same.)"""
    g = torch.Generator(device=DEV)
    g.manual_seed(T + D)
    k, v, q = (torch.randn(1, T, 1, D, generator=g, device=DEV, dtype=torch.bfloat16) for _ in range(3))
    q *= gain
    o, blocks = attend(k, v, q, K)
    s = scores(k, q, blocks)
    m = torch.full((T,), float("-inf"), dtype=torch.float64, device=DEV)
    num, den = torch.zeros(T, D, dtype=torch.float64, device=DEV), torch.zeros(T, dtype=torch.float64, device=DEV)
    for c in range(T // 64):
        x = s[:, c * 64:c * 64 + 64]
        top = x.max(1).values
        new = torch.where(top > m + 8, top, m)
        f = torch.where(m > float("-inf"), torch.exp2(m - new), torch.zeros_like(m))
        w = torch.exp2(x - new[:, None]).to(torch.bfloat16).double()
        num, den, m = num * f[:, None] + w @ v[0, c * 64:c * 64 + 64, 0].double(), den * f + w.sum(1), new
    want = (num / den[:, None]).to(torch.bfloat16)
    assert (o == want).double().mean().item() >= 0.996


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("height", [7.0, 12.0, 25.0, 31.0])
def test_large_values(height, D):
    """Values of 1e30 and a chosen block `height` powers of two above the first one: finite, as the values are.  A weight is at most
    2^8, a sum of 1024 of them times 1e30 at most 2^118."""
    T, K = 10 * BLOCK, 3
    g = torch.Generator(device=DEV)
    g.manual_seed(D)
    k, v, q = (torch.randn(1, T, 1, D, generator=g, device=DEV) for _ in range(3))
    k, v, q = k.to(torch.bfloat16), (v.abs() * 1e30).to(torch.bfloat16), q.to(torch.bfloat16)
    k[..., 0] = 0
    k[0, 2 * BLOCK:3 * BLOCK, 0, 0] = 4.0
    q[..., 0] = height / 1.4427 * D ** 0.5 / 4.0
    o, blocks = attend(k, v, q, K)
    want = torch.softmax(scores(k, q, blocks) * 0.6931471805599453, 1) @ v[0, :, 0].double()
    assert (blocks[4 * BLOCK:, 1] == 2).double().mean().item() > (0.9 if height >= 12 else 0.5)
    # weights and output rounded to bf16: 2^-8 of the largest value, a tenth on top for the rest
    assert (o.double() - want).abs().max().item() <= 1.1 * 2 ** -8 * v.double().max().item()
