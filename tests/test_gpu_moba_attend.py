"""MoBA attention on the tensor cores where it can go wrong: prompt lengths around the edges of a chunk (64), of an
accumulator (128 queries) and of a CTA (256), and scores that keep growing along the prompt, so that a query's running
maximum is raised again and again and its output rescaled.  A budget that covers every block, so that the oracle is
dense causal attention in fp64 on the stored cache.

Bound: the weights are rounded to bf16 (2^-9 of each) and so is the output (2^-9 of it), together at most 2^-8 of the
largest value; a tenth on top for the fp32 sums and the scores (up to about 200, good to 2^-16)."""
import pytest
import torch

import paper_2605_28640_b200 as rq

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("T", [1, 63, 64, 65, 127, 129, 255, 256, 257, 511, 700])
@pytest.mark.parametrize("growth", [0.0, 0.5, -0.5])
def test_dense_budget(growth, T, D):
    block, H = 64, 2
    nb = -(-T // block)
    K = max(2, nb)
    g = torch.Generator(device=DEV)
    g.manual_seed(T * D)
    k = torch.randn(1, T, H, D, generator=g, device=DEV)
    # scores in powers of two: growth per position, beside the random part
    t = torch.arange(T, device=DEV)
    k[..., 0] = growth * t[None, :, None] / 1.4427 * D ** 0.5 * 0.5
    v = torch.randn(1, T, H, D, generator=g, device=DEV)
    q = torch.randn(1, T, H, D, generator=g, device=DEV)
    q[..., 0] = 2.0
    k, v, q = (x.to(torch.bfloat16) for x in (k, v, q))
    cache = rq.Cache(1, H, D, 16, T, torch.bfloat16)
    cache.kv.fill_(0xFF)                                          # what the prefill does not write reads as NaN
    rq.rq_build_cache(cache.handle, k, v, torch.zeros_like(k))    # zero gates: the cache holds k and v themselves
    o = torch.full_like(q, float("nan"))
    scratch = torch.empty(rq.rq_moba_scratch_bytes(cache.handle, block, K), dtype=torch.uint8, device=DEV)
    rq.rq_moba_prefill(cache.handle, q, block, K, 0.0, o, None, None, scratch)
    torch.cuda.synchronize()
    assert rq.rq_device_status(cache.handle) == rq.RQ_OK
    ref = torch.nn.functional.scaled_dot_product_attention(*(x.double().transpose(1, 2) for x in (q, k, v)), is_causal=True)
    err = (o.double().transpose(1, 2) - ref).abs().max().item()
    assert err <= 1.1 * 2 ** -8 * v.float().abs().max().item()


@pytest.mark.parametrize("D,T,gain", [(64, 500, 3.0), (128, 700, 3.0), (128, 1300, 12.0)])
def test_weights_add_up_to_one(D, T, gain):
    """Where all values are the same, so is every output, whatever the weights: what divides the output is the sum of the
    weights as they were multiplied.  The fp32 sums are good to 2^-20, an eighth of a thousandth of a bf16 step: nothing that
    rounding to bf16 leaves visible (the values are bf16 themselves, in the middle of their rounding interval)."""
    block, H = 64, 2
    g = torch.Generator(device=DEV)
    g.manual_seed(T + D)
    k, q = (torch.randn(1, T, H, D, generator=g, device=DEV) for _ in range(2))
    v = torch.randn(1, 1, H, D, generator=g, device=DEV).to(torch.bfloat16).expand(1, T, H, D).contiguous()
    k, q = k.to(torch.bfloat16), (gain * q).to(torch.bfloat16)
    cache = rq.Cache(1, H, D, 16, T, torch.bfloat16)
    rq.rq_build_cache(cache.handle, k, v, torch.zeros_like(k))    # zero gates: the cache holds k and v themselves
    o = torch.empty_like(q)
    K = -(-T // block)
    scratch = torch.empty(rq.rq_moba_scratch_bytes(cache.handle, block, K), dtype=torch.uint8, device=DEV)
    rq.rq_moba_prefill(cache.handle, q, block, K, 0.0, o, None, None, scratch)
    torch.cuda.synchronize()
    assert rq.rq_device_status(cache.handle) == rq.RQ_OK
    assert torch.equal(o, v)
