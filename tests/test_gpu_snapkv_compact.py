"""Compaction where a run of 64 slots, a warp's 16 slots or a page ends inside: every row bit for bit, unused slots of the
last page zero, bounds the minimum and maximum of the rows, the state carried over, and a decode step on the result."""
import pytest
import torch

import paper_2605_28640_b200 as rq

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("S", [16, 64])
@pytest.mark.parametrize("keep", [1, 15, 16, 17, 63, 64, 65, 80, 129, 300])
def test_rows_bounds_and_state(keep, S, D, dtype):
    B, H, T = 2, 3, 300
    g = torch.Generator(device=DEV)
    g.manual_seed(keep * D + S)
    src = rq.Cache(B, H, D, S, T, dtype)
    k, v = (torch.randn(B, T, H, D, generator=g, device=DEV).to(dtype) for _ in range(2))
    gate = torch.rand(B, T, H, D, generator=g, device=DEV).to(dtype)
    rq.rq_build_cache(src.handle, k, v, gate)
    idx = torch.stack([torch.randperm(T, generator=g, device=DEV)[:keep].sort().values for _ in range(B * H)])
    idx = idx.to(torch.int32).view(B, H, keep)
    dst = rq.Cache(B, H, D, S, keep + 40, dtype)
    for t in (dst.kv, dst.meta, dst.state):
        t.fill_(0xFF)
    rq.rq_snapkv_compact(src.handle, idx, keep, dst.handle)
    torch.cuda.synchronize()
    assert len(dst) == keep and torch.equal(dst.state_view(), src.state_view())
    rows = src.kv_view().permute(3, 0, 1, 2, 4, 5).reshape(2, B, H, -1, D)          # [k / v][B][H][position][D]
    P = -(-keep // S)
    got = dst.kv_view()[:, :, :P].permute(3, 0, 1, 2, 4, 5).reshape(2, B, H, -1, D)
    want = torch.stack([torch.gather(r, 2, idx.long()[..., None].expand(-1, -1, -1, D)) for r in rows])
    assert torch.equal(got[:, :, :, :keep], want) and (got[:, :, :, keep:] == 0).all()
    for p in range(P):
        kp = want[0][:, :, p * S:(p + 1) * S]
        assert torch.equal(dst.meta_view()[:, :, p, 0], kp.amin(2)) and torch.equal(dst.meta_view()[:, :, p, 1], kp.amax(2))
    q, kt, vt = (torch.randn(B, H, D, generator=g, device=DEV).to(dtype) for _ in range(3))
    o = torch.empty_like(q)
    rq.rq_decode_step(dst.handle, q, kt, vt, torch.zeros_like(kt), dst.page_capacity, 0.0, o)   # zero gate: appends kt, vt
    kk, vv = (torch.cat([w, x[:, :, None]], 2).double() for w, x in zip(want, (kt, vt)))
    ref = torch.softmax((kk @ q.double()[..., None])[..., 0] * D ** -0.5, -1)[:, :, None] @ vv
    # bf16: the output's own rounding (2^-9 of it); fp32: 300 products and sums of 2^-24 each
    tol = 2 ** -8 if dtype == torch.bfloat16 else 1e-5
    assert (o.double() - ref[:, :, 0]).abs().max() <= tol * vv.abs().max()
