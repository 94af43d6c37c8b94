"""Prefill where its forms meet: lengths around a tile (256 positions), the first and last tile ragged, tiles taken in turn
by clusters of two and four CTAs, input layouts that a tensor map describes ([B][T][H][D], [B][H][T][D], heads of a wider
row) and one that it does not (a gate shared by all heads: a stride of zero), all element types, a call that starts inside a
page.  The reference is the recurrence in fp64, step by step; the cache is compared with the rounded reference.

Bounds: an fp32 recurrence with gates up to 0.999 carries at most about 1000 roundings of 2^-24, i.e. 6e-5 of the largest
state; a stored bf16 value next to a rounding boundary is one step of 2^-8 off, and nearly none are."""
import pytest
import torch

import paper_2605_28640_b200 as rq

pytestmark = pytest.mark.gpu
DEV = "cuda"
BF, F32 = torch.bfloat16, torch.float32


def laid_out(layout, x):
    """The same numbers as x [B][T][H][D] (contiguous) with other strides; "shared": the first head's for all heads."""
    B, T, H, D = x.shape
    if layout == "bhtd":
        return x.transpose(1, 2).contiguous().transpose(1, 2)
    if layout == "wide":                                         # heads inside a row of twice the width
        w = torch.zeros(B, T, 2 * H, D, device=DEV, dtype=x.dtype)
        w[:, :, :H] = x
        return w[:, :, :H]
    if layout == "shared":                                       # a stride of zero
        return x[:, :, :1].contiguous().expand(B, T, H, D)
    if layout == "batch":                                        # the first batch item's for all
        return x[:1].contiguous().expand(B, T, H, D)
    if layout == "constant":                                     # the first position's for all
        return x[:, :1].contiguous().expand(B, T, H, D)
    return x


def recurrence(k, v, g, T0=0):
    out = []
    for x in (k, v):
        s = torch.zeros(x.shape[0], x.shape[2], x.shape[3], dtype=torch.float64, device=DEV)
        rows = torch.empty(x.shape, dtype=torch.float64, device=DEV)
        for t in range(x.shape[1]):
            gt = g[:, t].double()
            s = gt * s + (1 - gt) * x[:, t].double()
            rows[:, t] = s
        out.append(rows)
    return out


@pytest.mark.parametrize("layout", ["bthd", "bhtd", "wide", "shared"])
@pytest.mark.parametrize("B,H,D,S,T,cuts,dtype,gdtype", [
    (1, 2, 64, 16, 255, [], BF, BF), (1, 2, 128, 16, 256, [], BF, BF), (2, 1, 64, 64, 257, [], F32, F32),
    (1, 3, 128, 16, 1300, [7, 300], BF, F32),                    # starts inside pages and tiles
    (1, 2, 128, 64, 2100, [100], BF, BF),                        # cluster of two or four: eight tiles and a bit
    (1, 8, 128, 16, 4200, [], BF, BF), (1, 4, 64, 16, 4300, [129], F32, BF), (1, 20, 128, 16, 2600, [], BF, BF),
    (2, 40, 64, 64, 600, [64], F32, F32)])
def test_states_cache_and_bounds(B, H, D, S, T, cuts, dtype, gdtype, layout):
    gen = torch.Generator(device=DEV)
    gen.manual_seed(T + H)
    k, v, g = (torch.randn(B, T, H, D, generator=gen, device=DEV) for _ in range(3))
    k, v, g = (laid_out(layout, x) for x in (k.to(dtype), v.to(dtype), torch.sigmoid(4.12 + 0.5 * g).to(gdtype)))
    c = rq.Cache(B, H, D, S, T + 70, dtype, gdtype)
    c.kv.fill_(0xFF)
    c.meta.fill_(0xFF)
    edges = [0, *cuts, T]
    for a, b in zip(edges[:-1], edges[1:]):
        rq.rq_build_cache(c.handle, k[:, a:b], v[:, a:b], g[:, a:b])
    torch.cuda.synchronize()
    assert rq.rq_device_status(c.handle) == rq.RQ_OK and len(c) == T
    P = -(-T // S)
    for i, want in enumerate(recurrence(k, v, g)):
        top = want.abs().max()
        assert (c.state_view()[:, :, i].double() - want[:, -1]).abs().max() <= 6e-5 * top
        got = c.kv_view()[:, :, :P, i].reshape(B, H, P * S, D)
        assert (got[:, :, T:] == 0).all()
        got, want = got[:, :, :T], want.transpose(1, 2)
        off = (got.double() - want.to(dtype).double()).abs()
        if dtype == BF:
            assert (off <= 2 ** -7 * want.abs() + 6e-5 * top).all() and (off > 0).float().mean() <= 2e-3
        else:
            assert off.max() <= 6e-5 * top
    keys = c.kv_view()[:, :, :P, 0]
    for p in range(P):
        rows = keys[:, :, p, :min(S, T - p * S)]
        assert torch.equal(c.meta_view()[:, :, p, 0], rows.amin(2)) and torch.equal(c.meta_view()[:, :, p, 1], rows.amax(2))


@pytest.mark.parametrize("layout", ["bthd", "shared"])
@pytest.mark.parametrize("B,H,D,S,T,cuts,dtype,gdtype", [
    (1, 40, 128, 16, 1, [], BF, BF), (2, 38, 64, 64, 16, [], BF, F32), (1, 38, 128, 64, 17, [16], F32, F32), (4, 20, 64, 16, 100, [7], BF, BF),
    (1, 75, 64, 16, 255, [3, 17, 200], F32, BF), (1, 37, 128, 16, 256, [], BF, BF), (1, 40, 128, 64, 256, [1, 63, 64, 130], BF, BF),
    (1, 40, 128, 64, 300, [250, 260], BF, F32), (1, 5, 128, 16, 1, [], BF, BF), (2, 3, 64, 64, 17, [], F32, F32),
    (1, 5, 128, 64, 130, [64], BF, F32), (1, 6, 64, 16, 290, [256, 257], F32, BF)])
def test_short_calls(B, H, D, S, T, cuts, dtype, gdtype, layout):
    """Calls inside one tile, with more units than SMs (two CTAs per SM, plain loads) and with fewer (tensor maps longer than
    the prompt)."""
    test_states_cache_and_bounds(B, H, D, S, T, cuts, dtype, gdtype, layout)


@pytest.mark.parametrize("layout", ["shared", "batch", "constant"])
@pytest.mark.parametrize("B,H,D,S,T,cuts,dtype,gdtype", [(3, 4, 128, 16, 1100, [300], BF, F32), (2, 9, 64, 64, 2600, [], F32, BF)])
def test_shared_numbers(B, H, D, S, T, cuts, dtype, gdtype, layout):
    """Heads, batch items or positions that share their numbers (a stride of zero)."""
    test_states_cache_and_bounds(B, H, D, S, T, cuts, dtype, gdtype, layout)


def test_shared_numbers_cost_no_more():
    """Heads that share their gates, keys and values read less, not more slowly: the time of a prefill, an eighth allowed for
    what runs differ (they came by plain loads, without anything ahead of them, at 1.7 times the time)."""
    T, H, D = 40000, 32, 128
    times = {}
    for layout in ("bthd", "shared"):
        k, v, g = (laid_out(layout, torch.rand(1, T, H, D, device=DEV).to(BF)) for _ in range(3))
        c = rq.Cache(1, H, D, 16, T, BF)
        best = float("inf")
        for _ in range(12):
            c.handle.len = 0
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            rq.rq_build_cache(c.handle, k, v, g)
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b))
        times[layout] = best
    assert times["shared"] <= 1.125 * times["bthd"], times


@pytest.mark.parametrize("H,D,S,T,dtype,gdtype", [(20, 128, 16, 16384, BF, BF), (32, 128, 64, 16500, BF, F32), (40, 64, 16, 16385, F32, BF),
                                                  (65, 64, 64, 16639, BF, BF)])
def test_units_abreast(H, D, S, T, dtype, gdtype):
    """The form that keeps a head's units abreast (64 tiles and more, nearly as many units as SMs) against two calls of fewer
    tiles each, cut between tiles: the order of the operations is the same, and so are the bits."""
    gen = torch.Generator(device=DEV)
    gen.manual_seed(T + H)
    k, v, g = (torch.randn(1, T, H, D, generator=gen, device=DEV) for _ in range(3))
    k, v, g = k.to(dtype), v.to(dtype), torch.sigmoid(4.12 + 0.5 * g).to(gdtype)
    caches = []
    for edges in ([0, T], [0, 8192, T]):
        c = rq.Cache(1, H, D, S, T, dtype, gdtype)
        for a, b in zip(edges[:-1], edges[1:]):
            rq.rq_build_cache(c.handle, k[:, a:b], v[:, a:b], g[:, a:b])
        torch.cuda.synchronize()
        assert rq.rq_device_status(c.handle) == rq.RQ_OK
        caches.append(c)
    a, b = caches
    assert torch.equal(a.state, b.state) and torch.equal(a.kv, b.kv) and torch.equal(a.meta, b.meta)
