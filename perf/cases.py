"""The work that is timed: the library's entry points over the sizes, types and options they are used at.

A case is a dict of plain values; `listed()` names the standing ones and `draw()` gives others of the same ranges.
`prepare()` makes what a program has in hand before the call (caches already prefilled where the call starts from
one), `run()` is one pass through the public entry points, `work()` the bytes and operations a pass cannot do without,
`tolerance()` how far another correct implementation of the same precision may be off.

Kinds of pass:
  decode   `steps` tokens through `layers` caches in turn (one cache per layer of a model, as a serving loop calls it),
           from a prompt of `tokens` positions.  The prompt's recurrence state is put back and the length set back at
           the start of every pass, so that all passes decode the same tokens.  `host`: the tensors live in pinned
           host memory and the result of every step is waited for.  `list`: the kept pages are asked for, too.
  prefill  a prompt of `tokens` positions into an emptied cache.
  snapkv   a prefilled cache reduced to `keep` entries per head under its last 64 queries, and the first token decoded
           on the reduced cache.
  moba     block-sparse attention of every position of a prefilled prompt.
"""
import math

import torch

import paper_2605_28640_b200 as rq

DEV = "cuda"
DTYPES = {"bf16": torch.bfloat16, "f32": torch.float32}
WINDOW = 64          # SnapKV's observation window
# Gates have a memory of about 64 tokens, so decayed keys have a standard deviation of about 0.25 (less between the
# tokens that start afresh).  Queries are scaled so that the attention logits have one of about 1.5, as a trained
# model's have; with unit queries every position would weigh the same and there would be nothing to select.
QUERY_GAIN = 6.0


def listed():
    return [
        # the smallest call: a small fp32 model (4 heads x 64 channels, 1K context, a quarter of the pages), page lists read back
        {"name": "decode-1k-f32", "kind": "decode", "batch": 1, "heads": 4, "dim": 64, "page": 16, "tokens": 1001, "budget": 16,
         "layers": 8, "steps": 2, "dtype": "f32", "gates": "f32", "host": False, "list": True},
        # the paper's own Quest setting: 4K context, pages of 64, 16 of 64 kept; a 7B model's 32 heads, one sequence
        {"name": "decode-4k-page64", "kind": "decode", "batch": 1, "heads": 32, "dim": 128, "page": 64, "tokens": 4090, "budget": 16,
         "layers": 8, "steps": 2, "dtype": "bf16", "gates": "bf16", "host": False, "list": False},
        # batched serving at 32K, an eighth of the pages
        {"name": "decode-32k-b8", "kind": "decode", "batch": 8, "heads": 32, "dim": 128, "page": 16, "tokens": 32700, "budget": 256,
         "layers": 2, "steps": 4, "dtype": "bf16", "gates": "bf16", "host": False, "list": False},
        # the headline: one sequence at 128K, a sixteenth of the pages
        {"name": "decode-128k", "kind": "decode", "batch": 1, "heads": 32, "dim": 128, "page": 16, "tokens": 131060, "budget": 512,
         "layers": 4, "steps": 4, "dtype": "bf16", "gates": "bf16", "host": False, "list": False},
        # the same for a caller whose tensors live in host memory and who reads every result before the next step
        {"name": "decode-128k-host", "kind": "decode", "batch": 1, "heads": 32, "dim": 128, "page": 16, "tokens": 131060, "budget": 512,
         "layers": 4, "steps": 2, "dtype": "bf16", "gates": "bf16", "host": True, "list": False},
        # a short prompt with a ragged end
        {"name": "prefill-4k", "kind": "prefill", "batch": 1, "heads": 32, "dim": 128, "page": 64, "tokens": 4001,
         "dtype": "bf16", "gates": "bf16"},
        # few heads (a tensor-parallel shard), a long ragged prompt, fp32 gates
        {"name": "prefill-50k-h8", "kind": "prefill", "batch": 1, "heads": 8, "dim": 128, "page": 16, "tokens": 50003,
         "dtype": "bf16", "gates": "f32"},
        # the long-context prefill
        {"name": "prefill-128k", "kind": "prefill", "batch": 1, "heads": 32, "dim": 128, "page": 16, "tokens": 131072,
         "dtype": "bf16", "gates": "bf16"},
        # the paper's SnapKV setting for a batch of prompts: 4K context, 1024 entries retained
        {"name": "snapkv-4k-b8", "kind": "snapkv", "batch": 8, "heads": 32, "dim": 128, "page": 16, "tokens": 4096, "keep": 1024,
         "dtype": "bf16", "gates": "bf16"},
        # the same reduction of one long prompt to a sixteenth
        {"name": "snapkv-128k", "kind": "snapkv", "batch": 1, "heads": 32, "dim": 128, "page": 16, "tokens": 131000, "keep": 8192,
         "dtype": "bf16", "gates": "bf16"},
        # the paper's MoBA setting: 4K context, blocks of 64, 16 per query
        {"name": "moba-4k", "kind": "moba", "batch": 1, "heads": 32, "dim": 128, "page": 64, "tokens": 4096, "block": 64, "blocks": 16,
         "dtype": "bf16", "gates": "bf16"},
        # a long ragged prompt: more than 400 blocks, a sixteenth of them per query
        {"name": "moba-30k", "kind": "moba", "batch": 1, "heads": 32, "dim": 128, "page": 16, "tokens": 30011, "block": 64, "blocks": 30,
         "dtype": "bf16", "gates": "bf16"},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _tokens(rng, lo, hi):
    n = _log(rng, lo, hi)
    return n if rng.random() < 0.7 else max(lo, n // 128 * 128)   # round lengths among the ragged ones


def draw(rng):
    kind = rng.choice(["decode", "decode", "prefill", "snapkv", "moba"])
    c = {"kind": kind, "batch": rng.choice([1, 1, 1, 2, 3, 4, 8]), "heads": rng.choice([4, 8, 12, 16, 32, 32, 40]),
         "dim": rng.choice([64, 128, 128]), "page": rng.choice([16, 64])}
    c["dtype"] = rng.choice(["bf16"] * 4 + ["f32"])
    c["gates"] = rng.choice([c["dtype"], c["dtype"], "f32"])
    row = c["batch"] * c["heads"] * c["dim"] * (2 if c["dtype"] == "bf16" else 4)     # one position of keys, bytes
    most = min(131072, (1 << 30) // row)                 # keys of a cache: at most those of 32 heads x 128 channels at 128K
    if kind == "moba":
        # attended pairs grow with the square of the prompt: at most the listed long one's; fp32 runs without tensor cores
        most = int(30000 * min(1.0, math.sqrt(32 / (c["batch"] * c["heads"]))) * (0.15 if c["dtype"] == "f32" else 1.0))
        c["tokens"] = _tokens(rng, 1000, min(most, 30000))
        c["block"] = rng.choice([64, 64, 128, 256])
        n = -(-c["tokens"] // c["block"])
        c["blocks"] = max(2, min(30, n // rng.choice([4, 8, 16])))
        return c
    c["tokens"] = _tokens(rng, 1000, most)
    if kind == "snapkv":
        c["keep"] = max(WINDOW, min(8192, c["tokens"] // rng.choice([4, 8, 16])))
    if kind == "decode":
        c["budget"] = max(4, -(-c["tokens"] // c["page"]) // rng.choice([4, 8, 16]))
        c["layers"] = max(1, min(8, (8 << 30) // (2 * row * c["tokens"])))
        c["steps"] = 2
        c["host"] = rng.random() < 0.2
        c["list"] = rng.random() < 0.1
    return c


class Caches:
    """`layers` caches of one shape with the caller's buffers; the recurrence states lie side by side."""

    def __init__(self, c, capacity, layers=1, budget=None):
        dt = {"bf16": rq.RQ_BF16, "f32": rq.RQ_F32}
        self.c, self.pages = c, -(-capacity // c["page"])
        cfg = rq.rq_config(c["batch"], c["heads"], c["dim"], c["page"], capacity, dt[c["dtype"]], dt[c["gates"]], 1, 1,
                           budget or self.pages, 0)
        kv, meta, state, ws = rq.rq_sizes(cfg)
        self.states = torch.empty(layers, state, dtype=torch.uint8, device=DEV)
        self.buffers = [[torch.empty(n, dtype=torch.uint8, device=DEV) for n in (kv, meta, ws)] for _ in range(layers)]
        self.handles = [rq.rq_cache_init(cfg, b[0], b[1], self.states[i], b[2]) for i, b in enumerate(self.buffers)]

    def kv(self, pages, layer=0, first=0):
        c = self.c
        t = self.buffers[layer][0].view(DTYPES[c["dtype"]])
        return t.view(c["batch"], c["heads"], self.pages, 2, c["page"], c["dim"])[:, :, first:pages]

    def bounds(self, pages, layer=0, first=0):
        c = self.c
        t = self.buffers[layer][1].view(DTYPES[c["dtype"]])
        return t.view(c["batch"], c["heads"], self.pages, 2, c["dim"])[:, :, first:pages]

    def state(self):
        c = self.c
        return self.states.view(torch.float32).view(-1, c["batch"], c["heads"], 2, c["dim"])


def _inputs(c, gen, *shape):
    """Keys, values and gates of that shape: unit normal keys and values; gates with a memory of about 64 tokens."""
    k = torch.randn(*shape, generator=gen, device=DEV, dtype=DTYPES[c["dtype"]])
    v = torch.randn(*shape, generator=gen, device=DEV, dtype=DTYPES[c["dtype"]])
    g = torch.randn(*shape, generator=gen, device=DEV, dtype=DTYPES[c["gates"]]).mul_(0.5).add_(4.12).sigmoid_()
    return k, v, g


def _prompt(c, gen):
    """A prompt's keys, values and gates; one token in a hundred starts afresh (half of the memory is dropped)."""
    k, v, g = _inputs(c, gen, c["batch"], c["tokens"], c["heads"], c["dim"])
    g.masked_fill_((torch.rand(c["batch"], c["tokens"], 1, 1, generator=gen, device=DEV) < 0.01), 0.5)
    return k, v, g


def _queries(c, gen, *shape):
    return torch.randn(*shape, generator=gen, device=DEV, dtype=DTYPES[c["dtype"]]).mul_(QUERY_GAIN)


def prepare(case, seed):
    c = dict(case)
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed)
    s = {"case": c}
    B, T, H, D = c["batch"], c["tokens"], c["heads"], c["dim"]
    if c["kind"] == "prefill":
        s["prompt"] = _prompt(c, gen)
        s["cache"] = Caches(c, T + 256)
        return s
    layers, steps = c.get("layers", 1), c.get("steps", 1)
    s["cache"] = Caches(c, T + max(64, steps), layers, c.get("budget"))
    for h in s["cache"].handles:
        rq.rq_build_cache(h, *_prompt(c, gen))
    if c["kind"] == "moba":
        s["q"] = _queries(c, gen, B, T, H, D)
        s["o"] = torch.empty_like(s["q"])
        s["scratch"] = torch.empty(rq.rq_moba_scratch_bytes(s["cache"].handles[0], c["block"], c["blocks"]), dtype=torch.uint8, device=DEV)
        return s
    # the tokens to be decoded, a set of tensors for each call
    q = _queries(c, gen, steps, layers, B, H, D)
    k, v, g = _inputs(c, gen, steps, layers, B, H, D)
    o = torch.empty_like(q)
    if c.get("host"):
        q, k, v, g, o = (x.cpu().pin_memory() for x in (q, k, v, g, o))
    s["o"] = o
    if c["kind"] == "snapkv":
        s["token"] = tuple(x[0, 0] for x in (q, k, v, g, o))
        s["window"] = _queries(c, gen, B, WINDOW, H, D)
        s["idx"] = torch.empty(B, H, c["keep"], dtype=torch.int32, device=DEV)
        s["importance"] = torch.empty(B, H, T, dtype=torch.float32, device=DEV)
        s["scratch"] = torch.empty(rq.rq_snapkv_scratch_bytes(s["cache"].handles[0]), dtype=torch.uint8, device=DEV)
        s["reduced"] = Caches(c, c["keep"] + 256)
        return s
    s["prompt_states"] = s["cache"].states.clone()
    # the pages that the decoded tokens are written to, and their bounds
    first, last = T // c["page"], -(-(T + steps) // c["page"])
    s["appended"] = [(s["cache"].kv(last, i, first), s["cache"].bounds(last, i, first)) for i in range(layers)]
    s["lists"] = None
    if c["list"]:
        s["lists"] = torch.empty(steps, layers, B, H, c["budget"], dtype=torch.int32, device="cpu" if c["host"] else DEV)
        s["lists"] = s["lists"].pin_memory() if c["host"] else s["lists"]
    s["calls"] = [(s["cache"].handles[j], q[i, j], k[i, j], v[i, j], g[i, j], c["budget"], 0.0, o[i, j],
                   None if s["lists"] is None else s["lists"][i, j]) for i in range(steps) for j in range(layers)]
    return s


def run(s):
    c, cache = s["case"], s["cache"]
    if c["kind"] == "decode":
        cache.states.copy_(s["prompt_states"])
        for h in cache.handles:
            h.len = c["tokens"]
        if c["host"]:
            for call in s["calls"]:
                rq.rq_decode_step_host(*call)
                torch.cuda.current_stream().synchronize()
        else:
            for call in s["calls"]:
                rq.rq_decode_step(*call)
        return [s["o"], cache.state(), s["lists"], s["appended"]]
    h = cache.handles[0]
    if c["kind"] == "prefill":
        rq.rq_cache_reset(h)
        rq.rq_build_cache(h, *s["prompt"])
        pages = -(-c["tokens"] // c["page"])
        return [cache.kv(pages), cache.bounds(pages), cache.state()]
    if c["kind"] == "moba":
        rq.rq_moba_prefill(h, s["q"], c["block"], c["blocks"], 0.0, s["o"], None, None, s["scratch"])
        return [s["o"]]
    # snapkv.  The retained positions are read through what they are for, the attention over the reduced cache: where two
    # importances at the cut are equal to within rounding, either position may be kept, and all rows behind it shift.
    d = s["reduced"].handles[0]
    rq.rq_snapkv_select(h, s["window"], WINDOW, c["keep"], 0.0, s["idx"], s["importance"], s["scratch"])
    rq.rq_snapkv_compact(h, s["idx"], c["keep"], d)
    q, k, v, g, o = s["token"]
    rq.rq_decode_step(d, q, k, v, g, s["reduced"].pages, 0.0, o)
    return [s["importance"], s["o"], s["reduced"].state()]


def work(case):
    c = case
    BH, T, D, S = c["batch"] * c["heads"], c["tokens"], c["dim"], c["page"]
    es, gs = 2 if c["dtype"] == "bf16" else 4, 2 if c["gates"] == "bf16" else 4
    token = BH * D * (4 * es + gs + 16)                 # q, k, v, o and g of a token, the state read and written
    if c["kind"] == "decode":
        nbytes = flops = 0
        for i in range(c["steps"]):
            n = T + i + 1
            P = -(-n // S)
            rows = min(c["budget"], P) * S
            nbytes += BH * (P * 2 * D * es + rows * 2 * D * es) + token
            flops += BH * (P * 3 * D + rows * 4 * D)
        return {"bytes": nbytes * c["layers"], "flops": flops * c["layers"]}
    if c["kind"] == "prefill":
        P = -(-T // S)
        return {"bytes": BH * D * (T * (2 * es + gs) + T * 2 * es + P * 2 * es + 8), "flops": BH * D * T * 6}
    if c["kind"] == "snapkv":
        rows = c["keep"] * 2 * D * es
        nbytes = BH * (T * D * es + T * 4 + c["keep"] * 4 + WINDOW * D * es + 2 * rows + rows) + token
        return {"bytes": nbytes, "flops": BH * (2 * WINDOW * D * T + 4 * D * c["keep"])}
    n, K = c["block"], c["blocks"]
    pairs = sum(min(t // n, K - 1) * n + t % n + 1 for t in range(T))                    # attended (query, key) pairs
    routed = sum(t // n for t in range(T) if t // n >= K)                                  # (query, block) scores
    return {"bytes": BH * T * D * es * 4, "flops": BH * (4 * D * pairs + 2 * D * routed)}


def tolerance(case):
    """About four times what each path showed against the same computation in 64 bits (on the cache as stored)."""
    if case["dtype"] == "f32":
        # observed: prefill 1.3e-7 (1e-6 at a single value); decode, moba 3e-7 (3e-6); importances 1.5e-6 (1e-5)
        return {"rel": 1e-6, "max": 1e-5} if case["kind"] == "prefill" else {"rel": 8e-6, "max": 8e-5}
    if case["kind"] == "prefill":
        # the states agree to 1.3e-7; 2.9e-5 is what the few stored values next to a rounding boundary make (one step: 2^-7)
        return {"rel": 1.2e-4, "max": 1e-2}
    # 1.7e-3 is the rounding of the results to bf16, 5e-3 its largest with weights rounded to bf16; two blocks (pages) whose
    # scores at the cut are equal to within fp32 rounding may change places, which moves the results of that query more
    return {"rel": 7e-3, "max": 0.5 if case["kind"] == "moba" else 0.1}
