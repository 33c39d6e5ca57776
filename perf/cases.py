"""What a user of this library has it do, as cases that can be timed and compared.

Four paths, all through the public entry points of `paper_2604_26837_b200.binding`:

  decode    one decode step of every layer for a batch of open requests
            (`spin_decode_step_append`: append one token per request, score, select, cache
            management, page fetch over the host link, attention)
  generate  cluster granularity: sixteen decode steps and the periodic fold of the local tail into
            the clusters (`spin_reindex`)
  prefill   a request's life up to its first output: open, prefill of every layer in chunks as a
            scheduler hands them over, first decode step, close
  static    `spin_paged_attention_static`: paged attention over lists the caller supplies, all pages
            in HBM, nothing allocated

A decode case keeps its context open, as a serving loop does: a pass appends a token, so contexts
grow a little from pass to pass, queries drift from step to step, and the cache is in the steady
state it has reached by then (`prime` steps are run beforehand).  When the room for new tokens is
used up the requests end and the next ones, with the same prompts, take their places.
"""
import math

import torch

from paper_2604_26837_b200 import binding as B

D, T = 128, 16                                   # head dimension and tokens per page of the library
ROW, PAGE = 2 * D, 2 * T * 2 * D                 # bytes of a K or V row, of a page
KINDS = {"minmax": B.PART_PAGE_MINMAX, "token": B.PART_TOKEN_DOT, "cluster": B.PART_CLUSTER_CENTROID,
         "mean": B.PART_PAGE_MEAN}
DEV = "cuda:0"


def _decode(**kw):
    # batch requests of `context` tokens (geometrically down to `shortest` of that), `budget` of each
    # request's pages as GPU slots, queries that drift by `drift` per step, `room` tokens to generate
    return {"path": "decode", "layers": 1, "shortest": 1.0, "buckets": 64, "clusters": 0, "io": "device", **kw}


def _prefill(**kw):
    return {"path": "prefill", "layers": 1, "buckets": 64, "clusters": 0, "ring_mb": 0, "budget": 0.25, **kw}


def listed():
    return [
        # one small request, one kv head: latency of the whole chain
        _decode(name="decode tiny", kind="minmax", batch=1, q_heads=4, kv_heads=1, context=4096, topk=16,
                budget=0.25, buckets=8, drift=0.1, room=1024, prime=24),
        # the Llama-3-8B-shaped layer: page granularity, a quarter of the pages in HBM
        _decode(name="decode pages", kind="minmax", batch=8, q_heads=32, kv_heads=8, context=32768, topk=128,
                budget=0.25, drift=0.05, room=6144, prime=100),
        # token granularity: 64K exact token scores per set, selected tokens folded into pages
        _decode(name="decode tokens", kind="token", batch=4, q_heads=4, kv_heads=1, context=65536, topk=2048,
                budget=0.2, drift=0.05, room=4096, prime=24),
        # mixed lengths, two layers, strongly drifting queries: one batch of a busy server
        _decode(name="decode mixed lengths", kind="minmax", batch=6, q_heads=32, kv_heads=8, context=131072,
                shortest=0.0625, layers=2, topk=256, budget=0.1, drift=0.1, room=512, prime=12),
        # short and middling contexts that HBM holds whole, mean-key landmarks, eight query heads per
        # kv head, q/k/v/out in pinned host memory: nothing but hits
        _decode(name="decode resident", kind="mean", batch=16, q_heads=64, kv_heads=8, context=6007, shortest=0.5,
                topk=64, budget=1.0, drift=0.05, room=8192, prime=100, io="pinned"),
        # cluster granularity with its periodic fold: the 1024-cluster configuration, two requests
        {"path": "generate", "name": "generate clusters", "kind": "cluster", "batch": 2, "layers": 1, "q_heads": 32,
         "kv_heads": 8, "context": 131072, "shortest": 1.0, "topk": 64, "clusters": 1024, "budget": 0.1,
         "buckets": 64, "drift": 0.05, "room": 4096, "prime": 16, "steps": 16, "io": "device"},
        # a short prompt: the calls' own cost
        _prefill(name="prefill short", kind="token", q_heads=8, kv_heads=4, tokens=1501, chunk=4096, topk=256),
        # a long prompt in one call, pages written through to host memory
        _prefill(name="prefill pages", kind="minmax", q_heads=32, kv_heads=8, tokens=32768, chunk=32768, topk=128),
        # the same in chunks, two layers, pages offloaded asynchronously through a staging ring
        _prefill(name="prefill chunks ring", kind="minmax", q_heads=32, kv_heads=8, tokens=16411, chunk=2048, topk=128,
                 layers=2, ring_mb=64),
        # cluster granularity: tokens packed into their clusters' pages
        _prefill(name="prefill clusters", kind="cluster", q_heads=32, kv_heads=8, tokens=32768, chunk=32768, topk=32,
                 clusters=512),
        # caller-made page lists: a few short ones, and a batch that fills HBM's bandwidth
        {"path": "static", "name": "static small", "sets": 8, "group": 4, "pages": 40, "ragged": 0.5, "masked": 0.1},
        {"path": "static", "name": "static large", "sets": 256, "group": 8, "pages": 56, "ragged": 0.0, "masked": 0.0},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges: any kind, group, batch and length, odd ones among them."""
    path = rng.choice(["decode", "decode", "decode", "decode", "generate", "prefill", "prefill", "static"])
    if path == "static":
        group = rng.choice([1, 2, 4, 8])
        pages = _log_int(rng, 3, 900)
        most = min(256, 14000 // pages, 2000000 // (group * (D + 2) * ((pages + 7) // 8)))
        return {"path": "static", "sets": _log_int(rng, 2, max(2, most)), "group": group, "pages": pages,
                "ragged": rng.choice([0.0, 0.3, 0.9]), "masked": rng.choice([0.0, 0.1])}
    group, kv_heads = rng.choice([1, 2, 4, 4, 8]), rng.choice([1, 2, 4, 8, 8])
    heads = {"q_heads": group * kv_heads, "kv_heads": kv_heads}
    if path == "prefill":
        kind = rng.choice(["minmax", "token", "cluster", "mean"])
        tokens = _log_int(rng, 400, 32768)
        chunk = tokens if kind == "cluster" else rng.choice([512, 2048, 8192, 32768])
        return _prefill(kind=kind, tokens=tokens, chunk=chunk, layers=rng.choice([1, 2]) if tokens < 16384 else 1,
                        topk=_log_int(rng, 64, 1024) if kind == "token" else _log_int(rng, 16, 128),
                        clusters=_log_int(rng, 128, 1024) if kind == "cluster" else 0,
                        ring_mb=rng.choice([0, 64]), **heads)
    if path == "generate":
        clusters = _log_int(rng, 256, 1024)
        return {"path": "generate", "kind": "cluster", "batch": rng.choice([1, 2, 3]), "layers": 1, **heads,
                "context": _log_int(rng, 8192, 65536), "shortest": rng.choice([1.0, 0.5]),
                "topk": clusters // rng.choice([16, 20, 32]), "clusters": clusters, "budget": rng.choice([0.1, 0.2, 0.3]),
                "buckets": 64, "drift": rng.choice([0.01, 0.05, 0.1]), "room": 4096, "prime": 8, "steps": 16, "io": "device"}
    kind = rng.choice(["minmax", "minmax", "token", "mean"])
    context = _log_int(rng, 1000, 65536)
    most = max(1, min(16, 1500000 // (context * kv_heads)))
    budget = rng.choice([0.1, 0.2, 0.25, 0.5, 1.0])
    return _decode(kind=kind, batch=rng.randint(1, most), **heads, context=context, shortest=rng.choice([1.0, 1.0, 0.25]),
                   topk=_log_int(rng, 128, 2048) if kind == "token" else _log_int(rng, 16, 256), budget=budget,
                   buckets=rng.choice([8, 64]), drift=rng.choice([0.01, 0.05, 0.1, 0.5]), room=4096, prime=32,
                   io=rng.choice(["device", "device", "pinned"]))


# ---- shapes ------------------------------------------------------------------------------------

def _contexts(case):
    n = case["batch"]
    if n == 1:
        return [case["context"]]
    return [max(T + 1, int(case["context"] * case["shortest"] ** (i / (n - 1)))) for i in range(n)]


def _slots(case, context):
    pages = (context + T - 1) // T
    if case["budget"] >= 1.0:
        return (context + case["room"]) // T + 2
    # never less than one step's own pages, as the paper's scheduler guarantees
    need = case["topk"] if case["kind"] in ("minmax", "mean") else min(pages, case["topk"] // 2)
    if case["kind"] == "cluster":
        need = 0
    return max(1, min(pages, need), int(case["budget"] * pages))


# ---- inputs ------------------------------------------------------------------------------------

def _keys(case, n, H, gen):
    """Keys and values as attention layers meet them: outlier channels (page granularity), tokens close
    to their page's centre (token granularity)."""
    k = torch.randn(n, H, D, dtype=torch.bfloat16, device=DEV, generator=gen)
    v = torch.randn(n, H, D, dtype=torch.bfloat16, device=DEV, generator=gen)
    if case["kind"] == "token":
        cen = torch.randn((n + T - 1) // T, H, D, dtype=torch.bfloat16, device=DEV, generator=gen)
        k = cen.repeat_interleave(T, 0)[:n] + 0.5 * k
    else:
        k[:, :, [3, 40, 77, 101]] *= 8.0
    return k.contiguous(), v


def _clustered(case, n, H, gen):
    C = case["clusters"]
    cen = torch.randn(C, H, D, dtype=torch.bfloat16, device=DEV, generator=gen)
    part = torch.randint(0, C, (n, H), dtype=torch.int32, device=DEV, generator=gen)
    k = cen[part.long(), torch.arange(H, device=DEV)[None]]
    k += 0.3 * torch.randn(n, H, D, dtype=torch.bfloat16, device=DEV, generator=gen)
    v = torch.randn(n, H, D, dtype=torch.bfloat16, device=DEV, generator=gen)
    return k, v, part.contiguous(), cen.contiguous()


def _queries(case, steps, batch, gen):
    """q_t = normalize(q_{t-1} + drift * N(0,1)): bf16 [steps][layers][batch][q_heads][D]."""
    shape = (case["layers"], batch, case["q_heads"], D)
    q = torch.nn.functional.normalize(torch.randn(shape, device=DEV, generator=gen), dim=-1)
    out = torch.empty((steps,) + shape, dtype=torch.bfloat16, device=DEV)
    for t in range(steps):
        out[t] = q
        q = torch.nn.functional.normalize(q + case.get("drift", 0.05) * torch.randn(shape, device=DEV, generator=gen), dim=-1)
    return out


class _Serving:
    """A context with a batch of open requests and the inputs of a generation that goes on."""

    RING = 128                                   # steps of inputs before they come round again

    def __init__(self, case, seed):
        self.case = case
        gen = torch.Generator(device=DEV)
        gen.manual_seed(seed)
        H, L, n = case["kv_heads"], case["layers"], case["batch"]
        self.contexts = _contexts(case)
        self.slots = [_slots(case, c) for c in self.contexts]
        cluster = case["kind"] == "cluster"
        pages = [(c + case["room"]) // T + 2 + (case["clusters"] + case["room"] // T if cluster else 0) for c in self.contexts]
        tail = 2 * T + case.get("steps", 0)
        biggest = 16 + 2 * max(self.contexts) // (T * case["clusters"]) if cluster else 1
        cfg = B.make_config(device=0, num_layers=L, num_q_heads=case["q_heads"], num_kv_heads=H, max_requests=n,
                            max_context_tokens=max(self.contexts) + case["room"] + T, partition_kind=KINDS[case["kind"]],
                            topk=case["topk"], num_clusters=case["clusters"],
                            max_selected_pages=case["topk"] * biggest if cluster else 0,
                            max_tail_tokens=tail if cluster else 0, lru_buckets=case["buckets"],
                            gpu_cache_pages=sum(self.slots) * L * H, host_pages=sum(pages) * L * H)
        self.spin = B.Spin(cfg, DEV)
        make = _clustered if cluster else (lambda *a: _keys(*a) + (None, None))
        self.prompts = [[make(case, c, H, gen) for _ in range(L)] for c in self.contexts]
        self.q = _queries(case, self.RING, n, gen)
        k, v = _keys(case, self.RING * L * n, H, gen)
        self.k, self.v = k.view(self.RING, L, n, H, D), v.view(self.RING, L, n, H, D)
        self.out = torch.empty((case.get("steps", 1), L, n, case["q_heads"], D), dtype=torch.bfloat16, device=DEV)
        if case["io"] == "pinned":
            self.q, self.k, self.v, self.out = (x.cpu().pin_memory() for x in (self.q, self.k, self.v, self.out))
        # the rows of every step, as the caller's loop holds them
        self.rows = [[(self.k[t, l], self.v[t, l], self.q[t, l]) for l in range(L)] for t in range(self.RING)]
        self.outs = [[self.out[s, l] for l in range(L)] for s in range(self.out.shape[0])]
        self.reqs, self.t = [], 0
        self.admit()
        for _ in range(case["prime"]):
            self.step(self.outs[0])
        self.fold()
        torch.cuda.synchronize()

    def admit(self):
        for r in self.reqs:
            self.spin.request_close(r)
        self.reqs = [self.spin.request_open(s) for s in self.slots]
        self.ids = self.spin.req_array(self.reqs)
        self.made = 0
        for r, layers in zip(self.reqs, self.prompts):
            for l, (k, v, part, cen) in enumerate(layers):
                self.spin.append_kv(r, l, k, v, k.shape[0], part, cen)

    def step(self, outs):
        if self.made == self.case["room"]:
            self.admit()
        row = self.rows[self.t % self.RING]
        for l, (k, v, q) in enumerate(row):
            self.spin.decode_step_append(l, self.ids, k, v, q, outs[l])
        self.t += 1
        self.made += 1

    def fold(self):
        if self.case["kind"] == "cluster":
            for r in self.reqs:
                for l in range(self.case["layers"]):
                    self.spin.reindex(r, l)


class _Prompt:
    """A context and one request's prompt, to be taken in from nothing."""

    def __init__(self, case, seed):
        self.case = case
        gen = torch.Generator(device=DEV)
        gen.manual_seed(seed)
        H, L, n = case["kv_heads"], case["layers"], case["tokens"]
        cluster = case["kind"] == "cluster"
        pages = n // T + 3 + case["clusters"]
        self.slots = max(64, int(case["budget"] * n / T))
        cfg = B.make_config(device=0, num_layers=L, num_q_heads=case["q_heads"], num_kv_heads=H, max_requests=1,
                            max_context_tokens=n + T, partition_kind=KINDS[case["kind"]], topk=case["topk"],
                            num_clusters=case["clusters"],
                            max_selected_pages=case["topk"] * (8 + 2 * n // (T * case["clusters"])) if cluster else 0,
                            max_tail_tokens=T if cluster else 0, lru_buckets=case["buckets"],
                            offload_stage_bytes=case["ring_mb"] << 20, gpu_cache_pages=self.slots * L * H,
                            host_pages=pages * L * H)
        self.spin = B.Spin(cfg, DEV)
        make = _clustered if cluster else (lambda *a: _keys(*a) + (None, None))
        self.prompt = [make(case, n, H, gen) for _ in range(L)]
        self.q = _queries(case, 1, 1, gen)[0]
        self.out = torch.empty((L, 1, case["q_heads"], D), dtype=torch.bfloat16, device=DEV)

    def first_token(self):
        case, spin = self.case, self.spin
        r = spin.request_open(self.slots)
        for l, (k, v, part, cen) in enumerate(self.prompt):
            for t in range(0, case["tokens"], case["chunk"]):
                kk, vv = k[t:t + case["chunk"]], v[t:t + case["chunk"]]
                spin.append_kv(r, l, kk, vv, kk.shape[0], part, cen)
        for l in range(case["layers"]):
            spin.decode_step(l, [r], self.q[l], self.out[l])
        torch.cuda.current_stream().synchronize()            # no work of a request may be in flight when it closes
        spin.request_close(r)
        return self.out


class _Lists:
    """Caller-made page lists over a pool in HBM."""

    def __init__(self, case, seed):
        self.case = case
        gen = torch.Generator(device=DEV)
        gen.manual_seed(seed)
        S, P, G = case["sets"], case["pages"], case["group"]
        n = S * P + 7
        self.pool = torch.randn(n, 2 * T * D, dtype=torch.bfloat16, device=DEV, generator=gen)
        self.ids = torch.randperm(n, device=DEV, generator=gen)[:S * P].to(torch.int32).view(S, P).contiguous()
        mask = torch.full((S, P), 0xFFFF, dtype=torch.int64, device=DEV)
        if case["masked"]:
            some = torch.rand(S, P, device=DEV, generator=gen) < case["masked"]
            mask = torch.where(some, torch.randint(1, 0x10000, (S, P), device=DEV, generator=gen), mask)
        self.masks = mask.to(torch.int32)
        self.n = (P - (torch.rand(S, device=DEV, generator=gen) * case["ragged"] * P).long()).to(torch.int32)
        q = torch.randn(S, G, D, device=DEV, generator=gen)
        self.q = q.to(torch.bfloat16)
        self.out = torch.empty(S, G, D, dtype=torch.bfloat16, device=DEV)


def prepare(case, seed):
    return {"static": _Lists, "prefill": _Prompt}.get(case["path"], _Serving)(case, seed)


def run(state):
    case = state.case
    if case["path"] == "static":
        rc = B.spin_paged_attention_static(state.q, state.pool, state.ids, state.masks, state.n, case["sets"],
                                           case["pages"], case["group"], 0.0, state.out)
        if rc:
            raise RuntimeError("spin_paged_attention_static: status %d" % rc)
        return state.out
    if case["path"] == "prefill":
        return state.first_token()
    for outs in state.outs:
        state.step(outs)
    if case["path"] == "generate":
        state.fold()
    elif case["io"] == "pinned":
        torch.cuda.current_stream().synchronize()            # the host reads this step's output
    return state.out


# ---- what a pass cannot do without -------------------------------------------------------------

def _step_bytes(case, context):
    """Summaries of one set, its selected K/V (in token granularity the selected rows) and the tail."""
    pages = context // T
    if case["kind"] == "token":
        return context * ROW + min(case["topk"], context) * 2 * ROW + PAGE / 2
    if case["kind"] == "cluster":
        return case["clusters"] * ROW + min(case["topk"], case["clusters"]) * context / case["clusters"] * 2 * ROW
    return pages * (2 * ROW if case["kind"] == "minmax" else ROW) + (min(case["topk"], pages) + 0.5) * PAGE


def _step_flops(case, context):
    group, kind = case["q_heads"] // case["kv_heads"], case["kind"]
    cands = context if kind == "token" else case["clusters"] if kind == "cluster" else context // T
    tokens = min(case["topk"], context) if kind == "token" else \
        min(case["topk"], case["clusters"]) * context // case["clusters"] if kind == "cluster" else min(case["topk"] * T, context)
    return 2.0 * D * group * (cands + 2 * tokens)


def work(case):
    if case["path"] == "static":
        tokens = case["sets"] * case["pages"] * (1 - case["ragged"] / 2) * T
        return {"bytes": tokens * 2 * ROW + case["sets"] * case["group"] * 2 * ROW,
                "flops": 4.0 * D * case["group"] * tokens}
    H, L = case["kv_heads"], case["layers"]
    if case["path"] == "prefill":
        # K and V are read once, written once to host memory, a summary per partition is written;
        # then one decode step
        n = case["tokens"]
        return {"bytes": L * H * (2.0 * n * 2 * ROW + _step_bytes(case, n)), "flops": L * H * _step_flops(case, n)}
    steps = case.get("steps", 1)
    ctx = _contexts(case)
    io = 2.0 * L * len(ctx) * (case["q_heads"] + H) * ROW
    return {"bytes": steps * (io + L * H * sum(_step_bytes(case, c) for c in ctx)),
            "flops": steps * L * H * sum(_step_flops(case, c) for c in ctx)}


def tolerance(case):
    # bf16 outputs (2^-9 per value) of tensor-core attention whose probabilities are rounded to bf16:
    # about 3e-3 against a float64 computation over the same selected pages, which are compared exactly
    # wherever the repository's tests compare them
    return {"rel": 1e-2}
