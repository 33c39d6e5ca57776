"""Paged attention at the edges of its work split, against float64 attention over the same rows.

A set's pages are dealt out to the warps of its CTAs: as many CTAs as the GPU holds at once, at least
eight pages for each (four where they are a cluster), a lane per page in batches of 32 pages per warp, two pages of a warp in flight.
"""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sets,group,pages", [
    (1, 1, 1), (1, 8, 7), (2, 4, 8), (3, 2, 9), (1, 4, 33), (5, 1, 72),   # one CTA; a CTA's remainder; several CTAs
    (64, 4, 129),                                                        # six CTAs per set
    (449, 1, 129), (450, 1, 140),                                        # one CTA per set: up to 33 and 35 pages per warp, more CTAs than fit
    (222, 8, 17), (223, 8, 17),                                          # two CTAs per set, then one
    (2, 1, 600),                                                         # 75 partials: three tiles of the merge
])
def test_attention_split_edges(sets, group, pages):
    import paper_2604_26837_b200 as P
    g = torch.Generator(device="cuda").manual_seed(sets * 1000 + group * 100 + pages)
    n = sets * pages + 3
    pool = torch.randn(n, 2, 16, 128, dtype=torch.bfloat16, device="cuda", generator=g)
    ids = torch.randperm(n, device="cuda", generator=g)[:sets * pages].to(torch.int32).view(sets, pages).contiguous()
    masks = torch.randint(0, 0x10000, (sets, pages), device="cuda", generator=g).to(torch.int32)
    counts = torch.full((sets,), pages, dtype=torch.int32, device="cuda")
    if sets > 4:
        counts[1::3] = torch.randint(0, pages + 1, (len(counts[1::3]),), device="cuda", generator=g).to(torch.int32)
        counts[4] = 0
    q = torch.randn(sets, group, 128, device="cuda", generator=g).to(torch.bfloat16)
    out = torch.full_like(q, 7.0)
    for _ in range(2):                       # the second call meets what the first left in the built-in arrays
        assert P.spin_paged_attention_static(q, pool, ids, masks, counts, sets, pages, group, 0.0, out) == 0
    torch.cuda.synchronize()
    rows = pool[ids.long()].double()                                      # [sets][pages][2][16][128]
    live = (masks[:, :, None].long() >> torch.arange(16, device="cuda")) & 1
    live = live.bool() & (torch.arange(pages, device="cuda")[None, :, None] < counts[:, None, None])
    k, v, live = rows[:, :, 0].reshape(sets, -1, 128), rows[:, :, 1].reshape(sets, -1, 128), live.reshape(sets, -1)
    s = torch.einsum("sgd,std->sgt", q.double(), k) / np.sqrt(128.0)
    s = s.masked_fill(~live[:, None], -torch.inf)
    p = torch.nan_to_num(torch.softmax(s, dim=-1))                        # a set without a token: zeros
    want = torch.einsum("sgt,std->sgd", p, v)
    # bf16 probabilities and bf16 outputs: 2^-9 relative each, against values of order one
    err = (out.double() - want).abs().max().item()
    assert err <= 2.0 ** -8 * max(1.0, want.abs().max().item()) * 2, err
    if sets > 4:
        assert not out[4].any()


@pytest.mark.parametrize("sets,pages", [(3, 5), (2, 40)])
def test_outputs_need_no_more_than_element_alignment(sets, pages):
    import paper_2604_26837_b200 as P
    g = torch.Generator(device="cuda").manual_seed(sets)
    pool = torch.randn(sets * pages, 2, 16, 128, dtype=torch.bfloat16, device="cuda", generator=g)
    ids = torch.arange(sets * pages, dtype=torch.int32, device="cuda").view(sets, pages)
    masks = torch.full((sets, pages), 0xFFFF, dtype=torch.int32, device="cuda")
    counts = torch.full((sets,), pages, dtype=torch.int32, device="cuda")
    counts[-1] = 0
    q = torch.randn(sets, 4, 128, device="cuda", generator=g).to(torch.bfloat16)
    outs = []
    for offset in (0, 1):                    # whole pieces; one element further on
        buf = torch.full((q.numel() + 8,), 7.0, dtype=torch.bfloat16, device="cuda")
        out = buf[offset:offset + q.numel()]
        assert P.spin_paged_attention_static(q, pool, ids, masks, counts, sets, pages, 4, 0.0, out) == 0
        torch.cuda.synchronize()
        assert (buf[:offset] == 7).all() and (buf[offset + q.numel():] == 7).all()
        outs.append(out.clone())
    assert torch.equal(outs[0], outs[1])


@pytest.mark.parametrize("sets,group,pages,sharpness", [(256, 8, 56, 1.0), (256, 2, 64, 1.0), (60, 1, 200, 1.0), (230, 8, 60, 2.0), (8, 4, 40, 1.0)])
def test_rounding_of_probabilities_does_not_grow_with_the_list(sets, group, pages, sharpness):
    """Error against fp64, beside that of the same sums with probabilities rounded to bf16 against the
    largest of every 32 tokens (a warp's two pages of eight): the kernel's may not be larger.  Both are sums of many
    independent roundings, so over sets * group * 128 >= 4096 outputs they agree to 1 / sqrt(2 * 4096) ~ 1 %."""
    import paper_2604_26837_b200 as P
    g = torch.Generator(device="cuda").manual_seed(sets + pages)
    pool = torch.randn(sets * pages, 2, 16, 128, dtype=torch.bfloat16, device="cuda", generator=g)
    ids = torch.randperm(sets * pages, device="cuda", generator=g).to(torch.int32).view(sets, pages).contiguous()
    masks = torch.full((sets, pages), 0xFFFF, dtype=torch.int32, device="cuda")
    counts = torch.full((sets,), pages, dtype=torch.int32, device="cuda")
    q = (torch.randn(sets, group, 128, device="cuda", generator=g) * sharpness).to(torch.bfloat16)
    out = torch.empty_like(q)
    assert P.spin_paged_attention_static(q, pool, ids, masks, counts, sets, pages, group, 0.0, out) == 0
    torch.cuda.synchronize()
    err, err32, norm = 0.0, 0.0, 0.0
    for i in range(sets):
        rows = pool[ids[i].long()].double()
        k, v = rows[:, 0].reshape(-1, 128), rows[:, 1].reshape(-1, 128)
        s = q[i].double() @ k.T / np.sqrt(128.0)
        want = torch.softmax(s, dim=-1) @ v
        base = s.view(group, -1, 32).amax(-1, keepdim=True).expand(-1, -1, 32).reshape(s.shape)
        p, scale = torch.exp(s - base), torch.exp(base - s.amax(-1, keepdim=True))
        rounded = ((p.to(torch.bfloat16).double() * scale) @ v / (p * scale).sum(-1, keepdim=True)).to(torch.bfloat16)
        err += (out[i].double() - want).square().sum().item()
        err32 += (rounded.double() - want).square().sum().item()
        norm += want.square().sum().item()
    assert err <= err32 * 1.02, ((err / norm) ** 0.5, (err32 / norm) ** 0.5)


def _lists(sets, group, pages, counts, seed=5):
    g = torch.Generator(device="cuda").manual_seed(seed)
    pool = torch.randn(sets * pages, 2, 16, 128, dtype=torch.bfloat16, device="cuda", generator=g)
    ids = torch.randperm(sets * pages, device="cuda", generator=g).to(torch.int32).view(sets, pages).contiguous()
    masks = torch.full((sets, pages), 0xFFFF, dtype=torch.int32, device="cuda")
    q = torch.randn(sets, group, 128, device="cuda", generator=g).to(torch.bfloat16)
    return q, pool, ids, masks, torch.tensor(counts, dtype=torch.int32, device="cuda")


@pytest.mark.parametrize("sets,group,pages,short,long", [
    (256, 1, 500, 8, {17: 500, 200: 499}),                  # 16 rows where one is the rule, done by other lists' CTAs
    (256, 1, 500, 8, {i: 500 for i in range(100, 256, 2)}), # further rows of many lists
    (64, 1, 500, 9, {0: 500, 63: 65}),                      # 16 rows where six are the rule
    (64, 8, 248, 9, {0: 248, 63: 65}),                      # lists too short for the counts to be looked at
    (72, 2, 288, 8, {0: 288, 71: 287}), (72, 2, 289, 8, {0: 289, 71: 288}),   # the longest such, one more
    (700, 1, 180, 3, {0: 180, 1: 33, 698: 95, 699: 97}),    # more sets than CTAs at once
    (223, 2, 280, 0, {5: 280}),                             # nothing in the other lists
    (1790, 1, 72, 1, {0: 72, 1789: 33}), (2048, 1, 56, 1, {0: 56, 2047: 33}),   # the most sets that the built-in arrays take with such lists
])
def test_uneven_lists(sets, group, pages, short, long):
    import paper_2604_26837_b200 as P
    counts = [long.get(i, short) for i in range(sets)]
    q, pool, ids, masks, n = _lists(sets, group, pages, counts)
    out = torch.full_like(q, 7.0)
    for _ in range(2):
        assert P.spin_paged_attention_static(q, pool, ids, masks, n, sets, pages, group, 0.0, out) == 0
    torch.cuda.synchronize()
    for i in list(long) + [2, 3, sets // 2]:
        rows = pool[ids[i, :counts[i]].long()].double()
        s = q[i].double() @ rows[:, 0].reshape(-1, 128).T / np.sqrt(128.0)
        want = torch.softmax(s, dim=-1) @ rows[:, 1].reshape(-1, 128)
        assert (out[i].double() - want).abs().max().item() <= 2.0 ** -7 * max([1.0] + want.abs().flatten().tolist()), i


def _best_us(f, calls=20):
    best = 1e9
    for _ in range(6):
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        torch.cuda.synchronize()
        e0.record()
        for _ in range(calls):
            f()
        e1.record()
        torch.cuda.synchronize()
        best = min(best, e0.elapsed_time(e1) * 1e3 / calls)
    return best


def test_a_long_list_among_short_ones_is_shared():
    """The batch takes about what its long list and its short ones take by themselves, not what four warps need for 500 pages
    (measured: 25 us, 8 + 7 apart, 128 where every set had one CTA)."""
    import paper_2604_26837_b200 as P

    def us(sets, counts):
        a = _lists(sets, 1, 500, counts)
        out = torch.empty_like(a[0])
        return _best_us(lambda: P.spin_paged_attention_static(*a, sets, 500, 1, 0.0, out))
    both, alone = us(256, [8] * 100 + [500] + [8] * 155), us(1, [500]) + us(256, [8] * 256)
    assert both <= 3 * alone, (both, alone)


def test_a_long_request_among_short_ones():
    """Decode: outputs of an uneven batch against those of the same requests one at a time."""
    import paper_2604_26837_b200 as P
    lengths, H, topk = [3000] + [37 + i for i in range(31)], 8, 170
    g = torch.Generator(device="cuda").manual_seed(3)
    kv = [torch.randn(2, n, H, 128, dtype=torch.bfloat16, device="cuda", generator=g) for n in lengths]
    q = torch.randn(4, len(lengths), 2 * H, 128, device="cuda", generator=g).to(torch.bfloat16)
    new = torch.randn(2, 4, len(lengths), H, 128, dtype=torch.bfloat16, device="cuda", generator=g)
    outs = []
    for together in (True, False):
        cfg = P.make_config(device=0, num_layers=1, num_q_heads=2 * H, num_kv_heads=H, max_requests=len(lengths), max_context_tokens=3100,
                            partition_kind=0, topk=topk, lru_buckets=8, gpu_cache_pages=H * (len(lengths) + 1) * 180,
                            host_pages=H * sum(n // 16 + 2 for n in lengths))
        s = P.Spin(cfg)
        reqs = [s.request_open(180) for _ in lengths]
        for r, x in zip(reqs, kv):
            s.append_kv(r, 0, x[0], x[1], x.shape[1])
        out = torch.zeros_like(q)
        for t in range(4):
            for i in ([slice(None)] if together else [slice(i, i + 1) for i in range(len(lengths))]):
                s.decode_step_append(0, s.req_array(reqs[i]), new[0, t, i], new[1, t, i], q[t, i], out[t, i])
        torch.cuda.synchronize()
        assert s.stats()["error_bits"] == 0
        outs.append(out.double())
        s.close()
    # two sums in different orders, each within 2^-8 of the exact one (bf16 probabilities, bf16 outputs)
    assert (outs[0] - outs[1]).abs().max().item() <= 2.0 ** -7 * max(1.0, outs[1].abs().max().item())


@pytest.mark.parametrize("sets,group,pages", [(445, 4, 4), (445, 8, 1), (600, 1, 3), (445, 2, 5), (444, 4, 4)])
def test_short_lists_of_many_sets(sets, group, pages):
    # a warp to itself for each list of up to four pages, from 445 sets on
    test_attention_split_edges(sets, group, pages)


def test_short_lists_of_many_sets_in_a_decode_step():
    import workloads as W
    from test_gpu_parity import _wl, run_parity
    w = _wl(W.PART_PAGE_MINMAX, num_layers=1, batch=60, num_q_heads=16, num_kv_heads=8, context=16 * 9 + 3, topk=3, slots_per_set=5, steps=6)
    assert run_parity(w, one_call=True, oracle_reqs=[0, 59])["stats"]["error_bits"] == 0


def test_many_one_page_lists_take_little_more_than_as_many_pages_in_longer_lists():
    import paper_2604_26837_b200 as P

    def us(sets, pages):
        a = _lists(sets, 1, pages, [pages] * sets)
        out = torch.empty_like(a[0])
        return _best_us(lambda: P.spin_paged_attention_static(*a, sets, pages, 1, 0.0, out))
    one, eight = us(16000, 1), us(2000, 8)
    assert one <= 2.5 * eight, (one, eight)
