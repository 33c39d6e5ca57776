"""Paged attention at the edges of its work split, against float64 attention over the same rows.

A set's pages are dealt out to the warps of its CTAs: as many CTAs as the GPU holds at once, at least
eight pages for each, a lane per page in batches of 32 pages per warp, two pages of a warp in flight.
"""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sets,group,pages", [
    (1, 1, 1), (1, 8, 7), (2, 4, 8), (3, 2, 9), (1, 4, 33), (5, 1, 72),   # one CTA; a CTA's remainder; several CTAs
    (64, 4, 129),                                                        # six CTAs per set
    (449, 1, 129), (450, 1, 140),                                        # one CTA per set: 32 and 35 pages per warp, more CTAs than fit
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
