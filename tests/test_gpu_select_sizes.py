"""Selection and cache manager at the sizes where they change form, bit for bit against the oracle."""
import pytest

import workloads as W
from test_gpu_parity import _wl, run_parity

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("pages,topk", [(3071, 40), (3073, 300), (4100, 7)])
def test_pages_around_the_compaction_rule(pages, topk):
    # up to 3072 candidates a thread compacts a run of them, beyond it a warp blocks of 128; with
    # tied scores the k-th place falls inside a group of equals
    w = _wl(W.PART_PAGE_MINMAX, num_layers=1, batch=1, num_q_heads=4, num_kv_heads=1, context=16 * pages + 16, steps=3,
            topk=topk, slots_per_set=400, kv_recipe="tied", tie_period=16 * 700)
    assert run_parity(w, one_call=True, check_bytes=False)["tied_at_k"] >= 1      # groups of four or five: a place may end one


@pytest.mark.parametrize("tokens,topk", [(16 * 9 + 1, 200), (16 * 64 + 3, 130), (16 * 301 + 16, 129)])
def test_tokens_folded_into_pages_by_rows_of_bits(tokens, topk):
    # every token chosen (an odd number of pages), a whole number of blocks, a ragged last block
    w = _wl(W.PART_TOKEN_DOT, num_layers=1, num_q_heads=4, num_kv_heads=2, context=tokens, steps=4, topk=topk,
            slots_per_set=200)
    assert run_parity(w, one_call=True, check_bytes=False)["stats"]["error_bits"] == 0


@pytest.mark.parametrize("kind,pages,topk,slots", [
    (W.PART_PAGE_MINMAX, 1300, 30, 1025), (W.PART_PAGE_MEAN, 4200, 60, 4096), (W.PART_PAGE_MINMAX, 4200, 60, 4097),
    (W.PART_TOKEN_DOT, 1100, 2048, 1024),
])
def test_slot_counts_around_the_shared_memory_cache_manager(kind, pages, topk, slots):
    # more than 1024 slots, the most it takes, one more (page table in global memory); the cluster
    # top-k with 2048 tokens and 1024 slots beside its keys
    w = _wl(kind, num_layers=1, batch=1, num_q_heads=4, num_kv_heads=1, context=16 * pages + 5, steps=4, topk=topk,
            slots_per_set=slots, lru_buckets=8, drift=0.5)
    assert run_parity(w, one_call=True, check_bytes=False)["stats"]["miss_pages"] > 0


def test_the_chosen_scoring_form_is_not_the_slower_one_for_large_caches():
    # 8 requests of 60000 tokens, 8 heads, everything cached and nothing missed: the form that the library
    # chooses against a CTA per work item (measured 83 us; the resident grid 108)
    import torch
    import paper_2604_26837_b200 as P
    n, H, R = 60000, 8, 8
    g = torch.Generator(device="cuda").manual_seed(1)
    k = torch.randn(n, H, 128, dtype=torch.bfloat16, device="cuda", generator=g)
    q = torch.randn(R, H, 128, device="cuda", generator=g).to(torch.bfloat16)
    new, out, us = k[:R].contiguous(), torch.empty_like(q), {}
    for form in (0, -1):
        s = P.Spin(P.make_config(device=0, num_layers=1, num_q_heads=H, num_kv_heads=H, max_requests=R, max_context_tokens=n + 512,
                                 partition_kind=0, topk=64, resident_scoring=form, gpu_cache_pages=R * H * 3780, host_pages=R * H * 3790))
        reqs = s.req_array([s.request_open(3780) for _ in range(R)])
        for r in reqs:
            s.append_kv(r, 0, k, k, n)
        us[form] = 1e9
        for _ in range(8):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            torch.cuda.synchronize()
            e0.record()
            for _ in range(15):
                s.decode_step_append(0, reqs, new, new, q, out)
            e1.record()
            torch.cuda.synchronize()
            us[form] = min(us[form], e0.elapsed_time(e1) * 1e3 / 15)
        s.close()
    assert us[0] <= 1.12 * us[-1], us
