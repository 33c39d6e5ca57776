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
