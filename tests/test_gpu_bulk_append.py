"""Appends on either side of the size from which page ids are copied to HBM ahead of the pages (192 pages of all heads
together), with and without those copies: the pages' bytes in host memory are those of the tokens."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("heads,pages", [(1, 191), (1, 192), (2, 95), (2, 96), (8, 24), (8, 300)])
@pytest.mark.parametrize("host_tables_only", [0, 1])
def test_bulk_appends(heads, pages, host_tables_only):
    import workloads as W
    from test_gpu_parity import _wl, run_parity
    # `pages` complete pages besides the newest, which is the tail
    w = _wl(W.PART_PAGE_MINMAX, num_layers=1, batch=1, num_q_heads=heads, num_kv_heads=heads, context=16 * pages + 5, topk=8, slots_per_set=12, steps=3)
    r = run_parity(w, one_call=True, check_bytes=True, host_tables_only=host_tables_only)
    assert r["stats"]["error_bits"] == 0 and r["stats"]["miss_pages"] > 0
