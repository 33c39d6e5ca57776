"""Decode steps whose lists give a warp of attention more pages than it has lanes, against the oracle: batches of 32
pages per warp, with missed pages in some and hits in others, the set's flags and slots known from the first on."""
import pytest

import workloads as W
from test_gpu_parity import _wl, run_parity

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("slots,kw", [
    (700, {}),                                   # fewer slots than pages: batches of misses, of both, of hits
    (120, {}),                                   # mostly bypassed: whole batches from host memory
    (1100, dict(host_tables_only=1)),            # few misses, resolved by the warps themselves
    (700, dict(fetch_mode=1)),                   # fetched by the copy kernel: no early descriptors
])
def test_batches_of_pages_per_warp(slots, kw):
    # 128 sets: three CTAs of four warps each; ~1000 pages per list, so ~84 for a warp
    w = _wl(W.PART_TOKEN_DOT, num_layers=1, batch=16, num_q_heads=32, num_kv_heads=8, context=16 * 1200 + 3, topk=2048,
            slots_per_set=slots, lru_buckets=8, drift=0.3, steps=4)
    r = run_parity(w, one_call=True, oracle_reqs=[5], check_bytes=slots == 700, **kw)
    st = r["stats"]
    assert st["error_bits"] == 0 and st["miss_pages"] > 0 and st["hit_pages"] > 0
    assert st["selected_pages"] / st["set_steps"] > 12 * 64
