"""Sets whose rows are a thread-block cluster (two to eight of them), against float64 attention: lists at the edges of four
pages per row and of eight rows, lists that reach fewer rows than the cluster has, empty lists among them, and
decode steps in which requests of other lengths share a batch."""
import pytest

import workloads as W
from test_gpu_attention_rows import test_attention_split_edges as check_static
from test_gpu_parity import _wl, run_parity

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sets,group,pages", [
    (1, 1, 4), (1, 2, 5), (7, 8, 8), (5, 4, 29), (5, 2, 32),             # one row; two; two; eight, the last with one page; eight whole ones
    (3, 8, 64), (55, 4, 64), (56, 1, 64),                                # the longest lists that go to a cluster of eight; of seven
    (111, 8, 40), (148, 2, 9), (222, 1, 150),                            # four, three and two rows by what the GPU holds
])
def test_rows_of_a_cluster(sets, group, pages):
    check_static(sets, group, pages)


@pytest.mark.parametrize("kind,heads", [(W.PART_PAGE_MINMAX, (8, 8)), (W.PART_TOKEN_DOT, (8, 4)), (W.PART_PAGE_MEAN, (16, 2))])
def test_decode_steps_of_clusters(kind, heads):
    w = _wl(kind, batch=5, num_layers=1, num_q_heads=heads[0], num_kv_heads=heads[1], context=16 * 90, ctx_range=(0, 16 * 90),
            topk=60 if kind == W.PART_TOKEN_DOT else 40, slots_per_set=45, steps=20, lru_buckets=8, drift_choices=(0.05, 0.5))
    r = run_parity(w, one_call=True)
    assert r["stats"]["error_bits"] == 0 and r["stats"]["miss_pages"] > 0
