"""Sets whose rows are a thread-block cluster (two to eight of them), against float64 attention: lists at the edges of four
pages per row and of eight rows, lists that reach fewer rows than the cluster has, empty lists among them, shapes just
beyond what goes to clusters, and decode steps in which requests of other lengths share a batch."""
import pytest

import workloads as W
from test_gpu_attention_rows import test_attention_split_edges as check_static
from test_gpu_parity import _wl, run_parity

pytestmark = pytest.mark.gpu


# sets, heads, pages, CTAs of a set that are a cluster (0: none); test_attention_plan.py asks the launcher's rule about them
SHAPES = [
    (1, 1, 4, 0), (1, 2, 5, 2), (7, 8, 8, 2), (148, 2, 9, 2), (222, 1, 96, 2),   # one row; two: the last with one page, whole, all that the GPU holds
    (7, 4, 12, 3), (138, 8, 48, 3), (101, 4, 40, 4), (80, 2, 40, 5),             # three whole rows; the most clusters of three, four and five
    (64, 8, 48, 6), (69, 1, 21, 6), (56, 4, 28, 7),
    (5, 4, 29, 8), (48, 2, 32, 8), (3, 8, 64, 8),                                # the last row with one page; whole; the longest lists
    (55, 4, 64, 0), (3, 1, 65, 0), (142, 8, 24, 0), (222, 1, 97, 0),             # through memory: a warp more pages, nine rows, too many clusters, counts
]


@pytest.mark.parametrize("sets,group,pages,cluster", SHAPES)
def test_rows_of_a_cluster(sets, group, pages, cluster):
    check_static(sets, group, pages)


@pytest.mark.parametrize("kind,heads", [(W.PART_PAGE_MINMAX, (8, 8)), (W.PART_TOKEN_DOT, (8, 4)), (W.PART_PAGE_MEAN, (16, 2))])
def test_decode_steps_of_clusters(kind, heads):
    w = _wl(kind, batch=5, num_layers=1, num_q_heads=heads[0], num_kv_heads=heads[1], context=16 * 90, ctx_range=(0, 16 * 90),
            topk=60 if kind == W.PART_TOKEN_DOT else 40, slots_per_set=45, steps=20, lru_buckets=8, drift_choices=(0.05, 0.5))
    r = run_parity(w, one_call=True)
    assert r["stats"]["error_bits"] == 0 and r["stats"]["miss_pages"] > 0
