"""The HBM a context needs: callers size their pools once, so it does not grow.  No GPU needed."""
import pytest


@pytest.mark.parametrize("kind,kv_heads,group,layers,requests,tokens,topk,segment,ring_mb,fetch_mode,host_tables,trace,most", [
    (0, 1, 4, 1, 1, 100, 16, 0, 0, 0, 0, 0, 12076800),
    (0, 8, 4, 32, 7, 32768, 16, 0, 0, 0, 0, 0, 168143104),
    (1, 8, 1, 1, 256, 1048576, 2048, 16, 0, 1, 1, 0, 18051309568),
    (3, 8, 8, 32, 256, 32768, 2048, 0, 64, 0, 0, 1, 8495399936),
    (2, 1, 1, 1, 1, 100, 16, 0, 0, 0, 0, 0, 9489664),
    (2, 8, 4, 1, 1, 32768, 16, 0, 0, 0, 0, 0, 18382592),
    (2, 8, 4, 32, 7, 1048576, 16, 16, 0, 0, 0, 0, 354132224),
    (2, 8, 8, 1, 256, 32768, 2048, 0, 0, 1, 0, 0, 9997906944),
    (2, 1, 8, 32, 7, 1048576, 2048, 0, 0, 0, 1, 1, 82745344),
    (2, 8, 4, 1, 7, 1048576, 16, 0, 64, 0, 0, 0, 128905984),
    (2, 8, 1, 32, 256, 100, 16, 0, 64, 0, 0, 0, 11592048896),
])
def test_a_context_fits_the_pool_it_has_always_fitted(kind, kv_heads, group, layers, requests, tokens, topk, segment, ring_mb, fetch_mode,
                                                      host_tables, trace, most):
    import paper_2604_26837_b200 as P
    cluster = kind == P.PART_CLUSTER_CENTROID
    cfg = P.make_config(device=0, num_layers=layers, num_q_heads=kv_heads * group, num_kv_heads=kv_heads, max_requests=requests,
                        max_context_tokens=tokens, partition_kind=kind, topk=topk, num_clusters=512 if cluster else 0,
                        max_selected_pages=topk * 4 if cluster else 0, max_tail_tokens=64 if cluster else 0, segment_entries=segment,
                        offload_stage_bytes=ring_mb << 20, fetch_mode=fetch_mode, host_tables_only=host_tables, trace=trace,
                        gpu_cache_pages=1000, host_pages=5000)
    assert P.spin_required_bytes(cfg)[0] <= most
