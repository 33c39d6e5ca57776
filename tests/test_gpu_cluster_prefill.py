"""Cluster prefill at the edges of the ranking kernel: counters of 16 warps, of fewer, of one, and in global memory."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("clusters,tokens,host_partition,host_rows", [
    (1, 33, False, False), (37, 16 * 64 + 5, True, False), (2600, 4100, False, True),    # 16, 16, 15 warps
    (25000, 700, True, True), (45000, 700, False, False),                                # one warp; counters in global memory
])
def test_rows_stand_in_their_clusters_in_arrival_order(clusters, tokens, host_partition, host_rows):
    import paper_2604_26837_b200 as P
    H = 2
    g = torch.Generator(device="cuda").manual_seed(clusters + tokens)
    used = min(clusters, 1000)                 # few enough that clusters repeat
    ids = torch.randperm(clusters, device="cuda", generator=g)[:used]
    part = ids[torch.randint(0, used, (tokens, H), device="cuda", generator=g)].to(torch.int32)
    kv = torch.randn(2, tokens, H, 128, dtype=torch.bfloat16, device="cuda", generator=g)
    cen = torch.randn(clusters, H, 128, dtype=torch.bfloat16, device="cuda", generator=g)
    pages = int(sum(((np.bincount(part[:, h].cpu().numpy(), minlength=clusters) + 15) // 16).sum() for h in range(H)))
    cfg = P.make_config(device=0, num_layers=1, num_q_heads=H, num_kv_heads=H, max_requests=1,
                        max_context_tokens=tokens + 16, partition_kind=2, topk=1, num_clusters=clusters,
                        max_selected_pages=64 + tokens // 16, max_tail_tokens=16, lru_buckets=8, gpu_cache_pages=H * 8, host_pages=pages + H)
    s = P.Spin(cfg)
    r = s.request_open(8)
    bad = part.clone()
    bad[tokens // 2, 1] = clusters
    with pytest.raises(P.SpinError) as e:
        s.append_kv(r, 0, kv[0], kv[1], tokens, bad, cen)
    assert e.value.code == 1 and "token_partition[%d][1] = %d" % (tokens // 2, clusters) in str(e.value)
    assert s.stats()["host_pages_in_use"] == 0
    rows = kv.cpu() if host_rows else kv
    s.append_kv(r, 0, rows[0], rows[1], tokens, part.cpu() if host_partition else part, cen)
    assert s.stats()["host_pages_in_use"] == pages and s.stats()["error_bits"] == 0
    kv_bits = kv.view(torch.int16).cpu().numpy()
    p = part.cpu().numpy()
    for h in range(H):
        d = s.debug_dump(r, 0, h, 1, 64 + tokens // 16 + 4, 8, clusters)
        assert np.array_equal(d["part_tokens"], np.bincount(p[:, h], minlength=clusters)) and not d["part_resident"].any()
        for c in np.unique(p[:, h])[:40]:
            where = np.nonzero(p[:, h] == c)[0]
            for i in range(0, len(where), 16):
                page = s.debug_read_page(r, 0, h, partition=int(c), page_idx=i // 16).view(np.int16)
                w = where[i:i + 16]
                assert np.array_equal(page[0, :len(w)], kv_bits[0, w, h]) and np.array_equal(page[1, :len(w)], kv_bits[1, w, h])
    s.close()
