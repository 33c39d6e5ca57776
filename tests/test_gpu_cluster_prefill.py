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


@pytest.mark.parametrize("clusters,tokens,slots,tail,host_partition,host_rows,ring_mb", [
    (37, 4500, 0, 16, False, False, 0),          # no slots: places through one tail page per head, 2048 tokens at a time
    (37, 4500, 0, 16, True, True, 0), (2600, 6145, 1, 16, True, False, 0), (6000, 4097, 0, 48, False, True, 0),   # 6000 clusters: two slices of counts
    (45000, 4200, 1, 16, False, False, 0),       # counters in global memory from one part to the next
    (300, 5000, 0, 16, True, False, 1),          # through the staging ring, which has room for all places
])
def test_places_in_parts(clusters, tokens, slots, tail, host_partition, host_rows, ring_mb):
    import paper_2604_26837_b200 as P
    H = 2
    g = torch.Generator(device="cuda").manual_seed(clusters + tokens)
    used = torch.randperm(clusters, device="cuda", generator=g)[:min(clusters, 400)]
    part = used[torch.randint(0, len(used), (tokens, H), device="cuda", generator=g)].to(torch.int32)
    kv = torch.randn(2, tokens, H, 128, dtype=torch.bfloat16, device="cuda", generator=g)
    cen = torch.randn(clusters, H, 128, dtype=torch.bfloat16, device="cuda", generator=g)
    p = part.cpu().numpy()
    counts = np.stack([np.bincount(p[:, h], minlength=clusters) for h in range(H)])
    pages = int(((counts + 15) // 16).sum())
    cfg = P.make_config(device=0, num_layers=2, num_q_heads=H, num_kv_heads=H, max_requests=2, max_context_tokens=tokens + 64,
                        partition_kind=2, topk=3, num_clusters=clusters, max_selected_pages=64 + tokens // 16, max_tail_tokens=tail,
                        lru_buckets=8, gpu_cache_pages=4 * H * 3, host_pages=pages + 4 * H, offload_stage_bytes=ring_mb << 20)
    s = P.Spin(cfg)
    other = s.request_open(1)                    # its pages come first: nothing starts at the pool's beginning
    r = s.request_open(slots)
    rows = kv.cpu() if host_rows else kv
    s.append_kv(r, 1, rows[0], rows[1], tokens, part.cpu() if host_partition else part, cen)
    st = s.stats()
    assert st["host_pages_in_use"] == pages and st["error_bits"] == 0
    bits = kv.view(torch.int16).cpu().numpy()
    for h in range(H):
        d = s.debug_dump(r, 1, h, 3, 64 + tokens // 16 + 4, max(1, slots), clusters)
        assert np.array_equal(d["part_tokens"], counts[h]) and not d["part_resident"].any()
        for c in np.unique(p[:, h])[::9]:
            where = np.nonzero(p[:, h] == c)[0]
            for i in range(0, len(where), 16):
                page = s.debug_read_page(r, 1, h, partition=int(c), page_idx=i // 16).view(np.int16)
                w = where[i:i + 16]
                assert np.array_equal(page[0, :len(w)], bits[0, w, h]) and np.array_equal(page[1, :len(w)], bits[1, w, h])
    q = torch.randn(1, H, 128, device="cuda", generator=g).to(torch.bfloat16)
    out = torch.zeros_like(q)
    for _ in range(3):                           # the pages that held the places are cache slots again
        s.decode_step(1, [r], q, out)
    torch.cuda.synchronize()
    chosen = s.debug_dump(r, 1, 0, 3, 64 + tokens // 16 + 4, max(1, slots), clusters)["selected"]
    rows0 = np.isin(p[:, 0], chosen)
    k, v = kv[0, :, 0].double().cpu().numpy()[rows0], kv[1, :, 0].double().cpu().numpy()[rows0]
    want = np.zeros(128)
    if len(k):
        x = k @ q[0, 0].double().cpu().numpy() / np.sqrt(128.0)
        e = np.exp(x - x.max())
        want = (e / e.sum()) @ v
    assert np.abs(out[0, 0].double().cpu().numpy() - want).max() <= 2.0 ** -7 * max(1.0, np.abs(want).max())
    assert s.stats()["error_bits"] == 0
    s.request_close(other)
    s.close()
