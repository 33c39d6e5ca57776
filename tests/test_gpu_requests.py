"""Requests that open in page pools which earlier ones have left in pieces: hundreds of runs of physical pages, sets whose
slots end within a table segment, slots in none; and prefills through the staging ring into a host pool in pieces."""
import ctypes
import os
import subprocess

import pytest
import torch

pytestmark = pytest.mark.gpu


def _context(P, **kw):
    return P.Spin(P.make_config(**dict(dict(device=0, num_layers=2, num_q_heads=4, num_kv_heads=2, max_requests=130, max_context_tokens=20000,
                                            partition_kind=0, topk=8, lru_buckets=8, gpu_cache_pages=6000, host_pages=12000), **kw)))


def _decode(P, s, slots, kv, steps, seed, chunk):
    g = torch.Generator(device="cuda").manual_seed(seed)
    r = s.request_open(slots)
    for l in range(2):
        for t in range(0, kv.shape[1], chunk):
            s.append_kv(r, l, kv[0, t:t + chunk], kv[1, t:t + chunk], kv[0, t:t + chunk].shape[0])
    out = torch.zeros(steps, 2, 1, 4, 128, dtype=torch.bfloat16, device="cuda")
    for t in range(steps):
        for l in range(2):
            k, v = torch.randn(2, 1, 2, 128, device="cuda", generator=g).to(torch.bfloat16)
            q = torch.randn(1, 4, 128, device="cuda", generator=g).to(torch.bfloat16)
            s.decode_step_append(l, s.req_array([r]), k, v, q, out[t, l])
    torch.cuda.synchronize()
    st = s.stats()
    assert st["error_bits"] == 0
    return r, out, st


@pytest.mark.parametrize("slots,segment_entries", [(300, 0), (256, 16), (1000, 64), (40, 0), (0, 0)])
@pytest.mark.parametrize("ring", [0, 4 * 2 * 7 * 8192])
def test_requests_in_pools_in_pieces(slots, segment_entries, ring):
    import paper_2604_26837_b200 as P
    g = torch.Generator(device="cuda").manual_seed(slots)
    kv = torch.randn(2, 1500, 2, 128, device="cuda", generator=g).to(torch.bfloat16)
    got = []
    for pieces in (False, True):
        s = _context(P, segment_entries=segment_entries, offload_stage_bytes=ring)
        if pieces:
            # small requests take the low pages, every other one leaves and the rest shrink: 320 holes of 3 and 20 pages
            small = [s.request_open(5) for _ in range(128)]
            for i, r in enumerate(small):
                s.append_kv(r, i % 2, kv[0, :40], kv[1, :40], 40)
            torch.cuda.synchronize()
            for r in small[::2]:
                s.request_close(r)
            for r in small[1::2]:
                s.set_budget(r, 2)
        before = s.stats()
        r, out, st = _decode(P, s, slots, kv, 6, 11, 700)
        assert st["gpu_pages_in_use"] - before["gpu_pages_in_use"] == 4 * slots
        got.append((out, st["hit_pages"], st["miss_pages"]))
        torch.cuda.synchronize()
        s.request_close(r)
        assert s.stats()["gpu_pages_in_use"] == before["gpu_pages_in_use"] and s.stats()["host_pages_in_use"] == before["host_pages_in_use"]
        # what the request has left behind is found whole by the next one
        r, again, _ = _decode(P, s, slots, kv, 6, 11, 700)
        assert torch.equal(again, out)
        s.close()
    assert torch.equal(got[0][0], got[1][0]) and got[0][1:] == got[1][1:]


def test_requests_come_and_go_while_the_sms_are_full(tmp_path):
    # beside work that fills every SM for a while, as decode steps on other streams do
    import paper_2604_26837_b200 as P
    from paper_2604_26837_b200 import build
    so = tmp_path / "full.so"
    subprocess.check_call([build._nvcc(), "-O2", "-std=c++17", "-gencode", "arch=compute_100a,code=sm_100a", "-shared", "-Xcompiler", "-fPIC",
                           os.path.join(os.path.dirname(os.path.abspath(__file__)), "full_sms.cu"), "-o", str(so)])
    full = ctypes.CDLL(str(so))
    s = _context(P, num_layers=1)
    s.request_close(s.request_open(500))                       # (first calls load what they need)
    for slots in (40, 1000):
        r = s.request_open(500)
        torch.cuda.synchronize()
        assert full.fill(400) == 1
        s.request_close(r)
        r = s.request_open(slots)
        assert full.still_full() == 1
        torch.cuda.synchronize()
        assert s.stats()["gpu_pages_in_use"] == 2 * slots
        s.request_close(r)
    s.close()
