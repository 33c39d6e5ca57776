"""Queries and new K/V rows in pinned host memory: read by the step's own kernels where they are."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind,q_heads,kv_heads", [(0, 8, 2), (1, 3, 3), (3, 16, 2)])
def test_pinned_step_inputs_give_the_outputs_of_device_ones(kind, q_heads, kv_heads):
    import paper_2604_26837_b200 as P
    lengths, steps = [300, 311, 47], 40       # some step completes a page of each request, some of none
    g = torch.Generator(device="cuda").manual_seed(7 + kind)
    kv = [torch.randn(2, n, kv_heads, 128, dtype=torch.bfloat16, device="cuda", generator=g) for n in lengths]
    q = torch.randn(steps, len(lengths), q_heads, 128, device="cuda", generator=g).to(torch.bfloat16)
    new = torch.randn(2, steps, len(lengths), kv_heads, 128, dtype=torch.bfloat16, device="cuda", generator=g)
    outs = []
    for pinned in (False, True):
        cfg = P.make_config(device=0, num_layers=1, num_q_heads=q_heads, num_kv_heads=kv_heads, max_requests=3,
                            max_context_tokens=512, partition_kind=kind, topk=60 if kind == 1 else 6, lru_buckets=8,
                            gpu_cache_pages=3 * kv_heads * 10, host_pages=3 * kv_heads * 33)
        s = P.Spin(cfg)
        reqs = [s.request_open(10) for _ in lengths]
        for r, (k, v) in zip(reqs, kv):
            s.append_kv(r, 0, k, v, k.shape[0])
        place = (lambda x: x.cpu().pin_memory()) if pinned else (lambda x: x)
        qq, nn = place(q), place(new)
        out = place(torch.zeros_like(q))
        for t in range(steps):
            s.decode_step_append(0, s.req_array(reqs), nn[0, t], nn[1, t], qq[t], out[t])
        torch.cuda.synchronize()
        assert s.stats()["error_bits"] == 0
        outs.append(out.cpu())
        s.close()
    assert torch.equal(outs[0], outs[1])
