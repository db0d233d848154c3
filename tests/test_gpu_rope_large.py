"""Positions inside the path: a batch large enough for the rotation's small blocks stores the same bits, and attends to the
same values, as its requests one at a time (the other block size, held to the oracle in test_gpu_parity.py)."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D,q_len,R", [(64, 237, 11), (128, 131, 11)])
def test_large_batch_equals_its_requests(D, q_len, R):
    import paper_2510_24051_b200 as pie
    from tests._gpu import TOL_O
    P, H_q, H_kv = 16, 4, 2
    n = (q_len + P - 1) // P
    gen = torch.Generator(device="cuda").manual_seed(D)
    x = [torch.randn((R * q_len, h, D), generator=gen, device="cuda").to(torch.bfloat16) for h in (H_q, H_kv, H_kv)]

    def run(requests):
        rows = torch.cat([torch.arange(r * q_len, (r + 1) * q_len, device="cuda") for r in requests])
        k = len(requests)
        ctx = pie.pie_create(R * n, P, H_q, H_kv, D, "bf16", R, R * q_len, 0, rope_theta=10000.0)
        try:
            ids = pie.pie_alloc_kvpages(ctx, k * n)
            plan = pie.pie_plan_forward(ctx, np.arange(k + 1) * q_len, np.arange(k + 1) * n, ids, np.full(k, (q_len - 1) % P + 1))
            t = [y[rows].contiguous() for y in x]
            out, lse = torch.empty_like(t[0]), torch.empty((k * q_len, H_q), device="cuda")
            pie.pie_forward(ctx, plan, *t, out, lse)
            K = torch.zeros((k * n, P, H_kv, D), dtype=torch.bfloat16, device="cuda")
            V = torch.zeros_like(K)
            pie.pie_kvpage_read(ctx, ids, K, V)
            torch.cuda.synchronize()
            assert pie.pie_get_last_device_status(ctx) == 0
            pie.pie_plan_destroy(plan)
            keep = lambda y: y.view(k, n * P, H_kv, D)[:, :q_len].clone()   # (slots past the end hold anything)
            return keep(K), keep(V), out, lse
        finally:
            pie.pie_destroy(ctx)

    assert R * q_len * D >= 2 * 512 * torch.cuda.get_device_properties(0).multi_processor_count
    K, V, out, lse = run(list(range(R)))
    for r in (0, R // 2, R - 1):
        K1, V1, out1, lse1 = run([r])
        assert torch.equal(K[r].view(torch.int16), K1[0].view(torch.int16)) and torch.equal(V[r].view(torch.int16), V1[0].view(torch.int16))
        o = out[r * q_len:(r + 1) * q_len].float()
        assert (o - out1.float()).abs().max() <= 2 * TOL_O["bf16"]     # (both within the tolerance of the exact result)
