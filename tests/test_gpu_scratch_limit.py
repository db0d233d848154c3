"""pie_forward_static_scratch with batches whose fastest plan - units cut across the chip, fp32 partials of every piece - does not
fit PIE_STATIC_SCRATCH_BYTES: they are laid out again with fewer partials and give the planned forward's results within rounding.
Bound: both are bf16 (fp32) results of the same inputs that sum in another order; twice the acceptance tolerance against fp64."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,H_q,H_kv,D,P,q,kv,masked", [
    ("bf16", 32, 1, 128, 32, [1] * 40, [1100 + 45 * r for r in range(40)], False),                       # multi-query decodes, as row tiles
    ("bf16", 32, 8, 128, 16, [107, 203, 1, 1, 1, 59, 1, 1, 1, 1, 1], [3111, 1763, 2910, 3930, 3741, 1162, 882, 860, 1142, 910, 2488], False),
    ("bf16", 16, 2, 128, 16, [1, 1, 262, 1, 262, 1, 1, 1, 1, 183, 1, 1, 1, 1],
     [635, 1673, 747, 293, 3716, 726, 2595, 1784, 2581, 710, 1103, 1455, 2219, 837], False),
    ("f32", 4, 1, 128, 32, [64] * 40, [24576] * 40, True),                                                # 8 MB of mask words beside 10 MB of partials
])
def test_plans_beyond_the_scratch_are_laid_out_again(dtype, H_q, H_kv, D, P, q, kv, masked):
    import paper_2510_24051_b200 as pie
    from tests._gpu import TDTYPE, TOL_LSE, TOL_O
    q, kv = np.array(q), np.array(kv)
    pages = (kv + P - 1) // P
    n, T, tdt = int(pages.sum()), int(q.sum()), TDTYPE[dtype]
    ctx = pie.pie_create(n, P, H_q, H_kv, D, dtype, len(q), T, 0)
    try:
        pie.pie_set_option(ctx, pie.PIE_OPT_OVERLAP, 2)
        ids = pie.pie_alloc_kvpages(ctx, n)
        g = torch.Generator(device="cuda").manual_seed(1)
        rand = lambda *shape: torch.randn(shape, generator=g, device="cuda", dtype=tdt)
        for i in range(0, n, 4096):
            m = len(ids[i:i + 4096])
            pie.pie_kvpage_write(ctx, ids[i:i + 4096], rand(m, P, H_kv, D), rand(m, P, H_kv, D))
        batch = [np.concatenate([[0], np.cumsum(q)]), np.concatenate([[0], np.cumsum(pages)]), ids, kv - (pages - 1) * P]
        mi = np.concatenate([[0], np.cumsum(q.astype(np.int64) * kv)]) if masked else None
        mask = (np.arange(int(mi[-1])) % 7 != 3).astype(np.uint8) if masked else None
        x = [rand(T, H_q, D), rand(T, H_kv, D), rand(T, H_kv, D)]
        ref, out = [(torch.zeros_like(x[0]), torch.zeros(T, H_q, device="cuda")) for _ in range(2)]
        plan = pie.pie_plan_forward(ctx, *batch, mi, mask)
        assert pie.pie_plan_get_info(plan)["workspace_bytes"] + pie.pie_plan_debug_read(plan, 3).nbytes > pie.PIE_STATIC_SCRATCH_BYTES
        pie.pie_forward(ctx, plan, *x, *ref)
        pie.pie_forward_static_scratch(ctx, *batch, *x, *out, mi, mask)
        torch.cuda.synchronize()
        assert pie.pie_get_last_device_status(ctx) == 0
        assert (out[0].double() - ref[0].double()).abs().max() <= 2 * TOL_O[dtype]
        assert (out[1] - ref[1]).abs().max() <= 2 * TOL_LSE
        pie.pie_plan_destroy(plan)
    finally:
        torch.cuda.synchronize()
        pie.pie_destroy(ctx)
