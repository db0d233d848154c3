"""Page import / export and copy_kvpage at the sizes of their parameter blocks (256, 1,536 and 8,000 words per launch) and
with head counts that are no power of two: bit for bit against index arithmetic on the canonical layout."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,P,H_kv,D,dtype", [(1, 16, 8, 128, "bf16"), (85, 32, 3, 64, "f32"), (86, 8, 12, 64, "bf16"), (256, 16, 5, 128, "bf16"),
                                              (257, 16, 1, 64, "f32"), (512, 8, 2, 64, "bf16"), (513, 8, 2, 64, "bf16"),
                                              (1537, 8, 1, 64, "bf16"), (2667, 8, 1, 64, "bf16"), (8001, 8, 1, 64, "bf16")])
def test_pages_in_out_and_copied(n, P, H_kv, D, dtype):
    import paper_2510_24051_b200 as pie
    rng = np.random.RandomState(n)
    tdt = torch.bfloat16 if dtype == "bf16" else torch.float32
    ctx = pie.pie_create(2 * n + 3, P, H_kv, H_kv, D, dtype, 4, 64, 0)
    try:
        ids = pie.pie_alloc_kvpages(ctx, 2 * n + 3)[rng.permutation(2 * n + 3)]
        src, dst = ids[:n].copy(), ids[n:2 * n].copy()
        K, V, K0, V0 = (torch.randn(n, P, H_kv, D, device="cuda").to(tdt) for _ in range(4))
        pie.pie_kvpage_write(ctx, src, K, V)
        pie.pie_kvpage_write(ctx, dst, K0.cpu() if n < 300 else K0, V0.cpu() if n < 300 else V0)   # (host memory too)
        ntok = rng.randint(0, P + 1, n)
        so, do = (rng.rand(2, n) * (P - ntok + 1)).astype(np.int64)
        pie.pie_copy_kvpage(ctx, src, dst, so, do, ntok)
        for got, was, new in zip(_read(pie, ctx, dst, K), (K0, V0), (K, V)):
            slot = torch.arange(P)[None]
            o, d, c = (torch.as_tensor(x)[:, None] for x in (so, do, ntok))
            hit = ((slot >= d) & (slot < d + c)).cuda()
            take = (slot - d + o).clamp(0, P - 1).cuda()[:, :, None, None].expand_as(new)
            want = torch.where(hit[:, :, None, None], torch.gather(new, 1, take), was)
            assert torch.equal(got, want)
        for got, want in zip(_read(pie, ctx, src, K), (K, V)):
            assert torch.equal(got, want)
    finally:
        pie.pie_destroy(ctx)


def _read(pie, ctx, ids, like):
    K, V = torch.empty_like(like), torch.empty_like(like)
    pie.pie_kvpage_read(ctx, ids, K, V)
    torch.cuda.synchronize()
    return K, V
