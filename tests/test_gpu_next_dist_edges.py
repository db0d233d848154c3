"""The sample-stage kernel at the edges of its dispatch, against the fp64 oracle (ids exact, probabilities as in
test_gpu_next_dist): rows shorter than a block, parts of one batch of loads and of several, one to eight blocks per row,
every alignment of the row, K from 1 to the number of a block's maxima and beyond, logits whose range leaves the counting
sort's bins, and ties of negative logits at the K-th place."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("n,V,K", [(1, 1, 1), (3, 9, 9), (2, 511, 100), (2, 4104, 513), (1, 8191, 1024), (1, 16385, 1024), (2, 32768, 1), (1, 65544, 700),
                                   (9, 33001, 50), (40, 20000, 256), (75, 70001, 256), (150, 9000, 1024), (310, 12345, 300)])
def test_dispatch_edges(n, V, K, dtype):
    from tests.test_gpu_next_dist import _check, _logits
    _check(_logits(n, V, dtype, seed=n + V).cuda(), K)


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
def test_alignments_and_wide_ranges(dtype):
    from tests.test_gpu_next_dist import _check, _logits
    x = _logits(3, 17003, dtype, seed=4)
    for lead in range(8):
        wide = torch.zeros(3, 17003 + 21, dtype=dtype)
        wide[:, lead:lead + 17003] = x
        _check(wide.cuda()[:, lead:lead + 17003], 200)
    g = torch.Generator().manual_seed(6)
    y = torch.randn(2, 30000, generator=g)
    _check((y * 10.0 ** torch.randint(-30, 2, (2, 30000), generator=g).float()).to(dtype).cuda(), 400)   # top values spread over many binades


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("fill", [-1.5, float("-inf")])
def test_ties_of_negative_logits_at_the_last_place(dtype, fill):
    from tests.test_gpu_next_dist import _check
    z = torch.full((2, 30000), fill)
    z[:, 5:400] = torch.randn(2, 395, generator=torch.Generator().manual_seed(6)).abs()    # fewer entries above `fill` than K
    _check(z.to(dtype).cuda(), 600)
