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


def _placed(kind, n, V, seed):
    """Rows whose K-th largest logit lies far below the largest: other sign, log-probabilities with a confident top, a common
    offset that leaves fp32 little resolution, most of the vocabulary masked out (in one run, or all but every 37th token),
    and all of it."""
    g = torch.Generator().manual_seed(seed)
    x = torch.randn(n, V, generator=g) * 2.5
    if kind == "negative":
        x = x - 8
        x[:, 3] = 1.5
    elif kind == "confident":
        x[:, V // 2] += 40
        x = torch.log_softmax(x, -1)
    elif kind == "offset":
        x = x + 1000
    elif kind == "far offset":
        x = x + 1e6
    elif kind == "half masked":
        x[:, V // 2:] = float("-inf")
    elif kind == "few allowed":
        x[:, V // 90 + 1:] = float("-inf")
    elif kind == "every 37th":
        keep = torch.arange(V) % 37 == 5
        keep[1] = True
        x[:, ~keep] = float("-inf")
    elif kind == "lowest":
        x[:, V // 2:] = torch.finfo(torch.float32).min
        x[:, 9:V // 2] = float("-inf")
    return x


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("kind", ["negative", "confident", "offset", "far offset", "half masked", "few allowed", "every 37th", "lowest"])
def test_thresholds_beyond_the_histogram(kind, dtype):
    from tests.test_gpu_next_dist import _check
    for n, V, K in ((1, 40003, 256), (3, 9001, 1000), (40, 17000, 50), (160, 8000, 256), (2, 700, 256), (1, 70001, 1024)):
        _check(_placed(kind, n, V, seed=V).to(dtype).cuda(), K)


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("n,V", [(64, 128256), (1, 128256), (512, 8000)])
def test_time_does_not_depend_on_where_the_logits_lie(n, V, dtype):
    """A common offset or a confident top costs at most a second threshold (about 10 us), not the row again on one block: 4 - 27
    times the time of centred logits while such rows were left to the radix selection, 1.0 - 2.1 times since."""
    import paper_2510_24051_b200 as pie
    from tests.test_gpu_next_dist import _ctx
    ids = torch.empty(n, 256, dtype=torch.int32, device="cuda")
    probs = torch.empty(n, 256, dtype=torch.float32, device="cuda")
    ctx = _ctx()

    def us(x):
        for _ in range(3):
            pie.pie_get_next_dist(ctx, x, 256, ids, probs)
        best = 1e9
        for _ in range(5):
            torch.cuda.synchronize()
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(20):
                pie.pie_get_next_dist(ctx, x, 256, ids, probs)
            b.record()
            b.synchronize()
            best = min(best, a.elapsed_time(b) * 50)
        return best
    try:
        centred = us(_placed("", n, V, 1).to(dtype).cuda())
        for kind in ("negative", "confident"):
            assert us(_placed(kind, n, V, 1).to(dtype).cuda()) <= 2.5 * centred + 2, kind
    finally:
        torch.cuda.synchronize()
        pie.pie_destroy(ctx)
