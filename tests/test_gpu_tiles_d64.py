"""Row tiles of 64-wide heads: every KV tile's two halves belong to different warpgroups, whose partial rows meet in the
epilogue.  Items of one half, of an odd number of halves, of one and of two Q tiles, rows past the end of an item, masks that
leave a half - or a whole row - without any position, and scores that outgrow the reference late in one half only, against
the fp64 oracle at the acceptance tolerance."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _run(shapes, H_q, H_kv, P, masks=None, seed=0, peak=None):
    import torch
    from tests._gpu import check_close
    from tests._util import SmallBatch, oracle_on, random_seqs
    from tests.test_gpu_matrix import run_gpu
    seqs = random_seqs(np.random.RandomState(seed), shapes, H_q, H_kv, 64, masks)
    for s in seqs:
        if peak is not None and len(s["K"]) > peak:
            s["K"][peak] *= 24.0                 # one position far above the rest: the sums of the half before it are rescaled
        for k in "QKV":
            s[k] = torch.from_numpy(s[k]).bfloat16().float().numpy()
    args = SmallBatch(seqs, H_q).paged(P, order="random", seed=seed)
    O_ref, L_ref = oracle_on(dict(args, pool={p: (k.copy(), v.copy()) for p, (k, v) in args["pool"].items()}))
    O, L, info = run_gpu(args, max(args["pool"]) + 1, H_kv, 64, "bf16")
    assert info["num_tile_items"] > 0
    check_close(O, L, O_ref, L_ref, "bf16", args["qo_indptr"])


@pytest.mark.parametrize("P", [8, 16, 32])
@pytest.mark.parametrize("shapes", [[(20, 20), (40, 64)], [(33, 65), (64, 128)], [(70, 129), (17, 191), (130, 257)]])
def test_halves_and_partial_tiles(P, shapes):
    _run(shapes, 8, 2, P, seed=P)


@pytest.mark.parametrize("peak", [70, 190, 254])
def test_reference_grows_in_one_half(peak):
    _run([(80, 300), (64, 256)], 8, 2, 16, seed=peak, peak=peak)


def test_masks_without_positions_in_a_half():
    rng = np.random.RandomState(5)
    masks = [rng.rand(48, 256) < 0.4, rng.rand(40, 200) < 0.5]
    masks[0][:, 64:128] = False                  # no position in the second half of the first tile
    masks[0][:24, :64] = False
    masks[1][7, :] = False                       # an empty row
    masks[1][9, :190] = False
    _run([(48, 256), (40, 200)], 8, 2, 16, masks)


@pytest.mark.parametrize("P", [8, 16, 32])
def test_nan_key_shows_at_every_position(P):
    """A NaN key that every row sees reaches every output of its kv head - no output of another - wherever it lies in a KV tile."""
    from tests._util import SmallBatch, random_seqs
    from tests.test_gpu_matrix import run_gpu
    seqs = random_seqs(np.random.RandomState(P), [(64, 1024)], 8, 2, 64)
    args = SmallBatch(seqs, 8).paged(P, order="random", seed=P)
    lse = []
    for pos in (0, 1, 2, 16, 17, 47, 64, 65, 80, 127, 256, 272, 959):
        page, slot = args["page_indices"][pos // P], pos % P
        pool = {p: (k.copy(), v.copy()) for p, (k, v) in args["pool"].items()}
        pool[int(page)][0][slot, 0, 5] = np.nan
        O, L, info = run_gpu(dict(args, pool=pool), max(pool) + 1, 2, 64, "bf16")
        assert info["num_tile_items"] > 0
        assert np.isnan(O[:, :4]).all(), pos
        assert np.isfinite(O[:, 4:]).all() and np.isfinite(L[:, 4:]).all(), pos
        lse.append(L[:, :4])
    assert all(np.array_equal(x, lse[0], equal_nan=True) for x in lse)
