"""The fp32 kernel (csrc/attn_f32_kernel.cu) against the fp64 oracle at the edges of its tiles: row counts around 4, 16
and 64 rows per item, contexts around its 16 / 32-token tiles, units cut across blocks (partials and merge), both
launches side by side, masked tails that hold NaN bit patterns.

Bound: scores of N(0, 1) rows are sums of D products scaled by 1/sqrt(D), so their rounding error is at most about
D * 2^-24 * |q||k|/sqrt(D) ~ 128 * 6e-8 = 8e-6 of a score of order 1 and far less on average; an output is a weighted mean of
V rows, |V| < 5, whose weights move by that much: 5 * 8e-6 = 4e-5."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
TOL = 4e-5


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("P", [8, 16, 32])
@pytest.mark.parametrize("H_q,H_kv", [(4, 1), (16, 1), (3, 3)])
def test_fp32_items_at_tile_edges(D, P, H_q, H_kv):
    from tests._util import SmallBatch, oracle_on, random_seqs
    from tests.test_gpu_matrix import run_gpu
    rng = np.random.RandomState(D + P + H_q)
    shapes = [(1, 1), (1, 15), (1, 16), (1, 33), (1, 700), (4, 31), (5, 64), (16, 32), (17, 65), (33, 97), (64, 300)]
    seqs = random_seqs(rng, shapes, H_q, H_kv, D)
    seqs[6]["mask"] = rng.rand(5, 64) < 0.5              # an explicit mask, one row of it empty
    seqs[6]["mask"][2] = False
    args = SmallBatch(seqs, H_q).paged(P, order="random", seed=3)
    total = max(args["pool"]) + 1
    gpu_args = dict(args, pool={p: (k.copy(), v.copy()) for p, (k, v) in args["pool"].items()})
    O_ref, L_ref = oracle_on(args)
    for options in ({}, {2: 1}):                         # one launch after the other, and side by side
        O, L, info = run_gpu(gpu_args, total, H_kv, D, "f32", 0, options)
        assert info["num_simple_rows"] == 0 and info["num_tile_items"] > 0
        assert np.abs(O - O_ref).max() <= TOL
        neg = np.isneginf(L_ref)
        assert np.array_equal(np.isneginf(L), neg) and np.abs(L[~neg] - L_ref[~neg]).max() <= TOL


def test_fp32_unit_cut_across_blocks():
    from tests._util import SmallBatch, oracle_on, random_seqs
    from tests.test_gpu_matrix import run_gpu
    rng = np.random.RandomState(1)
    for shapes in ([(1, 5000)], [(70, 2500)]):
        args = SmallBatch(random_seqs(rng, shapes, 4, 2, 64), 4).paged(16, order="random", seed=4)
        gpu_args = dict(args, pool={p: (k.copy(), v.copy()) for p, (k, v) in args["pool"].items()})
        O_ref, L_ref = oracle_on(args)
        O, L, info = run_gpu(gpu_args, max(args["pool"]) + 1, 2, 64, "f32")
        assert info["num_merge_groups"] > 0
        assert np.abs(O - O_ref).max() <= TOL and np.abs(L - L_ref).max() <= TOL


@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
@pytest.mark.parametrize("D,P", [(64, 8), (64, 16), (64, 32), (128, 16), (128, 32)])
def test_fp32_hidden_rows_may_hold_anything(D, P, bad):
    """K and V of a position that a row does not see do not reach it, even where they are infinite or NaN: a later token of
    the row's own chunk, a position hidden by an explicit mask.  Rows that see it show it."""
    import paper_2510_24051_b200 as pie
    from tests._util import SmallBatch, oracle_on, random_seqs
    from tests.test_gpu_matrix import run_gpu
    rng = np.random.RandomState(P)
    seqs = random_seqs(rng, [(40, 70), (4, 90), (2, 33)], 4, 1, D)
    seqs[1]["mask"] = rng.rand(4, 90) < 0.7
    seqs[1]["mask"][:, 50] = [False, True, False, False]
    hidden = [(0, 55), (1, 50), (2, 32)]                 # (request, position): the chunk's 26th token, masked for three rows of four, the last token
    clean = oracle_on(SmallBatch(seqs, 4).paged(P, order="random", seed=5))
    for r, j in hidden:
        seqs[r]["K"][j, 0, 3] = np.nan
        seqs[r]["V"][j] = bad
    args = SmallBatch(seqs, 4).paged(P, order="random", seed=5)
    sees = np.zeros(46, dtype=bool)
    sees[25:40] = sees[41] = sees[45] = True
    for flags in (0, pie.PIE_PLAN_FORCE_SIMPLE):
        gpu_args = dict(args, pool={p: (k.copy(), v.copy()) for p, (k, v) in args["pool"].items()})
        O, L, info = run_gpu(gpu_args, max(args["pool"]) + 1, 1, D, "f32", flags)
        assert (info["num_simple_rows"] == 0) == (flags == 0)
        assert np.abs(O[~sees] - clean[0][~sees]).max() <= TOL and np.abs(L[~sees] - clean[1][~sees]).max() <= TOL
        assert np.isnan(O[sees]).all()


def test_fp32_thousands_of_units():
    """Many short decodes: units dealt to the blocks by size, there and back, with every count left over."""
    from tests._util import SmallBatch, oracle_on, random_seqs
    from tests.test_gpu_matrix import run_gpu
    rng = np.random.RandomState(6)
    args = SmallBatch(random_seqs(rng, [(1, int(n)) for n in rng.randint(1, 25, 1301)], 8, 4, 64), 8).paged(8, order="random", seed=6)
    gpu_args = dict(args, pool={p: (k.copy(), v.copy()) for p, (k, v) in args["pool"].items()})
    O_ref, L_ref = oracle_on(args)
    O, L, info = run_gpu(gpu_args, max(args["pool"]) + 1, 4, 64, "f32")
    assert info["num_split_items"] == 1301 * 4 and info["num_merge_groups"] == 0
    assert np.abs(O - O_ref).max() <= TOL and np.abs(L - L_ref).max() <= TOL
