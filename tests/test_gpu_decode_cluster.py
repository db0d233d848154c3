"""Decode launches whose units own a cluster of thread blocks, or a block of 8, 4, 2 or 1 warps (decode_cluster_kernel), against
the fp64 oracle at the acceptance tolerance: every width the planner can pick, contexts shorter than the unit has warps, odd
pages at the end of a piece, two query tokens and explicit masks, and one unit far longer than the others."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _run(shapes, H_q, H_kv, D, P, masks=None, seed=0):
    import torch
    from tests._gpu import check_close
    from tests._util import SmallBatch, oracle_on, random_seqs
    from tests.test_gpu_matrix import run_gpu
    rng = np.random.RandomState(seed)
    seqs = random_seqs(rng, shapes, H_q, H_kv, D, masks)
    for s in seqs:
        for k in "QKV":
            s[k] = torch.from_numpy(s[k]).bfloat16().float().numpy()
    args = SmallBatch(seqs, H_q).paged(P, order="random", seed=seed)
    gpu_args = dict(args, pool={p: (k.copy(), v.copy()) for p, (k, v) in args["pool"].items()})
    O_ref, L_ref = oracle_on(args)
    total = max(args["pool"]) + 1
    O, L, info = run_gpu(gpu_args, total, H_kv, D, "bf16")
    O2, L2, info2 = run_gpu(gpu_args, total, H_kv, D, "bf16", options={3: 16})
    check_close(O, L, O_ref, L_ref, "bf16", args["qo_indptr"])
    check_close(O2, L2, O_ref, L_ref, "bf16", args["qo_indptr"])
    return info, info2


@pytest.mark.parametrize("H_q,H_kv,D,P", [(8, 2, 64, 16), (8, 2, 64, 8), (4, 2, 128, 16), (4, 2, 128, 8), (4, 2, 128, 32), (4, 2, 64, 32), (9, 3, 64, 8)])
@pytest.mark.parametrize("R,hi", [(1, 1900), (7, 700), (14, 400), (30, 200), (70, 100), (160, 60)])
def test_every_width_matches_oracle(H_q, H_kv, D, P, R, hi):
    rng = np.random.RandomState(R)
    kv = [hi] + [int(x) for x in rng.randint(1, hi + 1, R - 1)]
    info, _ = _run([(1, n) for n in kv], H_q, H_kv, D, P, seed=R)
    assert info["num_merge_groups"] == 0 and info["launches"] == 1


@pytest.mark.parametrize("D,P", [(64, 16), (128, 8)])
def test_two_query_tokens_and_masks(D, P):
    rng = np.random.RandomState(2)
    shapes = [(2, 300), (1, 17), (2, 2), (2, 77)]
    masks = [rng.rand(2, 300) < 0.3, None, None, rng.rand(2, 77) < 0.5]
    masks[0][1, :] = False                           # an empty row
    masks[0][0, 5] = True
    info, _ = _run(shapes, 8, 2, D, P, masks)
    assert info["num_tile_items"] == 0


@pytest.mark.parametrize("H_q,H_kv,D,P,long,short,R", [(12, 12, 64, 8, 20, 5, 210), (4, 2, 128, 16, 1500, 900, 24), (4, 2, 128, 32, 700, 100, 100)])
def test_more_units_than_are_resident_at_once(H_q, H_kv, D, P, long, short, R):
    """Blocks (or clusters) that start when others end: the largest units first, whatever their place in the batch."""
    rng = np.random.RandomState(R)
    kv = [int(x) for x in rng.randint(1, short + 1, R)]
    for k in (1, R // 2, R - 1):
        kv[k] = long
    info, _ = _run([(1, n) for n in kv], H_q, H_kv, D, P, seed=R)
    assert info["num_merge_groups"] == 0 and info["launches"] == 1
