"""The work a serving program has this library do, as measurable cases.

A case is one pass through the public entry points: a coalesced `forward` batch (decode, prefill, mixed, token
trees, application KV policies, forks that share a prompt), a few steps of a decode loop with their planning, the
sample stage (`get_next_dist`), or moving KvPages in and out of the pool.  Sizes are those of the repository's
workloads or generic ones.  Inputs are normal values made on the GPU; contexts lie on randomly placed pages.
"""
import math
import weakref

import numpy as np
import torch

import paper_2510_24051_b200 as pie

TORCH_TYPE = {"bf16": torch.bfloat16, "f32": torch.float32}


def listed():
    shape_1b = dict(H_q=32, H_kv=8, D=64, dtype="bf16")    # attention shapes of the repository's workloads
    shape_8b = dict(H_q=32, H_kv=8, D=128, dtype="bf16")
    return [
        # A handful of interactive users: four steps of their decode loop, each planned and run.  The smallest calls:
        # host work, launches and latency are all there is.
        dict(name="decode_loop_small", kind="decode_loop", R=4, lo=100, hi=1500, steps=4, P=16, rope=False, **shape_1b),
        # The batched text-completion decode step: 64 requests on scattered pages, the plan in hand (the repository's
        # batched_decode).
        dict(name="decode_batch", kind="decode", R=64, lo=512, hi=4096, P=16, rope=False, **shape_1b),
        # A large decode batch of a larger model with positions applied inside the path.
        dict(name="decode_large_rope", kind="decode", R=120, lo=1024, hi=8192, P=16, rope=True, **shape_8b),
        # Continuous batching: prefill chunks over existing prefixes next to decodes (the repository's
        # mixed_prefill_decode).
        dict(name="mixed_step", kind="mixed", n_prefill=8, chunk_lo=512, chunk_hi=512, prefix=2048, n_decode=120, lo=1024, hi=8192,
             P=16, rope=False, **shape_8b),
        # Fresh prompts of ragged lengths, no prefix, 32-token pages, positions inside the path.
        dict(name="prompts", kind="mixed", n_prefill=5, chunk_lo=300, chunk_hi=4000, prefix=0, n_decode=0, lo=1, hi=1, P=32,
             rope=True, **shape_1b),
        # Forked branches that share a prompt and verify a speculative token tree each (the repository's
        # shared_prefix_tree).  The largest tensor-bound batch.
        dict(name="tree_verify", kind="tree", groups=16, branches=16, prefix=4096, suffix=256, nodes=64, P=16, rope=False, **shape_8b),
        # Long contexts under an application's KV policy - sink, window, a fifth of the pages between - and a copy of
        # every request's last page (the repository's long_context_policy).  The largest memory-bound batch.
        dict(name="long_context_policy", kind="policy", R=256, lo=16384, hi=32768, window=2048, keep=0.2, P=16, rope=False, **shape_8b),
        # Parallel samples of a prompt: branches share the prompt's pages, one token each (the repository's
        # shared_prefix_decode).
        dict(name="parallel_samples", kind="shared", groups=16, branches=32, prefix=4096, lo=16, hi=256, P=16, rope=False, **shape_8b),
        # The small fp32 path (numerical debugging, fp32 models): decodes and short prefill chunks.
        dict(name="fp32_mixed", kind="mixed", n_prefill=4, chunk_lo=8, chunk_hi=100, prefix=1000, n_decode=20, lo=17, hi=2000, P=16,
             rope=False, H_q=32, H_kv=8, D=64, dtype="f32"),
        # The sample stage after a decode step: bf16 logits of 64 rows, the default top 256 (the repository's next_dist).
        dict(name="next_dist_batch", kind="next_dist", rows=64, vocab=128256, top_k=256, dtype="bf16"),
        # The same with fp32 logits of a smaller batch and an odd vocabulary.
        dict(name="next_dist_f32", kind="next_dist", rows=24, vocab=50257, top_k=100, dtype="f32"),
        # Export / import and fork: pages written from and read back into canonical tensors, token ranges copied.
        dict(name="page_moves", kind="pages", n=384, P=16, **shape_8b),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["decode", "decode", "decode", "decode_loop", "mixed", "mixed", "prompts", "tree", "policy", "shared", "fp32",
                       "next_dist", "next_dist", "pages"])
    if kind == "next_dist":
        vocab = _log_int(rng, 4000, 160000)
        if rng.random() < 0.5:
            vocab = (vocab + 63) // 64 * 64
        return dict(kind=kind, rows=_log_int(rng, 1, 512), vocab=vocab, top_k=rng.choice([1, 20, 50, 256, 256, 256, rng.randint(2, 1024)]),
                    dtype=rng.choice(["bf16", "bf16", "f32"]))
    H_q, H_kv = rng.choice([(32, 8), (32, 8), (32, 8), (16, 8), (16, 2), (12, 12)])
    c = dict(P=rng.choice([8, 16, 16, 16, 32]), H_q=H_q, H_kv=H_kv, D=rng.choice([64, 128]), dtype="bf16")
    if kind == "pages":
        return dict(kind=kind, n=_log_int(rng, 8, 1500), **c)
    c["rope"] = rng.random() < 0.3
    if kind == "fp32":
        hi = _log_int(rng, 30, 2000)
        c["dtype"] = "f32"
        return dict(kind="mixed", n_prefill=rng.randint(0, 4), chunk_lo=2, chunk_hi=_log_int(rng, 8, 100), prefix=hi,
                    n_decode=_log_int(rng, 1, 32), lo=10, hi=hi, **c)
    if kind == "decode":
        hi = _log_int(rng, 200, 16000)
        return dict(kind=kind, R=_log_int(rng, 1, 256), lo=max(1, hi // rng.choice([2, 8, 20])), hi=hi, **c)
    if kind == "decode_loop":
        hi = _log_int(rng, 200, 6000)
        return dict(kind=kind, R=_log_int(rng, 1, 96), lo=max(1, hi // 8), hi=hi, steps=4, **c)
    if kind == "mixed":
        hi = _log_int(rng, 300, 8000)
        chunk = _log_int(rng, 32, 512)
        return dict(kind=kind, n_prefill=rng.randint(1, 8), chunk_lo=max(8, chunk // rng.choice([1, 1, 4])), chunk_hi=chunk,
                    prefix=_log_int(rng, 16, 2048), n_decode=_log_int(rng, 2, 120), lo=max(1, hi // 8), hi=hi, **c)
    if kind == "prompts":
        hi = _log_int(rng, 64, 4096)
        return dict(kind="mixed", n_prefill=rng.randint(1, 6), chunk_lo=max(17, hi // rng.choice([1, 4, 10])), chunk_hi=max(17, hi), prefix=0,
                    n_decode=0, lo=1, hi=1, **c)
    if kind == "tree":
        return dict(kind=kind, groups=rng.randint(1, 12), branches=rng.randint(2, 16), prefix=32 * rng.randint(4, 128),
                    suffix=32 * rng.randint(1, 8), nodes=rng.choice([8, 16, 24, 32, 48, 64]), **c)
    if kind == "policy":
        hi = _log_int(rng, 4096, 32768)
        return dict(kind=kind, R=_log_int(rng, 4, 160), lo=hi // 2, hi=hi, window=rng.choice([256, 1024, 2048]), keep=rng.choice([0.1, 0.2, 0.5]),
                    **c)
    return dict(kind="shared", groups=rng.randint(1, 12), branches=_log_int(rng, 2, 32), prefix=32 * rng.randint(8, 128), lo=16,
                hi=rng.randint(32, 400), **c)


# ------------------------------------------------------------------------------------ the batches
def _requests(case):
    """Query and context length of every request and the group whose prompt it shares (None: nothing is shared).
    Lengths belong to the case: the seed of prepare() moves pages, masks and values only."""
    kind, rng = case["kind"], np.random.RandomState(1)
    if kind in ("decode", "decode_loop", "policy"):
        kv = rng.randint(case["lo"], case["hi"] + 1, case["R"])
        return np.ones_like(kv), kv, None
    if kind == "mixed":
        chunk = rng.randint(case["chunk_lo"], case["chunk_hi"] + 1, case["n_prefill"])
        prefix = rng.randint(0, case["prefix"] + 1, case["n_prefill"])
        dec = rng.randint(case["lo"], case["hi"] + 1, case["n_decode"])
        return np.concatenate([chunk, np.ones_like(dec)]), np.concatenate([chunk + prefix, dec]), None
    R = case["groups"] * case["branches"]
    shared = np.repeat(np.arange(case["groups"]), case["branches"])
    if kind == "tree":
        return np.full(R, case["nodes"]), np.full(R, case["prefix"] + case["suffix"] + case["nodes"]), shared
    return np.ones(R, dtype=np.int64), case["prefix"] + rng.randint(case["lo"], case["hi"] + 1, R) + 1, shared


def _masks(case, rng, kv):
    """Explicit masks (one bool matrix per request), or None for the inferred causal masks."""
    P = case["P"]
    if case["kind"] == "policy":
        out = []
        for n in kv:
            m = np.zeros(n, dtype=np.uint8)
            w0 = max(int(n) - case["window"], 0)
            m[w0:], m[:4] = 1, 1
            mid = w0 // P - 1                      # pages between the sink's page and the window
            if mid > 0:
                for p in 1 + rng.permutation(mid)[:int(round(case["keep"] * mid))]:
                    m[p * P:(p + 1) * P] = 1
            out.append(m)
        return out
    if case["kind"] == "tree":
        out, n = [], case["nodes"]
        for k in kv:
            anc = np.eye(n, dtype=np.uint8)
            for i in range(1, n):
                anc[i] |= anc[rng.randint(i)]      # a parent drawn among the earlier nodes: its ancestors, and itself
            m = np.ones((n, int(k)), dtype=np.uint8)
            m[:, int(k) - n:] = anc
            out.append(m)
        return out
    return None


class _Session:
    """What a serving program holds: the context with its pool, a plan, tensors.  Freed with the object."""

    def __init__(self, kind, *config, **options):
        self.kind, self.plan = kind, None
        self.ctx = pie.pie_create(*config, **options)
        self._held = {"ctx": self.ctx}
        weakref.finalize(self, _release, self._held)

    def keep_plan(self, batch):
        self.plan = self._held["plan"] = pie.pie_plan_forward(self.ctx, **batch)


def _release(held):
    if "plan" in held:
        pie.pie_plan_destroy(held["plan"])
    pie.pie_destroy(held["ctx"])


def _page_lists(case, q, kv, group, extra_tokens, rng):
    P, R = case["P"], len(q)
    n_pages = (kv + extra_tokens + P - 1) // P
    n_shared = 0 if group is None else case["prefix"] // P
    need = int(n_pages.sum()) if group is None else int((n_pages - n_shared).sum()) + n_shared * case["groups"]
    num_pages = need + need // 8 + 8
    order = rng.permutation(num_pages).astype(np.int32)
    lists, at = [], 0
    heads = []
    if group is not None:
        for _ in range(case["groups"]):
            heads.append(order[at:at + n_shared])
            at += n_shared
    for r in range(R):
        own = int(n_pages[r]) - n_shared
        mine = order[at:at + own]
        at += own
        lists.append(mine if group is None else np.concatenate([heads[group[r]], mine]))
    return num_pages, order[:at], lists, order[at:]


def _batch(case, q, kv, lists, masks):
    P = case["P"]
    n_pages = (kv + P - 1) // P
    b = dict(qo_indptr=np.concatenate([[0], np.cumsum(q)]).astype(np.int32),
             page_indptr=np.concatenate([[0], np.cumsum(n_pages)]).astype(np.int32),
             page_indices=np.concatenate([p[:n] for p, n in zip(lists, n_pages)]).astype(np.int32),
             last_page_len=(kv - (n_pages - 1) * P).astype(np.int32))
    if masks is not None:
        b["mask_indptr"] = np.concatenate([[0], np.cumsum([m.size for m in masks])]).astype(np.int64)
        b["mask"] = np.concatenate([m.reshape(-1) for m in masks])
    return b


def _normal(gen, shape, dtype):
    return torch.randn(shape, generator=gen, device="cuda", dtype=TORCH_TYPE[dtype])


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    rng = np.random.RandomState(seed % (1 << 32))
    kind = case["kind"]
    if kind == "next_dist":
        s = _Session(kind, 4, 16, 4, 2, 64, "bf16", 4, 64, 0)
        s.logits = (_normal(gen, (case["rows"], case["vocab"]), "f32") * 2.5).to(TORCH_TYPE[case["dtype"]])
        s.top_k = case["top_k"]
        s.ids = torch.empty(case["rows"], s.top_k, dtype=torch.int32, device="cuda")
        s.probs = torch.empty(case["rows"], s.top_k, dtype=torch.float32, device="cuda")
        return s
    P, H_q, H_kv, D, dtype = (case[k] for k in ("P", "H_q", "H_kv", "D", "dtype"))
    if kind == "pages":
        n = case["n"]
        s = _Session(kind, 3 * n, P, H_q, H_kv, D, dtype, 4, 64, 0)
        ids = pie.pie_alloc_kvpages(s.ctx, 3 * n)[rng.permutation(3 * n)]
        s.src, s.dst = ids[:n].copy(), ids[n:2 * n].copy()
        s.K, s.V = _normal(gen, (n, P, H_kv, D), dtype), _normal(gen, (n, P, H_kv, D), dtype)
        s.K_out, s.V_out = torch.empty_like(s.K), torch.empty_like(s.V)
        s.ntok = rng.randint(1, P + 1, n).astype(np.int32)
        s.src_off = (rng.rand(n) * (P - s.ntok + 1)).astype(np.int32)
        s.dst_off = (rng.rand(n) * (P - s.ntok + 1)).astype(np.int32)
        return s
    q, kv, group = _requests(case)
    steps = case.get("steps", 1)
    num_pages, used, lists, spare = _page_lists(case, q, kv, group, steps - 1, rng)
    T = int(q.sum())
    s = _Session(kind, num_pages, P, H_q, H_kv, D, dtype, len(q), T, 0, rope_theta=500000.0 if case["rope"] else 0.0)
    pie.pie_alloc_kvpages(s.ctx, num_pages)
    chunk = max(1, (256 << 20) // (P * H_kv * D * 4))
    for i in range(0, len(used), chunk):
        ids = used[i:i + chunk]
        pie.pie_kvpage_write(s.ctx, ids, _normal(gen, (len(ids), P, H_kv, D), dtype), _normal(gen, (len(ids), P, H_kv, D), dtype))
    s.batches = [_batch(case, q, kv + k, lists, _masks(case, rng, kv)) for k in range(steps)]
    s.tensors = []
    for _ in range(steps):
        x = [_normal(gen, (T, h, D), dtype) for h in (H_q, H_kv, H_kv)]
        s.tensors.append(x + [torch.empty_like(x[0]), torch.empty(T, H_q, dtype=torch.float32, device="cuda")])
    if kind != "decode_loop":
        s.keep_plan(s.batches[0])
    if kind == "policy":     # (after the forward) every request's last page is copied to a fresh one
        zero = np.zeros(len(q), dtype=np.int32)
        s.copy = (np.array([p[-1] for p in lists], dtype=np.int32), spare[:len(q)].copy(), zero, zero, s.batches[0]["last_page_len"])
    return s


# ------------------------------------------------------------------------------------ one pass
def run(s):
    if s.kind == "next_dist":
        pie.pie_get_next_dist(s.ctx, s.logits, s.top_k, s.ids, s.probs)
        return s.ids, s.probs
    if s.kind == "pages":
        pie.pie_kvpage_write(s.ctx, s.src, s.K, s.V)
        pie.pie_copy_kvpage(s.ctx, s.src, s.dst, s.src_off, s.dst_off, s.ntok)
        pie.pie_kvpage_read(s.ctx, s.dst, s.K_out, s.V_out)
        return s.K_out, s.V_out
    if s.kind == "decode_loop":
        for b, x in zip(s.batches, s.tensors):
            plan = pie.pie_plan_forward(s.ctx, **b)
            pie.pie_forward(s.ctx, plan, *x)
            pie.pie_plan_destroy(plan)
        return [x[3:] for x in s.tensors]
    x = s.tensors[0]
    pie.pie_forward(s.ctx, s.plan, *x)
    if s.kind == "policy":
        pie.pie_copy_kvpage(s.ctx, *s.copy)
    return x[3:]


# ------------------------------------------------------------------------------------ what a pass cannot do without
def work(case):
    kind = case["kind"]
    if kind == "next_dist":
        n = case["rows"] * case["vocab"]
        return {"bytes": n * (2 if case["dtype"] == "bf16" else 4) + case["rows"] * case["top_k"] * 8, "flops": 2 * n}
    P, H_q, H_kv, D = (case[k] for k in ("P", "H_q", "H_kv", "D"))
    es = 2 if case["dtype"] == "bf16" else 4
    token = 2 * H_kv * D * es                                     # K and V of one token
    if kind == "pages":
        return {"bytes": case["n"] * P * token * 4 + case["n"] * (P + 1) * token, "flops": 0}
    q, kv, group = _requests(case)
    steps = case.get("steps", 1)
    kept = kv.copy()
    if kind == "policy":
        kept = np.array([int(m.sum()) for m in _masks(case, np.random.RandomState(1), kv)])
    pairs = q * kv - q * (q - 1) // 2 if kind != "policy" else kept
    if kind == "tree":
        pairs = q * (kv - q) + q * (q - 1) // 8                   # (ancestors: a few per node)
    tokens = int(kept.sum())
    if group is not None:                                         # a shared prefix is read once per group
        tokens -= case["prefix"] * (len(q) - case["groups"])
    T = int(q.sum())
    rows = T * H_q * (2 * D * es + 4) + 2 * T * token             # Q, O, LSE; the new rows read and stored
    return {"bytes": float(steps * (tokens * token + rows)), "flops": float(steps * 4 * D * H_q * int(pairs.sum()))}


def tolerance(case):
    # About four times what was measured: bf16 outputs against the same batch with fp32 probabilities 2.3e-3, fp32
    # outputs against fp64 6.5e-7, probabilities of the sample stage against fp64 6e-8 (another exponential: more).
    if case["kind"] == "pages":
        return "exact"
    if case["kind"] == "next_dist":
        return {"rel": 1e-6, "differ": 0.0}                       # (the token ids are exact)
    return {"rel": 4e-6} if case["dtype"] == "f32" else {"rel": 9e-3}
