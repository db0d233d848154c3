"""pie_plan_forward only enqueues its upload: forwards on the planning stream, on another stream and inside a captured graph
must all see it, and plans recycled while earlier ones are still in flight must not disturb them.  Results are compared
bit for bit with the same batches run one at a time (the kernels are deterministic)."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def _loop_batches(n_steps):
    from workloads import configs
    wl = configs.small("batched_decode")
    spare = np.setdiff1d(np.arange(wl.num_pages), wl.used_pages())
    return wl, configs.decode_loop(wl, n_steps, spare)


def test_plans_in_flight_on_one_and_on_two_streams():
    import paper_2510_24051_b200 as pie
    from tests._gpu import GpuPool
    wl, steps = _loop_batches(12)
    with GpuPool(wl.num_pages, wl.P, wl.H_q, wl.H_kv, wl.D, wl.dtype) as gp:
        gp.install(wl)
        q, k, v = wl.q("cuda"), wl.k_new("cuda"), wl.v_new("cuda")
        args = [{n: b[n] for n in ("qo_indptr", "page_indptr", "page_indices", "last_page_len")} for b in steps]

        def outputs():
            return [(torch.zeros_like(q), torch.zeros(wl.T, wl.H_q, device="cuda")) for _ in steps]

        ref = outputs()
        for a, o in zip(args, ref):
            plan = pie.pie_plan_forward(gp.ctx, **a)
            torch.cuda.synchronize()
            pie.pie_forward(gp.ctx, plan, q, k, v, *o)
            torch.cuda.synchronize()
            pie.pie_plan_destroy(plan)
        s1, s2 = torch.cuda.Stream(), torch.cuda.Stream()
        busy = torch.randn(4096, 4096, device="cuda")
        for other in (False, True):
            got = outputs()
            torch.cuda.synchronize()
            for i, (a, o) in enumerate(zip(args, got)):
                with torch.cuda.stream(s1):
                    if i % 3 == 0:
                        busy @ busy                       # the upload queues behind this
                    plan = pie.pie_plan_forward(gp.ctx, **a)
                with torch.cuda.stream(s2 if other else s1):
                    pie.pie_forward(gp.ctx, plan, q, k, v, *o)
                pie.pie_plan_destroy(plan)
            torch.cuda.synchronize()
            for (o, l), (o_ref, l_ref) in zip(got, ref):
                assert torch.equal(o, o_ref) and torch.equal(l, l_ref)
        # captured right behind the planning, on another stream than the one that uploads
        o = (torch.zeros_like(q), torch.zeros(wl.T, wl.H_q, device="cuda"))
        torch.cuda.synchronize()
        with torch.cuda.stream(s1):
            busy @ busy
            plan = pie.pie_plan_forward(gp.ctx, **args[5])
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s2):
            pie.pie_forward(gp.ctx, plan, q, k, v, *o)
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(o[0], ref[5][0]) and torch.equal(o[1], ref[5][1])
        del g
        pie.pie_plan_destroy(plan)
        assert pie.pie_get_last_device_status(gp.ctx) == 0
