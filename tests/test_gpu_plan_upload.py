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


def test_planning_while_a_stream_is_captured():
    """On the captured stream planning is refused and leaves the capture as it was - the upload must not become part of the
    graph, whose replays would read a pinned image that serves other plans by then.  Next to a capture of another stream a plan
    is made and run as ever."""
    import paper_2510_24051_b200 as pie
    from tests._gpu import GpuPool
    wl, steps = _loop_batches(6)
    with GpuPool(wl.num_pages, wl.P, wl.H_q, wl.H_kv, wl.D, wl.dtype) as gp:
        gp.install(wl)
        q, k, v = wl.q("cuda"), wl.k_new("cuda"), wl.v_new("cuda")
        args = [{n: b[n] for n in ("qo_indptr", "page_indptr", "page_indices", "last_page_len")} for b in steps]
        ref, out = [(torch.zeros_like(q), torch.zeros(wl.T, wl.H_q, device="cuda")) for _ in range(2)]
        for _ in range(2):                                # (the second time with a parked plan: nothing is allocated any more)
            plan = pie.pie_plan_forward(gp.ctx, **args[3])
            pie.pie_forward(gp.ctx, plan, q, k, v, *ref)
            torch.cuda.synchronize()
            pie.pie_plan_destroy(plan)
        free0 = pie.pie_num_free_kvpages(gp.ctx)
        x, y = torch.ones(64, device="cuda"), torch.zeros(64, device="cuda")
        s1, s2 = torch.cuda.Stream(), torch.cuda.Stream()
        busy = torch.zeros(1 << 26, device="cuda")
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s1):
            with pytest.raises(pie.PieError) as e:
                pie.pie_plan_forward(gp.ctx, **args[3])
            assert e.value.status == pie.PIE_ERR_CUDA
            with torch.cuda.stream(s2):
                for _ in range(20):
                    busy.add_(1.0)                    # the upload queues behind this
                plan = pie.pie_plan_forward(gp.ctx, **args[3])
                pie.pie_forward(gp.ctx, plan, q, k, v, *out)
                pie.pie_forward(gp.ctx, plan, q, k, v, *out)
                pie.pie_plan_destroy(plan)
            torch.add(x, 1.0, out=y)
        g.replay()
        torch.cuda.synchronize()
        assert (y == 2).all() and torch.equal(out[0], ref[0]) and torch.equal(out[1], ref[1])
        assert pie.pie_num_free_kvpages(gp.ctx) == free0
        for a in args:                                    # (and planning goes on)
            plan = pie.pie_plan_forward(gp.ctx, **a)
            pie.pie_forward(gp.ctx, plan, q, k, v, *out)
            pie.pie_plan_destroy(plan)
        torch.cuda.synchronize()
        assert pie.pie_get_last_device_status(gp.ctx) == 0
