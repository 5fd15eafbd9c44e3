"""Two contexts on two threads and streams, whose layers launch the same group
MAC kernels with different amounts of shared memory: every call gives the
words it gives alone."""
import threading

import pytest

from paper_2506_10399_gb300 import workloads as wl

pytestmark = pytest.mark.gpu
PRM = dict(log_n=10, q_bits=[60] + [45] * 7, p_bits=[60], alpha=1, log_scale=45)


@pytest.mark.parametrize("V,radix,widths", [(16, 5, (1, 8)), (200, 2, (1, 7))])
def test_layers_of_two_threads(V, radix, widths):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    fg = __graft_entry__.build()
    work = []
    for Fp in widths:
        stream = torch.cuda.Stream()
        ctx = fg.Context(**PRM, stream=stream.cuda_stream)
        w = wl.make_workload(graph="er", V=V, deg=3.0, F=2, Fp=Fp, seed=3)
        plan = fg.plan_build(ctx, w.row_ptr, w.col, w.val, w.W, wl.random_order(w.V, ctx.slots, 3), t=1,
                             radix_bits=radix)
        keys = fg.load_evk(ctx, fg.keygen(ctx, 1, plan.rotation_amounts())[1])
        x = torch.stack([torch.randint(0, q, (2, 2, ctx.n), device="cuda") for q in ctx.q], 2).contiguous()
        torch.cuda.synchronize()
        n0 = ctx.launch_count()
        want = fg.gcn_layer_axw(ctx, keys, plan, x)[0].clone()
        launches = ctx.launch_count() - n0
        torch.cuda.synchronize()
        work.append((ctx, keys, plan, x, want, stream, launches))
    failures = []

    def loop(ctx, keys, plan, x, want, stream, launches):
        out = torch.empty_like(want)
        try:
            n0 = ctx.launch_count()
            for _ in range(2000):
                fg.gcn_layer_axw(ctx, keys, plan, x, out=out)
            if ctx.launch_count() - n0 != 2000 * launches:
                failures.append("launches counted on another context")
            with torch.cuda.stream(stream):
                if not torch.equal(out, want):
                    failures.append("words differ")
        except fg.FicgcnError as e:
            failures.append(str(e))

    threads = [threading.Thread(target=loop, args=a) for a in work]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for ctx, keys, plan, *_ in work:
        for h in (plan, keys, ctx):
            h.close()
    assert not failures, failures
