"""Plans and keys destroyed after their context: what a Python program does
whenever a handle is collected late.  Host memory is churned in between, so
that whatever the context's object held is overwritten."""
import numpy as np
import pytest

from paper_2506_10399_gb300 import workloads as wl

pytestmark = pytest.mark.gpu
PRM = dict(log_n=10, q_bits=[60, 45, 45, 45], p_bits=[60], alpha=1, log_scale=45)


def test_plans_and_keys_outlive_their_context():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    fg = __graft_entry__.build()
    w = wl.make_workload(graph="er", V=16, deg=3.0, F=2, Fp=1, seed=3)
    handles = []
    for _ in range(8):
        ctx = fg.Context(**PRM)
        plan = fg.plan_build(ctx, w.row_ptr, w.col, w.val, w.W, wl.random_order(w.V, ctx.slots, 3), t=1)
        handles += [plan, fg.load_evk(ctx, fg.keygen(ctx, 1, [3])[1])]
        ctx.close()
        junk = [bytes([0xA5]) * n for n in range(64, 4096, 8)]
    for h in handles:
        h.close()
    del junk
    ctx = fg.Context(**PRM)
    one = np.zeros((4, ctx.n), np.uint64)
    one[:, 0] = 1
    a = wl.random_words(ctx.q, ctx.n, 1)
    assert np.array_equal(fg.poly_mul(ctx, a, one, 3), a)
    ctx.close()
