"""The tensor-core combination's bounded waits made to run out: the kernel
ends, the call returns FG_ETIMEOUT, and the same context then gives the words
it gave before.  Column counts below, at and above the stages that are under
way at once, so that a role gives up while another has finished."""
from types import SimpleNamespace

import numpy as np
import pytest

from paper_2506_10399_gb300 import workloads as wl

pytestmark = pytest.mark.gpu
PRM = dict(log_n=10, q_bits=[60, 45, 40, 45], p_bits=[60], alpha=1, log_scale=45)
EKEY, ETIMEOUT = -3, -6


def setup(F, Fp=16):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    fg = __graft_entry__.build()
    from paper_2506_10399_gb300 import _native
    ctx = fg.Context(**PRM)
    rng = np.random.default_rng(F)
    V = 30
    nbr, wts = np.arange(V, dtype=np.int32)[:, None], rng.uniform(0.5, 1.0, (V, 1))
    plan = fg.plan_build_inter(ctx, nbr, wts, rng.uniform(-1, 1, (F, Fp)), wl.random_order(V, ctx.slots, 1))
    keys = fg.load_evk(ctx, fg.keygen(ctx, 1, [])[1])
    x = torch.stack([torch.randint(0, q, (F, 2, ctx.n), device="cuda") for q in ctx.q], 2).contiguous()

    def limit(tries):
        assert _native.lib.fg_ctx_set_wait_tries(ctx._h, tries) == 0

    def layer():
        return fg.gcn_layer_axw(ctx, keys, plan, x)[0]

    def close():
        for h in (plan, keys, ctx):
            h.close()

    return SimpleNamespace(torch=torch, fg=fg, ctx=ctx, keys=keys, plan=plan, x=x, limit=limit, layer=layer, close=close)


@pytest.mark.parametrize("F", [40, 96, 97, 300])
def test_waits_that_give_up_at_once_end_in_a_timeout(F):
    v = setup(F)
    want = v.layer().clone()
    for _ in range(2):
        v.limit(0)
        with pytest.raises(v.fg.FicgcnError) as e:
            v.layer()
        assert e.value.code == ETIMEOUT
        v.limit(1 << 18)
        assert v.torch.equal(v.layer(), want)
    v.close()


@pytest.mark.parametrize("F,Fp", [(96, 16), (300, 48), (1000, 16)])
@pytest.mark.parametrize("tries", [1, 2, 4, 16])
def test_waits_that_may_give_up_midway_end_in_a_timeout_or_in_the_words(F, Fp, tries):
    """A limit of a few polls runs out in some warps and lanes and not in others."""
    v = setup(F, Fp)
    want = v.layer().clone()
    v.limit(tries)
    for _ in range(3):
        try:
            assert v.torch.equal(v.layer(), want)
        except v.fg.FicgcnError as e:
            assert e.code == ETIMEOUT
    v.limit(1 << 18)
    assert v.torch.equal(v.layer(), want)
    v.close()


def test_a_call_that_fails_otherwise_leaves_no_timeout_behind():
    """A batch whose first query's waits run out and whose second has no
    rotation key: the call reports the key, and the next call its words."""
    v = setup(96)
    want = v.layer().clone()
    w = wl.make_workload(graph="er", V=16, deg=3.0, F=2, Fp=1, seed=3)
    rotating = v.fg.plan_build(v.ctx, w.row_ptr, w.col, w.val, w.W, wl.random_order(w.V, v.ctx.slots, 3), t=1)
    out = v.torch.empty(1, 2, rotating.info()["out_level"] + 1, v.ctx.n, dtype=v.torch.int64, device="cuda")
    v.limit(0)
    with pytest.raises(v.fg.FicgcnError) as e:
        v.fg.gcn_layer_batch(v.ctx, v.keys, [v.plan, rotating], [v.x, v.x[:2].contiguous()],
                             [v.torch.empty_like(want), out], streams=1, graph=False)
    assert e.value.code == EKEY
    v.limit(1 << 18)
    assert v.torch.equal(v.layer(), want)
    rotating.close()
    v.close()
