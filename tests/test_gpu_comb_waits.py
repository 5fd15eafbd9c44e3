"""The tensor-core combination's bounded waits made to run out: the kernel
ends, the call returns FG_ETIMEOUT, and the same context then gives the words
it gave before.  Column counts below, at and above the stages that are under
way at once, so that a role gives up while another has finished."""
import numpy as np
import pytest

from paper_2506_10399_gb300 import workloads as wl

pytestmark = pytest.mark.gpu
PRM = dict(log_n=10, q_bits=[60, 45, 40, 45], p_bits=[60], alpha=1, log_scale=45)
ETIMEOUT = -6


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

    return torch, fg, limit, layer, close


@pytest.mark.parametrize("F", [40, 96, 97, 300])
def test_waits_that_give_up_at_once_end_in_a_timeout(F):
    torch, fg, limit, layer, close = setup(F)
    want = layer().clone()
    for _ in range(2):
        limit(0)
        with pytest.raises(fg.FicgcnError) as e:
            layer()
        assert e.value.code == ETIMEOUT
        limit(1 << 18)
        assert torch.equal(layer(), want)
    close()


@pytest.mark.parametrize("F,Fp", [(96, 16), (300, 48), (1000, 16)])
@pytest.mark.parametrize("tries", [1, 2, 4, 16])
def test_waits_that_may_give_up_midway_end_in_a_timeout_or_in_the_words(F, Fp, tries):
    """A limit of a few polls runs out in some warps and lanes and not in others."""
    torch, fg, limit, layer, close = setup(F, Fp)
    want = layer().clone()
    limit(tries)
    for _ in range(3):
        try:
            assert torch.equal(layer(), want)
        except fg.FicgcnError as e:
            assert e.code == ETIMEOUT
    limit(1 << 18)
    assert torch.equal(layer(), want)
    close()
