"""How many passes a transform at N = 2^12 or 2^13 takes: at 2^13 by the limbs
it works on, not by those it leaves alone, and by how full the last wave of one
limb an SM is.  A product of eight pairs (12 limbs a polynomial, of
which ModDown transforms four) by its launches, and word for word the products
one at a time, whose transforms take the other form."""
import pytest

pytestmark = pytest.mark.gpu
NQ, NP, ALPHA, PAIRS = 9, 3, 3, 8


def passes(log_n, limbs):
    if log_n == 12:
        return 1 if limbs >= 80 else 2
    waves = -(-limbs // 152)
    return 1 if limbs >= 150 * waves - 50 else 2


def launches_of_one_product():
    """Launches of fg_mul_relin_rescale on PAIRS pairs at the top level."""
    nl, E, beta = NQ, NQ + NP, NQ // ALPHA
    transforms = [2 * PAIRS * nl] * 2                       # both operands
    transforms += [PAIRS * nl]                              # ModUp: c1 back to coefficients
    transforms += [PAIRS * (beta * E - nl)]                 # ModUp: every digit's other limbs
    transforms += [2 * PAIRS * (NP + 1)]                    # ModDown: the special limbs and the dropped one
    transforms += [2 * PAIRS * (nl - 1)] * 2                # ModDown's conversion; the result
    others = 5                                              # tensor, ModUp, inner product, P d1, ModDown conversion
    return others + sum(passes(13, t) for t in transforms)


def test_limbs_left_alone_do_not_count():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    fg = __graft_entry__.build()
    ctx = fg.Context(log_n=13, q_bits=[60] + [45] * (NQ - 1), p_bits=[60] * NP, alpha=ALPHA, log_scale=45)
    keys = fg.load_evk(ctx, fg.keygen(ctx, 1, [], relin=True)[1])
    a, b = (torch.stack([torch.randint(0, q, (PAIRS, 2, ctx.n), device="cuda") for q in ctx.q], 2).contiguous()
            for _ in range(2))
    n0 = ctx.launch_count()
    got = fg.mul_relin_rescale(ctx, keys, a, b, NQ - 1)
    assert ctx.launch_count() - n0 == launches_of_one_product()
    for c in range(PAIRS):
        one = fg.mul_relin_rescale(ctx, keys, a[c].contiguous(), b[c].contiguous(), NQ - 1)
        assert torch.equal(got[c], one)
    keys.close()
    ctx.close()


@pytest.mark.parametrize("log_n,limbs", [(12, 79), (12, 80), (13, 99), (13, 100), (13, 152), (13, 153), (13, 249),
                                         (13, 250), (13, 305), (13, 400)])
def test_both_sides_of_every_line(log_n, limbs):
    """The batch's words against each limb's own transform (two passes)."""
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    fg = __graft_entry__.build()
    ctx = fg.Context(log_n=log_n, q_bits=[60, 45], p_bits=[60], alpha=1, log_scale=45)
    for prime in (0, 1):
        x = torch.randint(0, ctx.q[prime], (limbs, ctx.n), device="cuda")
        n0 = ctx.launch_count()
        y = fg.ntt(ctx, x.clone(), [prime])
        assert ctx.launch_count() - n0 == passes(log_n, limbs)
        for c in (0, limbs // 2, limbs - 1):
            assert torch.equal(fg.ntt(ctx, x[c:c + 1].clone(), [prime])[0], y[c])
        assert torch.equal(fg.ntt(ctx, y.clone(), [prime], inverse=True), x)
    ctx.close()
