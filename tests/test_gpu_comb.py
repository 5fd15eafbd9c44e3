"""The combination on the tensor cores, word for word against the oracle:
column counts around its stages (16) and segments (128), output counts around
a block of 16, constants from one 8-bit digit to eight, and the words that make
the digit sums largest."""
import numpy as np
import pytest

from oracle import ckks, layer, planner
from paper_2506_10399_gb300 import workloads as wl

pytestmark = pytest.mark.gpu
PRM = dict(log_n=10, q_bits=[60, 45, 40, 45], p_bits=[60], alpha=1, log_scale=45)


@pytest.mark.parametrize("F,Fp,w,words", [
    (40, 1, 1.0, "random"), (63, 8, 2.0 ** -40, "random"), (128, 16, 1.0, "max"), (129, 16, 2.0 ** 17, "max"),
    (257, 17, 0.1, "random"), (33, 33, 2.0 ** 9, "zero"), (144, 16, 2.6e5, "random"), (400, 3, 0.03, "mixed")])
def test_combination_matches_the_oracle(F, Fp, w, words):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    fg = __graft_entry__.build()
    P = ckks.Params(PRM["log_n"], PRM["q_bits"], PRM["p_bits"], PRM["alpha"], PRM["log_scale"])
    ctx = fg.Context(**PRM)
    rng = np.random.default_rng(F)
    V = 30
    # every weight at the largest magnitude w, so that digit sums do not cancel by chance
    W = np.full((F, Fp), -w) if words == "max" else rng.uniform(-w, w, (F, Fp))
    nbr, wts = np.arange(V, dtype=np.int32)[:, None], rng.uniform(0.5, 1.0, (V, 1))
    perm = wl.random_order(V, P.slots, 1)
    op = planner.build_inter_plan(P, P.L, nbr, wts, V, W, perm)
    plan = fg.plan_build_inter(ctx, nbr, wts, W, perm)
    _, evk = fg.keygen(ctx, 1, [])
    keys = fg.load_evk(ctx, evk)
    pts = layer.encode_plan_masks(P, op)
    for i, pt in enumerate(pts):
        plan.set_plaintext(i, pt)
    q = np.array(P.q, np.uint64)[:, None]
    cts = []
    for f in range(F):
        c = np.stack([wl.random_words(P.q, P.n, 2 * f + p) for p in (0, 1)])
        if words == "max" or (words == "mixed" and f % 2):
            c[:] = q - np.uint64(1)
        elif words == "zero" or (words == "mixed" and f % 4 == 2):
            c[:] = 0
        cts.append(c)
    x = np.ascontiguousarray(np.stack(cts))
    want = layer.inter_ca_layer(P, op, cts, pts)
    for src in (x, torch.from_numpy(x.view(np.int64)).cuda()):
        out, _, _ = fg.gcn_layer_axw(ctx, keys, plan, src)
        out = out if isinstance(out, np.ndarray) else out.cpu().numpy().view(np.uint64)
        for j in range(Fp):
            assert np.array_equal(out[j], want[j])
    ctx.close()
