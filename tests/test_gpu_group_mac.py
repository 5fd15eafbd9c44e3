"""The group's masked sums at the shapes where their two forms and tiles
change: one to seven outputs (up to six streamed, more as tiles), column
counts that leave a ragged last block, source counts around a stage, word for
word against the oracle's layer on shared inputs."""
import numpy as np
import pytest

from oracle import ckks, layer, planner
from paper_2506_10399_gb300 import workloads as wl

pytestmark = pytest.mark.gpu
# one 60-bit and 45-bit limbs, special primes; N = 2^10 keeps the oracle quick
PRM = dict(log_n=10, q_bits=[60] + [45] * 5, p_bits=[60] * 2, alpha=2, log_scale=45)


@pytest.mark.parametrize("V,deg,radix,Fp,seed", [
    (16, 2.0, 5, 1, 1), (40, 3.0, 5, 9, 2), (100, 4.0, 3, 3, 3), (200, 5.0, 3, 2, 4), (300, 6.0, 3, 1, 5)])
def test_group_outputs_match_the_oracle(V, deg, radix, Fp, seed):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    fg = __graft_entry__.build()
    P = ckks.Params(PRM["log_n"], PRM["q_bits"], PRM["p_bits"], PRM["alpha"], PRM["log_scale"])
    ctx = fg.Context(**PRM)
    w = wl.make_workload(graph="chung_lu", V=V, deg=deg, gamma=2.5, F=2, Fp=Fp, x="uniform", w="normal16", seed=seed)
    perm = wl.random_order(w.V, P.slots, seed)
    op = planner.build_plan(P, P.L, w.row_ptr, w.col, w.val, w.V, w.W, perm, 1, radix)
    plan = fg.plan_build(ctx, w.row_ptr, w.col, w.val, w.W, perm, t=1, radix_bits=radix)
    sk, evk = fg.keygen(ctx, seed, plan.rotation_amounts())
    keys = fg.load_evk(ctx, evk)
    s = ckks.keygen_secret(P, seed)
    okeys = {k: ckks.keygen_rotation(P, seed, s, k) for k in op.rotation_amounts()}
    pts = layer.encode_plan_masks(P, op)
    for i, pt in enumerate(pts):
        plan.set_plaintext(i, pt)
    cts = [np.stack([wl.random_words(P.q, P.n, 10 * seed + 2 * f + p) for p in (0, 1)]) for f in range(2)]
    out, lvl, _ = fg.gcn_layer_axw(ctx, keys, plan, np.ascontiguousarray(np.stack(cts)))
    ref = layer.layer_axw(P, op, cts, okeys, pts)
    for j in range(Fp):
        assert np.array_equal(out[j], ref[j])
    ctx.close()
