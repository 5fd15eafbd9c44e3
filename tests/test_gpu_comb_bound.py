"""The tensor-core combination where its digit sums come closest to the 2^24
that f32 accumulation holds exactly: 128 columns of one sign, words whose
8-bit digits lie next to -128 (or +127) and constants of six random digits
next to -128 (or +127) above a low digit of -128 -- 49 significant bits, so a
double weight gives each constant exactly.  The low bits of every sum vary, so
that a sum rounded anywhere on the way differs from the oracle's words."""
import numpy as np
import pytest

from oracle import ckks, layer, planner
from paper_2506_10399_gb300 import workloads as wl

pytestmark = pytest.mark.gpu
PRM = dict(log_n=10, q_bits=[60, 45, 40, 45], p_bits=[60], alpha=1, log_scale=45)
SEG = 128   # columns an accumulator sums before it is read


def constants(rng, F, Fp, near, ql):
    """[F][Fp] integers and the double weights that round(w ql) maps onto them."""
    c = np.full((F, Fp), -128, np.int64)
    for b in range(1, 7):
        c += (-128 + rng.integers(0, 4, (F, Fp)) if near < 0 else 127 - rng.integers(0, 4, (F, Fp))) << (8 * b)
    w = c / float(ql)
    for _ in range(8):   # neighbouring doubles where the quotient's rounding missed
        d = np.round(w * float(ql)).astype(np.int64) - c
        w = np.where(d == 0, w, np.nextafter(w, np.where(d > 0, -np.inf, np.inf)))
    assert (np.round(w * float(ql)).astype(np.int64) == c).all()
    return c, w


def words(rng, q, n, near):
    """Words below q of which every byte but the topmost is within 3 of 0 or 255."""
    nb = (q.bit_length() + 7) // 8
    top = 0 if near < 0 else (q >> (8 * (nb - 1))) - 1
    x = np.full(n, max(top, 0) << (8 * (nb - 1)), np.uint64)
    for a in range(nb - 1):
        x += (rng.integers(0, 4, n) if near < 0 else 255 - rng.integers(0, 4, n)).astype(np.uint64) << np.uint64(8 * a)
    assert int(x.max()) < q
    return x


def largest_sum(x, c):
    """max |D_e| over segments: D_e = sum over a + b = e of digit a of the words times digit b of the constants."""
    dx = [((x >> np.uint64(8 * a)) & np.uint64(255)).astype(np.int64) - 128 for a in range(8)]
    dc, r = [], c.copy()
    for _ in range(7):
        d = r.astype(np.int8).astype(np.int64)
        dc.append(d)
        r = (r - d) >> 8
    assert (r == 0).all()
    best = 0
    for f0 in range(0, x.shape[0], SEG):
        for e in range(14):
            s = sum(dx[a][f0:f0 + SEG].T @ dc[e - a][f0:f0 + SEG] for a in range(8) if 0 <= e - a < 7)
            best = max(best, int(np.abs(s).max()))
    return best


@pytest.mark.parametrize("F,Fp,near_x,near_c", [(128, 16, -1, -1), (256, 16, 1, -1), (128, 3, -1, 1), (200, 17, 1, 1)])
def test_sums_next_to_the_bound_are_exact(F, Fp, near_x, near_c):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    fg = __graft_entry__.build()
    P = ckks.Params(PRM["log_n"], PRM["q_bits"], PRM["p_bits"], PRM["alpha"], PRM["log_scale"])
    ctx = fg.Context(**PRM)
    rng = np.random.default_rng(F + Fp)
    V = 30
    c, W = constants(rng, F, Fp, near_c, P.q[P.L])
    nbr, wts = np.arange(V, dtype=np.int32)[:, None], rng.uniform(0.5, 1.0, (V, 1))
    perm = wl.random_order(V, P.slots, 1)
    op = planner.build_inter_plan(P, P.L, nbr, wts, V, W, perm)
    assert (np.array(op.comb_consts, np.int64) == c).all()
    plan = fg.plan_build_inter(ctx, nbr, wts, W, perm)
    _, evk = fg.keygen(ctx, 1, [])
    keys = fg.load_evk(ctx, evk)
    pts = layer.encode_plan_masks(P, op)
    for i, pt in enumerate(pts):
        plan.set_plaintext(i, pt)
    x = np.stack([np.stack([np.stack([words(rng, q, P.n, near_x) for q in P.q]) for _ in range(2)]) for _ in range(F)])
    reached = largest_sum(x[:, 0, 0], c)   # the 60-bit limb: eight digits a word
    assert (0.70 if near_c > 0 else 0.84) * 2 ** 24 < reached <= 2 ** 24
    want = layer.inter_ca_layer(P, op, list(x), pts)
    out, _, _ = fg.gcn_layer_axw(ctx, keys, plan, torch.from_numpy(x.view(np.int64)).cuda())
    out = out.cpu().numpy().view(np.uint64)
    for j in range(Fp):
        assert np.array_equal(out[j], want[j])
    ctx.close()
