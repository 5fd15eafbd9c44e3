"""bench.py's products that the kernels perform: the key switch takes three per
product of words on limbs below 2^46 and four above (counted from the oracle's
plan), and the combination leaves the integer pipe exactly where the library's
rule says.  Host only."""
import os
import re
import sys

from oracle import ckks, planner
from paper_2506_10399_gb300 import workloads as wl

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)
PARAMS = dict(log_n=12, q_bits=[60] + [45] * 4 + [47], p_bits=[60] * 2, alpha=2, log_scale=45)


class _Fg:
    @staticmethod
    def int_mul_peak(ctx, op):
        return 1e13


def test_key_switch_products_performed():
    import __graft_entry__
    fg = __graft_entry__.build()
    import bench
    P = ckks.Params(PARAMS["log_n"], PARAMS["q_bits"], PARAMS["p_bits"], PARAMS["alpha"], PARAMS["log_scale"])
    w = wl.make_workload(graph="chung_lu", V=300, deg=4.0, gamma=2.5, F=20, Fp=3, x="tfidf", w="glorot", seed=5)
    perm = wl.random_order(w.V, P.slots, 6)
    rec = fg.plan_dry_run(PARAMS, w.row_ptr, w.col, w.val, w.W, perm, t=1, radix_bits=3)
    op = planner.build_plan(P, P.L, w.row_ptr, w.col, w.val, w.V, w.W, perm, 1, 3)
    want = 0
    for g in op.groups:
        limbs = list(P.q[:g.level + 1]) + list(P.p)
        digits = -(-(g.level + 1) // PARAMS["alpha"])
        want += sum(len(g.rotations) * 3 * P.n * 2 * digits * (3 if q < 1 << 46 else 4) for q in limbs)
    ctx = type("Ctx", (), {"n": P.n, "np": len(P.p), "q": list(P.q)})
    plan = type("Plan", (), {"describe": lambda self: rec})()
    out = bench.alu_roofline(_Fg(), ctx, plan, {"ks_ip": {"ms": 2.0}}, 20, 3, PARAMS["alpha"])["kernels"]["ks_ip"]
    assert out["performed"] == want < out["mults"]
    assert out["achieved"] == want / 2e-3
    assert out["frac"] == round(out["achieved"] / 1e13, 4)


def test_combination_rule_is_the_library_s():
    import bench
    with open(os.path.join(ROOT, "paper_2506_10399_gb300", "csrc", "fg_internal.h")) as f:
        least = int(re.search(r"kCombMmaMin = (\d+)", f.read()).group(1))
    for F, Fp in [(least - 1, 8), (least, 8), (least // 2 - 1, 16), (least // 2, 16), (least, 1), (least - 1, 24), (500, 16)]:
        assert bench.comb_on_tensor_cores(F, Fp, 1) == (F * ((Fp + 7) // 8) >= least * ((Fp + 15) // 16))
        assert not bench.comb_on_tensor_cores(F, Fp, 2)
