"""What a user of this library has the GPU do, as cases that can be timed.

Every case goes through the package's public calls on buffers the user
already holds: uniform residues as ciphertexts (an RLWE ciphertext is
computationally indistinguishable from them, and every kernel's work is
independent of the values), real rotation keys, and plans of synthetic
power-law graphs.  Outputs are the calls' whole outputs: 64-bit residues, so
they are compared word for word and no floating-point reference exists.

Parameter sets are the repository's own (workloads.CONFIGS, BATCH_PARAMS and
the tests' N = 2^13 set); drawn cases take other sizes of the same kinds.
"""
import math

import numpy as np
import torch

import paper_2506_10399_gb300 as fg
from paper_2506_10399_gb300 import workloads as wl


def _case(name, op, log_n, n45, bits, np_, alpha, **kw):
    c = dict(name=name, op=op, log_n=log_n, n_scale=n45, bits=bits, n_special=np_, alpha=alpha)
    c.update(kw)
    return c


def listed():
    return [
        # the smallest server call: one rotation on the toy parameters
        # (N = 2^12, 3 primes), where launches and latency are all there is
        _case("rotate_toy", "rotate", 12, 2, 40, 1, 1, level=2, k=5),
        # one plaintext-sized negacyclic product (N = 2^13, 8 primes)
        _case("poly_mul_n13", "poly_mul", 13, 7, 45, 3, 3, level=7),
        # a whole layer on the toy graph: 64 nodes, packed columns (t = 4)
        _case("layer_toy", "layer", 12, 2, 40, 1, 1, graph="er", V=64, deg=4.0, gamma=0.0, F=16, Fp=8, t=4,
              radix=11, min_out=0),
        # single rotations at the two large parameter sets' top levels
        _case("rotate_n15", "rotate", 15, 9, 40, 4, 4, level=9, k=3001),
        _case("rotate_n16", "rotate", 16, 19, 45, 4, 4, level=19, k=17),
        # the x^2 activation between two layers: 16 ciphertexts squared,
        # relinearised and rescaled where the first layer of the large set ends
        _case("square_n16", "square", 16, 19, 45, 4, 4, level=10, n=16),
        # transforms alone: the batch a 16-column lane has (N = 2^16), and an
        # odd count at N = 2^15, one direction each
        _case("ntt_fwd_n16", "ntt", 16, 19, 45, 4, 4, period=15, rows=32, inverse=False),
        _case("ntt_inv_n15", "ntt", 15, 9, 40, 4, 4, period=9, rows=37, inverse=True),
        # three uneven small queries in one batched call: seeded client
        # ciphertexts in page-locked memory, two streams, one CUDA graph
        _case("batch_seeded_n13", "batch", 13, 9, 45, 3, 3, V=260, F=50, Fp=16, queries=3),
        # one layer of the cora-like set (N = 2^15, 1433 feature columns)
        _case("layer_cora", "layer", 15, 9, 40, 4, 4, graph="chung_lu", V=2708, deg=3.9, gamma=2.5, F=1433, Fp=16,
              t=1, radix=0, min_out=0),
        # one query of the batched workload (N = 2^16, 14 primes): its mean size
        _case("layer_query", "layer", 16, 13, 45, 4, 4, graph="chung_lu", V=2250, deg=4.0, gamma=2.5, F=288, Fp=16,
              t=1, radix=0, min_out=0),
        # the first layer as Inter-CA at the large set (N = 2^16, 20 primes,
        # 500 columns): each node and two sampled neighbours
        _case("inter_pubmed", "inter", 16, 19, 45, 4, 4, V=19717, deg=4.5, gamma=2.5, F=500, Fp=16, copies=3),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    c = _drawn(rng)
    del c["name"]
    return c


def _drawn(rng):
    op = rng.choice(["rotate", "rotate", "poly_mul", "ntt", "ntt", "square", "layer", "layer", "inter", "batch"])
    log_n = rng.randint(12, 16)
    bits = rng.choice([40, 45])
    np_ = rng.randint(1, 4)
    nq = rng.randint(4, 19)
    alpha = rng.randint(1, np_)
    while -(-(nq + 1) // alpha) > 16:   # at most 16 key-switching digits
        alpha += 1
    np_ = max(np_, alpha)
    if op == "rotate":
        return _case("drawn", op, log_n, nq, bits, np_, alpha, level=rng.randint(1, nq),
                     k=rng.randint(1, 2 ** (log_n - 1) - 1))
    if op == "poly_mul":
        return _case("drawn", op, log_n, nq, bits, np_, alpha, level=rng.randint(1, nq))
    if op == "ntt":
        return _case("drawn", op, log_n, nq, bits, np_, alpha, period=rng.randint(1, nq + 1), rows=_log(rng, 1, 64),
                     inverse=rng.random() < 0.5)
    if op == "square":
        return _case("drawn", op, log_n, nq, bits, np_, alpha, level=rng.randint(1, min(nq, 12)), n=_log(rng, 1, 24))
    if op == "inter":
        log_n = rng.randint(13, 15)
        return _case("drawn", op, log_n, rng.randint(3, 12), bits, np_, alpha, V=_log(rng, 200, 2 ** (log_n - 1) - 1),
                     deg=4.0, gamma=2.5, F=_log(rng, 16, 500), Fp=rng.choice([3, 7, 8, 16]), copies=rng.randint(2, 5))
    if op == "batch":
        return _case("drawn", op, rng.randint(12, 13), 9, bits, 3, 3, V=_log(rng, 60, 400), F=_log(rng, 8, 64),
                     Fp=rng.choice([4, 8, 16]), queries=rng.randint(2, 5))
    log_n = rng.randint(13, 15)
    return _case("drawn", op, log_n, 9, bits, 4, 4, graph="chung_lu", V=_log(rng, 100, 2 ** (log_n - 3)), deg=4.0,
                 gamma=round(rng.uniform(2.1, 3.0), 3), F=_log(rng, 16, 1433), Fp=rng.choice([3, 7, 8, 16]), t=1,
                 radix=0, min_out=0)


def _params(case):
    return dict(log_n=case["log_n"], q_bits=[60] + [case["bits"]] * case["n_scale"], p_bits=[60] * case["n_special"],
                alpha=case["alpha"], log_scale=case["bits"])


def _residues(primes, lead, n, gen):
    """Uniform residues [*lead][len(primes)][n] on the GPU."""
    out = torch.empty(*lead, len(primes), n, dtype=torch.int64, device="cuda")
    for i, q in enumerate(primes):
        out[..., i, :] = torch.randint(0, q, (*lead, n), generator=gen, device="cuda", dtype=torch.int64)
    return out


def _graph(case, seed):
    return wl.make_workload(graph=case.get("graph", "chung_lu"), V=case["V"], deg=case.get("deg", 4.0),
                            gamma=case.get("gamma", 2.5), F=case["F"], Fp=case["Fp"], x="tfidf", w="glorot", seed=seed)


def prepare(case, seed):
    prm = _params(case)
    ctx = fg.Context(**prm)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    op, n = case["op"], ctx.n
    st = dict(op=op, ctx=ctx, case=case)
    if op == "rotate":
        _, evk = fg.keygen(ctx, seed, [case["k"]])
        st.update(keys=fg.load_evk(ctx, evk), x=_residues(ctx.q[:case["level"] + 1], (2,), n, gen))
    elif op == "poly_mul":
        q = ctx.q[:case["level"] + 1]
        st.update(a=_residues(q, (), n, gen), b=_residues(q, (), n, gen))
    elif op == "ntt":
        pid = list(range(case["period"]))
        pr = (ctx.q + ctx.p)[:case["period"]]
        st.update(pid=pid, x=_residues(pr, (case["rows"],), n, gen).reshape(-1, n))
    elif op == "square":
        _, evk = fg.keygen(ctx, seed, [], relin=True)
        st.update(keys=fg.load_evk(ctx, evk), x=_residues(ctx.q[:case["level"] + 1], (case["n"], 2), n, gen))
    elif op == "layer":
        w = _graph(case, 0)   # one graph; the client's features and keys are new
        perm = wl.random_order(w.V, ctx.slots // case["t"], 2025)
        plan = fg.plan_build(ctx, w.row_ptr, w.col, w.val, w.W, perm, t=case["t"], radix_bits=case["radix"],
                             min_out_level=case["min_out"])
        _, evk = fg.keygen(ctx, seed, plan.rotation_amounts())
        n_in = plan.info()["n_in"]
        st.update(keys=fg.load_evk(ctx, evk), plan=plan, x=_residues(ctx.q, (n_in, 2), n, gen))
    elif op == "inter":
        w = _graph(case, 0)
        nbr, wts = wl.sample_neighbors(w, case["copies"] - 1, 0)
        perm = wl.random_order(w.V, ctx.slots, 2025)
        plan = fg.plan_build_inter(ctx, nbr, wts, w.W, perm)
        _, evk = fg.keygen(ctx, seed, [])
        st.update(keys=fg.load_evk(ctx, evk), plan=plan, x=_residues(ctx.q, (plan.info()["n_in"], 2), n, gen))
    else:   # batch
        plans, ins, outs, seeds, amounts = [], [], [], [], set()
        for i in range(case["queries"]):
            c = dict(case, V=max(20, case["V"] - 41 * i), F=max(4, case["F"] - 7 * i))
            w = _graph(c, i)
            plan = fg.plan_build(ctx, w.row_ptr, w.col, w.val, w.W, wl.random_order(w.V, ctx.slots, 2025 + i), t=1)
            info = plan.info()
            amounts |= set(plan.rotation_amounts())
            plans.append(plan)
            ins.append(_residues(ctx.q, (info["n_in"],), n, gen).cpu().pin_memory())
            outs.append(torch.empty(info["n_out"], 2, info["out_level"] + 1, n, dtype=torch.int64, device="cuda"))
            seeds.append(1000 * seed + i)
        _, evk = fg.keygen(ctx, seed, sorted(amounts))
        st.update(keys=fg.load_evk(ctx, evk), plans=plans, ins=ins, outs=outs, seeds=seeds)
    torch.cuda.synchronize()
    return st


def run(st):
    op, ctx, case = st["op"], st["ctx"], st["case"]
    if op == "rotate":
        return fg.rotate(ctx, st["keys"], st["x"], case["level"], case["k"])
    if op == "poly_mul":
        return fg.poly_mul(ctx, st["a"], st["b"], case["level"])
    if op == "ntt":
        return fg.ntt(ctx, st["x"], st["pid"], inverse=case["inverse"])
    if op == "square":
        return fg.mul_relin_rescale(ctx, st["keys"], st["x"], st["x"], case["level"])
    if op in ("layer", "inter"):
        out, level, _ = fg.gcn_layer_axw(ctx, st["keys"], st["plan"], st["x"])
        return out, level
    levels, _ = fg.gcn_layer_batch(ctx, st["keys"], st["plans"], st["ins"], st["outs"], streams=2, graph=True,
                                   seeds=st["seeds"])
    return st["outs"], levels


def exact(case, seed):
    return None   # every output is a tensor of residues (whole numbers): equal or wrong


# ---------------------------------------------------------------------- work
# bytes: every input, key, mask and output word once.  flops: integer
# operations on residues, two per multiply-accumulate, three per butterfly.
def _ntt(limbs, n):
    return 3.0 * limbs * (n / 2) * math.log2(n)


def _switch(n, level, np_, alpha, ncol, rots):
    """ModUp of ncol ciphertexts and the inner products of `rots` rotations."""
    nl = level + 1
    E, beta = nl + np_, -(-nl // alpha)
    up = ncol * (_ntt(nl, n) + _ntt(beta * E - nl, n) + 2.0 * n * alpha * (beta * E - nl))
    return up + rots * ncol * 4.0 * beta * E * n


def _down(n, level, np_, ncol):
    nl = level + 1
    return 2 * ncol * (_ntt(np_, n) + _ntt(nl, n) + 2.0 * n * nl * (np_ + 1))


def _plan_groups(case, w, perm, t, radix, min_out):
    """Per group (level, rotations by source lane, terms, outputs, amounts), t-packing rotations, masks, out level."""
    r = fg.plan_dry_run(_params(case), w.row_ptr, w.col, w.val, w.W, perm, t=t, radix_bits=radix, min_out_level=min_out)
    V, F, Fp, out_level, ng = (int(r[i]) for i in (4, 5, 6, 8, 11))
    o = 13 + V
    crots = []
    if t == 1:
        o += F * Fp
    else:
        o += -(-F // t) * Fp
        crots = [int(v) for v in r[o + 1:o + 1 + int(r[o])]]
        o += 1 + len(crots)
    groups = []
    for _ in range(ng):
        level, n_out, n_rot = int(r[o + 2]), int(r[o + 4]), int(r[o + 5])
        rots = r[o + 6:o + 6 + 2 * n_rot].reshape(-1, 2)
        o += 6 + 2 * n_rot
        n_term = int(r[o])
        groups.append((level, len(set(rots[:, 0])), n_rot, n_term, n_out + 1, [int(k) for k in rots[:, 1]]))
        o += 1 + 4 * n_term
    return groups, crots, out_level


def _layer_work(case, w, slots, t, radix, min_out):
    n, np_, alpha, Fp = 2 ** case["log_n"], case["n_special"], case["alpha"], case["Fp"]
    l0 = case["n_scale"]
    perm = wl.random_order(w.V, slots // t, 2025)
    groups, crots, out_level = _plan_groups(case, w, perm, t, radix, min_out)
    F = case["F"]
    n_in = -(-F // t)
    words = 2.0 * n_in * (l0 + 1) * n + 2.0 * Fp * (out_level + 1) * n
    ops = 4.0 * n_in * Fp * (l0 + 1) * n + _ntt(2 * Fp * l0, n)
    keys = {}   # amount -> the highest level it is used at
    for k in crots:
        keys[k % slots] = l0 - 1
        ops += _switch(n, l0 - 1, np_, alpha, Fp, 1) + _down(n, l0 - 1, np_, Fp)
    for level, lanes, rots, terms, outs, ks in groups:
        E = level + 1 + np_
        ops += lanes * _switch(n, level, np_, alpha, Fp, 0) + rots * Fp * 4.0 * -(-(level + 1) // alpha) * E * n
        ops += 4.0 * terms * Fp * E * n + outs * _down(n, level, np_, Fp)
        words += float(terms) * E * n
        for k in ks:
            keys[k % slots] = max(level, keys.get(k % slots, -1))
    for level in keys.values():
        words += 2.0 * -(-(level + 1) // alpha) * (level + 1 + np_) * n
    return words, ops


def work(case):
    n, op = 2 ** case["log_n"], case["op"]
    np_, alpha = case["n_special"], case["alpha"]
    if op == "rotate":
        nl = case["level"] + 1
        E, beta = nl + np_, -(-nl // alpha)
        words = (4.0 * nl + 2.0 * beta * E) * n
        ops = _ntt(4 * nl, n) + _switch(n, case["level"], np_, alpha, 1, 1) + _down(n, case["level"], np_, 1)
    elif op == "poly_mul":
        nl = case["level"] + 1
        words, ops = 3.0 * nl * n, _ntt(3 * nl, n) + 2.0 * nl * n
    elif op == "ntt":
        limbs = case["period"] * case["rows"]
        words, ops = 2.0 * limbs * n, _ntt(limbs, n)
    elif op == "square":
        nl, c = case["level"] + 1, case["n"]
        E, beta = nl + np_, -(-nl // alpha)
        words = (2.0 * c * nl + 2.0 * beta * E + 2.0 * c * (nl - 1)) * n
        ops = _ntt(2 * c * nl + 2 * c * (nl - 1), n) + 6.0 * c * nl * n + _switch(n, case["level"], np_, alpha, c, 1) \
            + _down(n, case["level"], np_, c)
    elif op == "layer":
        words, ops = _layer_work(case, _graph(case, 0), n // 2, case["t"], case["radix"], case["min_out"])
    elif op == "inter":
        nl, Fp, c = case["n_scale"] + 1, case["Fp"], case["copies"]
        words = (2.0 * c * case["F"] * nl + c * (nl - 1) + 2.0 * Fp * (nl - 2)) * n
        ops = 4.0 * c * case["F"] * Fp * nl * n + c * (_ntt(2 * Fp * (nl - 1), n) + 4.0 * Fp * (nl - 1) * n) \
            + _ntt(2 * Fp * (2 * nl - 3), n)
    else:   # batch: seeded inputs (c0 only)
        words = ops = 0.0
        for i in range(case["queries"]):
            c = dict(case, V=max(20, case["V"] - 41 * i), F=max(4, case["F"] - 7 * i))
            a, b = _layer_work(c, _graph(c, i), n // 2, 1, 0, 0)
            words += a - float(c["F"]) * (case["n_scale"] + 1) * n
            ops += b
    return dict(bytes=8.0 * words, flops=float(ops))
