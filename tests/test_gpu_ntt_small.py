"""Transforms at N = 2^10 .. 2^15: every ring degree, primes below and above
2^47 (lazy and reduced butterflies), one limb, the two sides of the batch sizes
where N = 2^12 and 2^13 change from two passes to one, limbs left alone in between;
forward then inverse, and products against the oracle's negacyclic product."""
import numpy as np
import pytest

from oracle import _ref, ckks
from paper_2506_10399_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("log_n", range(10, 16))
@pytest.mark.parametrize("rows", [1, 19, 20, 24, 25, 40])
def test_round_trip_and_product(log_n, rows):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    fg = __graft_entry__.build()
    prm = dict(log_n=log_n, q_bits=[60, 45, 40, 50], p_bits=[60], alpha=1, log_scale=40)
    ctx = fg.Context(**prm)
    P = ckks.Params(log_n, prm["q_bits"], prm["p_bits"], 1, 40)
    q = np.array(P.q, np.uint64)[:, None]
    a = np.stack([wl.random_words(P.q, ctx.n, r) for r in range(rows)])
    a[0] = q - np.uint64(1)
    x = torch.from_numpy(a.view(np.int64)).cuda().reshape(-1, ctx.n)
    y = fg.ntt(ctx, x.clone(), [0, 1, 2, 3])
    assert not bool((y == x).all())
    back = fg.ntt(ctx, y.clone(), [0, 1, 2, 3], inverse=True)
    assert bool((back == x).all())
    # one limb batch (row 0, the largest residues) as a product with row rows - 1
    b = a[rows - 1]
    got = fg.poly_mul(ctx, np.ascontiguousarray(a[0]), np.ascontiguousarray(b), 3)
    for i, p in enumerate(P.q):
        np.testing.assert_array_equal(got[i], _ref.negacyclic_mul(a[0, i], b[i], p, P.psi(p)))
    # the batch transform is the single transform of every row
    for r in (0, rows - 1):
        one = fg.ntt(ctx, torch.from_numpy(a[r].view(np.int64)).cuda(), [0, 1, 2, 3])
        assert bool((one == y.reshape(rows, 4, ctx.n)[r]).all())
    ctx.close()
