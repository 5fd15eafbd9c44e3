"""The key switch's and the base conversions' sums where their forms change:
5 to 9 digits (30-bit halves in one step, in 128 bits, as 128-bit sums), 6 to 8
primes a digit and 6 or 7 special primes, primes just below and above 2^46, on
random residues and on the largest ones; word for word against the oracle."""
import numpy as np
import pytest

from oracle import ckks

pytestmark = pytest.mark.gpu

SETS = [
    (5, 1, 1, 45), (6, 1, 1, 46), (7, 1, 1, 45), (8, 1, 1, 47), (9, 1, 1, 60),   # digits
    (7, 6, 6, 45), (8, 7, 7, 60), (9, 8, 7, 46), (4, 2, 2, 60), (6, 5, 5, 45),   # primes a digit, special primes
]


@pytest.mark.parametrize("nq,alpha,np_,bits", SETS)
@pytest.mark.parametrize("words", ["random", "max"])
def test_rotation_and_product_match_the_oracle(nq, alpha, np_, bits, words):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    fg = __graft_entry__.build()
    prm = dict(log_n=10, q_bits=[60] + [bits] * (nq - 1), p_bits=[60] * np_, alpha=alpha, log_scale=40)
    ctx = fg.Context(**prm)
    P = ckks.Params(prm["log_n"], prm["q_bits"], prm["p_bits"], alpha, 40)
    seed, level = 11, nq - 1
    _, evk = fg.keygen(ctx, seed, [3], relin=True)
    keys = fg.load_evk(ctx, evk)
    s = ckks.keygen_secret(P, seed)
    rng = np.random.default_rng(nq)
    q = np.array(P.q, np.uint64)[:, None]

    def ct():
        if words == "max":
            return np.broadcast_to(q - np.uint64(1), (2, nq, P.n)).copy()
        return np.stack([np.stack([rng.integers(0, v, P.n, dtype=np.uint64) for v in P.q]) for _ in range(2)])

    a, b = ct(), ct()
    rot = ckks.keygen_rotation(P, seed, s, 3)
    np.testing.assert_array_equal(fg.rotate(ctx, keys, a, level, 3), ckks.rotate(P, a, 3, rot))
    want = ckks.mul_relin_rescale(P, a, b, ckks.keygen_relin(P, seed, s))
    np.testing.assert_array_equal(fg.mul_relin_rescale(ctx, keys, a, b, level), want)
    ctx.close()
