"""Forward and inverse transforms at the ends of the NTT's range analysis: every
ring size, the smallest and largest primes, and the primes farthest below their
power of two (the last of a long chain), on random and extreme residues, word
for word against the oracle's stage-by-stage transform.
"""
import numpy as np
import pytest

import oracle


@pytest.fixture(scope="module")
def g():
    from paper_2003_04510_gb300 import build
    build.build()
    import paper_2003_04510_gb300 as pkg
    return pkg


def smallest_root(q, logN):
    """The smallest primitive 2N-th root of unity mod q, as the library picks it."""
    N = 1 << logN
    x = 2
    while pow(x, (q - 1) // 2, q) != q - 1:  # a quadratic non-residue gives a primitive 2N-th root
        x += 1
    psi = pow(x, (q - 1) // (2 * N), q)
    sq, cur, best = psi * psi % q, psi, psi
    for _ in range(N - 1):
        cur = cur * sq % q
        best = min(best, cur)
    return best


# (logN, bits, L, K): 80 primes of one size reach farthest below 2^bits
CASES = [(12, 30, 3, 1), (12, 57, 17, 1), (13, 33, 6, 2), (14, 57, 64, 16), (15, 56, 64, 16), (15, 40, 9, 2),
         (16, 30, 24, 8), (16, 46, 64, 16), (16, 57, 64, 16), (17, 31, 44, 12), (17, 46, 64, 16), (17, 57, 64, 16)]


@pytest.mark.parametrize("logN,bits,L,K", [(17, 57, 64, 16), (17, 30, 64, 16), (12, 57, 64, 16)])
def test_every_prime_has_a_range_analysis(g, logN, bits, L, K):
    """A context whose primes reach farthest below their power of two is accepted."""
    ctx = g.Context(g.Params(logN, L, K, 8, bits, bits, 64), device=False)
    assert len(ctx.moduli) == L + K
    ctx.close()


@pytest.mark.gpu
@pytest.mark.parametrize("logN,bits,L,K", CASES)
def test_transforms_at_range_ends(g, logN, bits, L, K):
    import torch
    ctx = g.Context(g.Params(logN, L, K, 8, bits, bits, 64), device=True)
    N, E = 1 << logN, L + K
    idx = sorted({K, E - 1, K - 1})  # the nearest prime to the power of two, and the two farthest
    rows, want_of = [], []
    for e in idx:
        q = int(ctx.moduli[e])
        rng = np.random.Generator(np.random.PCG64(1000 * logN + e))
        a = rng.integers(0, q, size=(3, N), dtype=np.uint64)
        a[1, :] = q - 1
        a[2, :] = 0
        a[2, ::3] = q - 1
        rows.append(a)
        want_of.append(e)
    x = np.concatenate(rows)
    pi = [e for e in idx for _ in range(3)]
    t = g.to_device(x)
    g.he_step_ntt(ctx, t, pi, inverse=False)
    torch.cuda.synchronize()
    got = g.to_host(t)
    for k, e in enumerate(idx):
        q = int(ctx.moduli[e])
        psi = smallest_root(q, logN)
        for r in range(3):
            assert np.array_equal(got[3 * k + r], oracle.ntt(x[3 * k + r], q, psi, logN)), (e, r)
    g.he_step_ntt(ctx, t, pi, inverse=True)
    torch.cuda.synchronize()
    assert np.array_equal(g.to_host(t), x)
    t = g.to_device(x)  # the inverse on extreme inputs of its own
    g.he_step_ntt(ctx, t, pi, inverse=True)
    g.he_step_ntt(ctx, t, pi, inverse=False)
    torch.cuda.synchronize()
    assert np.array_equal(g.to_host(t), x)
    ctx.close()
