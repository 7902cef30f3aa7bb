"""BigInt HE Mul at the edges of the tensor-core CRT and iCRT: word counts around
the iCRT's chunks of ten, prime counts around its stages of eight and both
accumulators and around the CRT's 32 per CTA, primes that fold and that do not,
moduli at and off word boundaries, the smallest and largest; coefficients at zero,
at the modulus less one and random.  Word for word against the oracle.
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


def words(k, N, seed):
    rng = np.random.default_rng(seed)
    a = rng.integers(0, 1 << 63, size=(oracle.nwords(k), N), dtype=np.uint64) * np.uint64(2) + \
        rng.integers(0, 2, size=(oracle.nwords(k), N), dtype=np.uint64)
    a[:, :100] = np.uint64(2**64 - 1)
    a[:, 100:130] = 0
    if k % 64:
        a[-1] &= np.uint64((1 << (k % 64)) - 1)
    return a


@pytest.mark.gpu
@pytest.mark.parametrize("bits,logN,logQ,logqs", [
    (57, 12, 64, (64, 31)), (57, 12, 65, (65,)), (57, 12, 66, (66,)), (57, 13, 129, (129, 128)), (57, 12, 200, (137,)),
    (57, 12, 320, (320, 319)), (57, 12, 321, (321, 65)), (57, 12, 640, (640, 600)), (57, 12, 700, (700,)),
    (57, 12, 1001, (1001, 2 * 64)), (57, 12, 1205, (1205, 1000)), (57, 15, 130, (130,)),
    (41, 12, 260, (260,)), (54, 12, 600, (600, 599)), (55, 12, 600, (600,)), (56, 13, 330, (330,))])
def test_he_mul_at_icrt_edges(g, bits, logN, logQ, logqs):
    import torch
    prm = oracle.nr_params(logN, logQ, 20, bits)
    ctx = g.Context(g.Params(logN, prm.np2, 1, 16, bits, bits, 64), device=True)
    assert np.array_equal(ctx.q[: prm.np2], prm.primes)
    plan = g.NrPlan(ctx, logQ, 20)
    assert (plan.np1, plan.np2) == (prm.np1, prm.np2)
    evk = np.stack([words(2 * logQ, prm.N, 5), words(2 * logQ, prm.N, 6)])
    prep, n = plan.prepare_evk(g.to_device(evk)), plan.workspace().numel()
    guarded = torch.full((n + 64 * prm.N,), 0x5A5A5A5A, dtype=torch.int64, device="cuda")
    ws = guarded[:n]  # nothing is written behind the workspace
    for logq in logqs:
        c1, c2 = (np.stack([words(logq, prm.N, 10 * c + h) for h in range(2)]) for c in (1, 2))
        out = torch.zeros((2, oracle.nwords(logq), prm.N), dtype=torch.int64, device="cuda")
        plan.mul(g.to_device(c1), g.to_device(c2), prep, logq, out, ws)
        torch.cuda.synchronize()
        assert np.array_equal(g.to_host(out), oracle.nr_he_mul(prm, c1, c2, evk, logq)), logq
    assert bool((guarded[n:] == 0x5A5A5A5A).all())
    plan.close()
    ctx.close()
