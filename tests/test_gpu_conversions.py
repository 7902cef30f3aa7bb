"""The base conversions at the edges of the tensor-core kernels' rule: every
limb count around their groups of four, target counts around their chunks of 24,
primes of 52 to 55 bits and just outside, short last digits; residues at zero, at
the modulus less one and random.  Word for word against the oracle.
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


# (L, K, alpha, q_bits, p_bits, levels)
CASES = [(4, 1, 1, 52, 52, (4, 1)), (9, 3, 3, 53, 54, (9, 7)), (20, 4, 4, 55, 55, (20, 17)), (25, 5, 5, 53, 53, (25, 21)),
         (24, 8, 8, 55, 55, (24, 24 - 7)), (26, 9, 6, 55, 54, (26, 25)), (33, 11, 11, 54, 55, (33, 12)),
         (49, 12, 12, 55, 55, (49, 48, 25)), (28, 14, 14, 52, 52, (28, 15)), (32, 16, 16, 55, 55, (32, 17)),
         (8, 4, 4, 51, 55, (8, 5)), (8, 4, 4, 55, 51, (8, 5)), (8, 4, 4, 55, 56, (8, 5)), (8, 4, 4, 56, 55, (8, 5))]


def residues(mods, N, seed):
    """Uniform residues; in the first 384 coefficients all q - 1, all 0, and either."""
    rng = np.random.Generator(np.random.PCG64(seed))
    x = np.stack([rng.integers(0, int(q), size=N, dtype=np.uint64) for q in mods])
    for i, q in enumerate(mods):
        x[i, :128] = int(q) - 1
        x[i, 128:256] = 0
        x[i, 256:384] = rng.integers(0, 2, size=128, dtype=np.uint64) * np.uint64(int(q) - 1)
    return x


def scaled(y, mods):
    """x_i = y_i prod_{k != i} m_k mod m_i: the residues whose conversion multiplies y_i."""
    out = np.empty_like(y)
    for i, q in enumerate(mods):
        h = 1
        for k, m in enumerate(mods):
            if k != i:
                h = h * int(m) % int(q)
        out[i] = (y[i].astype(object) * h % int(q)).astype(np.uint64)
    return out


@pytest.mark.gpu
@pytest.mark.parametrize("L,K,alpha,qb,pb,levels", CASES)
def test_conversions_at_rule_edges(g, L, K, alpha, qb, pb, levels):
    import torch
    op = oracle.make_params(12, L, K, alpha, qb, pb)
    ctx = g.Context(g.Params(12, L, K, alpha, qb, pb, 64), device=True)
    assert [int(x) for x in ctx.moduli] == [int(x) for x in op.ext]
    N = op.N
    evk = np.stack([np.stack([residues(op.ext, N, 90 + 2 * j + h) for h in range(2)]) for j in range(op.dnum)])
    evk_t = g.to_device(evk)
    for level in levels:
        E, beta, q, p = K + level, op.beta(level), op.q[:level], op.ext[:K]
        ws = g.workspace(ctx, level)
        # ModUp
        y = residues(q, N, level)
        x = np.concatenate([scaled(y[op.digit(j, level).start:op.digit(j, level).stop],
                                   q[op.digit(j, level).start:op.digit(j, level).stop]) for j in range(beta)])
        d2 = np.stack([oracle.ntt(x[i], int(q[i]), int(op.psi_q[i]), 12) for i in range(level)])
        U = torch.zeros((beta, E, N), dtype=torch.int64, device="cuda")
        g.he_step_modup(ctx, g.to_device(d2), level, U, ws)
        torch.cuda.synchronize()
        got = g.to_host(U)
        for j in range(beta):
            own = {K + i for i in op.digit(j, level)}
            want = oracle.modup_digit(op, x, level, j)
            rows = [e for e in range(E) if e not in own]
            assert np.array_equal(got[j, rows], want[rows]), (level, j)
        # ModDown
        X = residues(op.ext[:E], N, 50 + level)
        Y = scaled(residues(p, N, 60 + level), p)
        for k in range(K):
            X[k] = oracle.ntt(Y[k], int(p[k]), int(op.psi_p[k]), 12)
        out = torch.empty((level, N), dtype=torch.int64, device="cuda")
        g.he_step_moddown(ctx, g.to_device(X), level, out, ws)
        torch.cuda.synchronize()
        assert np.array_equal(g.to_host(out), oracle.moddown(op, X, level)), level
        # the fused tails
        if level < 2:
            continue
        ct = [np.stack([residues(q, N, 70 + 2 * c + h) for h in range(2)]) for c in range(2)]
        a, b = g.to_device(ct[0]), g.to_device(ct[1])
        res = torch.empty((2, level - 1, N), dtype=torch.int64, device="cuda")
        g.he_mul_rescale(ctx, a, b, evk_t, level, res, ws)
        torch.cuda.synchronize()
        full = oracle.he_mul(op, ct[0], ct[1], evk, level)
        assert np.array_equal(g.to_host(res), oracle.rescale(op, full, level)), level
        g.he_mul_rescale_pq(ctx, a, b, evk_t, level, res, ws)
        torch.cuda.synchronize()
        assert np.array_equal(g.to_host(res), oracle.he_mul_rescale_pq(op, ct[0], ct[1], evk, level)), level
    ctx.close()
