"""Key-switch sums at the ends of their accumulators: every digit count's kernel
width up to sixteen digits, 57-bit primes, words at the modulus less one, zero and
random; single and batched (key words shared by jobs of uneven level).  Word for
word against the oracle.
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


def words(mods, N, seed):
    rng = np.random.Generator(np.random.PCG64(seed))
    x = np.stack([rng.integers(0, int(q), size=N, dtype=np.uint64) for q in mods])
    for i, q in enumerate(mods):
        x[i, :512] = int(q) - 1
        x[i, 512:600] = 0
    return x


def key(op, seed):
    return np.stack([np.stack([words(op.ext, op.N, seed + 2 * j + h) for h in range(2)]) for j in range(op.dnum)])


@pytest.mark.gpu
@pytest.mark.parametrize("L,K,alpha,bits,levels", [
    (2, 1, 1, 57, (2, 1)), (3, 1, 1, 57, (3, 2)), (4, 1, 1, 57, (4, 3)), (7, 2, 2, 55, (7, 5)), (8, 1, 1, 57, (8, 5)),
    (16, 1, 1, 57, (16, 9)), (9, 3, 3, 30, (9, 7))])
def test_sums_at_accumulator_ends(g, L, K, alpha, bits, levels):
    import torch
    op = oracle.make_params(12, L, K, alpha, bits, bits)
    ctx = g.Context(g.Params(12, L, K, alpha, bits, bits, 64), device=True)
    evk = key(op, 10)
    evk_t = g.to_device(evk)
    for level in levels:
        E, beta = K + level, op.beta(level)
        U = np.stack([words(op.ext[:E], op.N, 100 + j) for j in range(beta)])
        d2 = words(op.q[:level], op.N, 200)
        for j in range(beta):
            for i in op.digit(j, level):
                U[j, K + i] = d2[i]
        KS = torch.empty((2, E, op.N), dtype=torch.int64, device="cuda")
        g.he_step_inner_product(ctx, g.to_device(U), g.to_device(d2), evk_t, level, KS, g.workspace(ctx, level))
        torch.cuda.synchronize()
        assert np.array_equal(g.to_host(KS), oracle.inner_product(op, U, evk, level)), level
    ctx.close()


@pytest.mark.gpu
@pytest.mark.parametrize("L,K,alpha,bits", [(4, 2, 2, 57), (6, 2, 2, 55), (8, 2, 2, 57), (5, 8, 8, 54)])
def test_shared_sums_at_accumulator_ends(g, L, K, alpha, bits):
    import torch
    op = oracle.make_params(12, L, K, alpha, bits, bits)
    ctx = g.Context(g.Params(12, L, K, alpha, bits, bits, 64), device=True)
    evk = key(op, 10)
    evk_t = g.to_device(evk)
    levels = [L, 2, L - 1, L, 3, L, L - 1, 2, L, L, 3]
    cts, jobs, outs = [], [], []
    for k, lv in enumerate(levels):
        c = [np.stack([words(op.q[:lv], op.N, 300 + 10 * k + 2 * i + h) for h in range(2)]) for i in range(2)]
        out = torch.empty((2, lv - 1, op.N), dtype=torch.int64, device="cuda")
        cts.append(c)
        outs.append(out)
        jobs.append((g.to_device(c[0]), g.to_device(c[1]), out, lv))
    ws = torch.empty(g.he_batch_workspace_bytes(ctx, levels) // 8, dtype=torch.int64, device="cuda")
    g.he_mul_batch(ctx, jobs, evk_t, ws)
    torch.cuda.synchronize()
    for (a, b), lv, out in zip(cts, levels, outs):
        assert np.array_equal(g.to_host(out), oracle.rescale(op, oracle.he_mul(op, a, b, evk, lv), lv)), lv
    ctx.close()
