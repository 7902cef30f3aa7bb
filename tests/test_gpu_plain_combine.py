"""HE Mul without rescale (the final additions inside the last NTT pass of a plain
ModDown) at every ring size, full and short last digits and level 1.  Word for word
against the oracle.
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
        x[i, :100] = int(q) - 1
        x[i, 100:150] = 0
    return x


@pytest.mark.gpu
@pytest.mark.parametrize("logN,L,K,alpha,bits,levels", [
    (12, 3, 2, 2, 57, (3, 1)), (13, 5, 2, 2, 50, (5, 4)), (14, 4, 2, 2, 57, (4,)), (15, 6, 3, 3, 54, (6, 4, 1)),
    (16, 5, 4, 4, 55, (5, 2)), (17, 4, 2, 2, 56, (4, 3))])
def test_he_mul_without_rescale(g, logN, L, K, alpha, bits, levels):
    import torch
    op = oracle.make_params(logN, L, K, alpha, bits, bits)
    ctx = g.Context(g.Params(logN, L, K, alpha, bits, bits, 64), device=True)
    evk = np.stack([np.stack([words(op.ext, op.N, 10 + 2 * j + h) for h in range(2)]) for j in range(op.dnum)])
    evk_t = g.to_device(evk)
    for level in levels:
        a, b = (np.stack([words(op.q[:level], op.N, 50 + 10 * c + h) for h in range(2)]) for c in range(2))
        ta, tb = g.to_device(a), g.to_device(b)
        out = torch.full((2, level, op.N), -1, dtype=torch.int64, device="cuda")
        g.he_mul(ctx, ta, tb, evk_t, level, out, g.workspace(ctx, level))
        torch.cuda.synchronize()
        assert np.array_equal(g.to_host(out), oracle.he_mul(op, a, b, evk, level)), level
    ctx.close()
