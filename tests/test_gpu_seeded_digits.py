"""Key-switch sums with a seeded key at many digits (its sixteen-digit width takes them
in halves): full, one more than half, one in the second half, one digit.  Word for
word against the oracle's seeded key.
"""
import numpy as np
import pytest

import oracle

from test_gpu_parity import dev, g, gpu_mul, rand_ct  # noqa: F401


@pytest.mark.gpu
@pytest.mark.parametrize("logN,L,K,alpha,bits,levels", [(12, 16, 1, 1, 57, (16, 9, 8, 2)), (12, 8, 1, 1, 54, (8, 5)),
                                                        (13, 30, 2, 2, 50, (30, 17, 15))])
def test_seeded_sums_of_many_digits(g, logN, L, K, alpha, bits, levels):
    op = oracle.make_params(logN, L, K, alpha, bits, bits)
    ctx = g.Context(g.Params(logN, L, K, alpha, bits, bits, 64), device=True)
    seed = 8118
    full = oracle.keygen_evk_seeded(op, oracle.keygen_sk(op, 5), seed)
    evk_b = dev(g, np.ascontiguousarray(full[:, 0]))
    g.he_evk_register_seeded(ctx, evk_b, seed)
    for level in levels:
        c1, c2 = rand_ct(op, level, 20 + level), rand_ct(op, level, 60 + level)
        want = oracle.rescale(op, oracle.he_mul(op, c1, c2, full, level), level)
        assert np.array_equal(gpu_mul(g, ctx, c1, c2, evk_b, level, fused=True), want), level
    ctx.close()
