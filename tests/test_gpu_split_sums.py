"""Contexts whose primes keep the base conversions on the CUDA cores, at the sizes
where a single HE Mul splits its key-switch sums: the special limbs' inside their
inverse transform or ahead of it, the others beside the ModDown conversion; every
kernel width of the conversions (1 to 16) and of the sums (2 to 4 digits), two-pass
rings, short last digits, all tails, seeded keys.  Word for word against the oracle, in
every combination of the fusions; the event profile says which kernels ran.
"""
import numpy as np
import pytest

import oracle

from test_gpu_parity import dev, g, host, rand_ct, rand_evk  # noqa: F401

CASES = [(13, 4, 1, 1, 50, 50, (4, 2)), (14, 7, 1, 4, 56, 57, (7, 5)), (13, 12, 8, 4, 57, 57, (12, 5, 2)),
         (15, 9, 5, 3, 57, 57, (9, 4)), (13, 24, 12, 12, 57, 56, (24, 13)), (14, 18, 10, 5, 50, 50, (18, 6)),
         (16, 6, 8, 2, 56, 57, (6, 3)), (17, 5, 8, 2, 50, 51, (4,)), (13, 32, 16, 16, 57, 57, (32, 17)),
         (13, 6, 2, 2, 50, 50, (6, 3)), (14, 8, 4, 4, 57, 57, (8, 5))]


@pytest.mark.gpu
@pytest.mark.parametrize("logN,L,K,alpha,qb,pb,levels", CASES)
def test_split_sums(g, logN, L, K, alpha, qb, pb, levels):
    import torch
    op = oracle.make_params(logN, L, K, alpha, qb, pb)
    ctx = g.Context(g.Params(logN, L, K, alpha, qb, pb, 64), device=True)
    evk = rand_evk(op, 60)
    seed = 91
    seeded = oracle.keygen_evk_seeded(op, oracle.keygen_sk(op, 6), seed)
    keys = [(dev(g, evk), evk), (dev(g, np.ascontiguousarray(seeded[:, 0])), seeded)]
    g.he_evk_register_seeded(ctx, keys[1][0], seed)
    splits = K == 1 or 5 <= K <= 12  # the widths that have the mixed launch
    for level in levels:
        c1, c2 = rand_ct(op, level, 70 + level), rand_ct(op, level, 170 + level)
        a, b, ws = dev(g, c1), dev(g, c2), g.workspace(ctx, level)
        for k, (key, words) in enumerate(keys):
            full = oracle.he_mul(op, c1, c2, words, level)
            want = {"mul": full, "rescale": oracle.rescale(op, full, level),
                    "pq": oracle.he_mul_rescale_pq(op, c1, c2, words, level)}
            call = {"mul": g.he_mul, "rescale": g.he_mul_rescale, "pq": g.he_mul_rescale_pq}
            for fuse in (7, 3, 2, 0) if k == 0 else (7, 0):
                g.he_set_shape(ctx, 4, 8, 1, 0, 8, fuse)
                for tail in want:
                    out = torch.full(want[tail].shape, -1, dtype=torch.int64, device="cuda")
                    g.he_profile(ctx, True)
                    call[tail](ctx, a, b, key, level, out, ws)
                    ran = set(g.he_profile_read(ctx))
                    g.he_profile(ctx, False)
                    assert np.array_equal(host(g, out), want[tail]), (level, k, fuse, tail)
                    split, inside = splits and fuse & 2, splits and fuse & 6 == 6 and k == 0
                    assert ("moddown_conv_ipq" in ran) == bool(split) and ("moddown_conv" in ran) != bool(split), ran
                    assert ("intt_special.ip_inv_pass1" in ran) == bool(inside), ran
                    assert ("inner_product_special" in ran) == bool(split and not inside), ran
    ctx.close()
