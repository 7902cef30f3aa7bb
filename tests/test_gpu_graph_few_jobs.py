"""Batch graphs launched with fewer jobs, and lower levels, than they were captured
for: the conversions' grids follow each launch (several chunks of targets, several
digits, CTAs with and without tiles).  Every result equals the job's own HE Mul, one
of them the oracle's.
"""
import numpy as np
import pytest

import oracle

from test_gpu_parity import dev, g, gpu_mul, host, rand_ct, rand_evk  # noqa: F401


@pytest.mark.gpu
@pytest.mark.parametrize("logN,L,K,alpha,qb,pb", [(13, 26, 9, 6, 55, 54), (14, 9, 3, 3, 53, 54), (12, 5, 2, 2, 50, 50)])
@pytest.mark.parametrize("pdl", [1, 2])
def test_few_jobs_on_a_large_graph(g, logN, L, K, alpha, qb, pb, pdl):
    import torch
    op = oracle.make_params(logN, L, K, alpha, qb, pb)
    ctx = g.Context(g.Params(logN, L, K, alpha, qb, pb, 64), device=True)
    evk = rand_evk(op, 40)
    evk_t = dev(g, evk)
    g.he_set_shape(ctx, 4, 8, pdl)
    graph = g.BatchGraph(ctx, 12, evk_t)
    lv = [L, 2, L - 1, 3, alpha + 1, L] * 2
    cts = {l: (rand_ct(op, l, 100 + l), rand_ct(op, l, 200 + l)) for l in set(lv)}
    want = {l: gpu_mul(g, ctx, *cts[l], evk_t, l, fused=True) for l in cts}
    assert np.array_equal(want[3], oracle.rescale(op, oracle.he_mul(op, *cts[3], evk, 3), 3))
    dv = {l: tuple(dev(g, c) for c in cts[l]) for l in cts}
    for pick in ([0], [1], [3], [1, 4, 3], range(12), [0], [2, 5]):
        jobs = [(*dv[lv[k]], torch.full((2, lv[k] - 1, op.N), -1, dtype=torch.int64, device="cuda"), lv[k]) for k in pick]
        graph.launch(jobs)
        torch.cuda.synchronize()
        for j in jobs:
            assert np.array_equal(host(g, j[2]), want[j[3]]), (list(pick), j[3])
    graph.close()
    ctx.close()
