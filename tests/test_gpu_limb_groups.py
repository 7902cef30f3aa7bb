"""Batches and batch graphs across the limb-group rule's lines: few jobs (single
limbs) to many (groups), a graph captured for many jobs and launched with fewer, at a
ring of one pass and one of two.  Every result equals the job's own HE Mul, and the
first ones the oracle's.
"""
import numpy as np
import pytest

import oracle

from test_gpu_parity import dev, g, host, rand_ct, rand_evk  # noqa: F401


@pytest.mark.gpu
@pytest.mark.parametrize("logN,L,K,bits,counts", [(12, 3, 2, 50, (200, 45, 77, 1, 200)), (13, 6, 2, 54, (150, 20, 3))])
@pytest.mark.parametrize("cap", [4, 3, 1])
def test_batches_across_group_sizes(g, logN, L, K, bits, counts, cap):
    import torch
    ctx = g.Context(g.Params(logN, L, K, 2, bits, bits, 64), device=True)
    op = oracle.make_params(logN, L, K, 2, bits, bits)
    evk = rand_evk(op, 77)
    evk_t = dev(g, evk)
    levels = [2 + k % (L - 1) for k in range(max(counts))]
    base = {lv: (rand_ct(op, lv, 10 + lv), rand_ct(op, lv, 30 + lv)) for lv in set(levels)}
    ops, want = {}, {}
    for lv, (a, b) in base.items():
        ops[lv] = (dev(g, a), dev(g, b))
        want[lv] = oracle.rescale(op, oracle.he_mul(op, a, b, evk, lv), lv)
    outs = [torch.empty((2, lv - 1, op.N), dtype=torch.int64, device="cuda") for lv in levels]
    jobs = [(*ops[lv], out, lv) for lv, out in zip(levels, outs)]
    g.he_set_shape(ctx, cap, 8, 1)
    graph = g.BatchGraph(ctx, max(counts), evk_t)
    ws = torch.empty(g.he_batch_workspace_bytes(ctx, levels) // 8, dtype=torch.int64, device="cuda")
    for n in counts:
        for run in (lambda: graph.launch(jobs[:n]), lambda: g.he_mul_batch(ctx, jobs[:n], evk_t, ws)):
            for o in outs[:n]:
                o.fill_(-1)
            run()
            torch.cuda.synchronize()
            for lv, o in zip(levels[:n], outs):
                assert np.array_equal(host(g, o), want[lv]), (n, lv)
    graph.close()
    ctx.close()
