"""Kernels started early behind an NTT pass read its finished limbs: the rescale
(whose last kernel follows a forward pass at once) in every launch mode, over
changing inputs in the same buffers, word for word against the oracle.
"""
import numpy as np
import pytest

import oracle

from test_gpu_parity import ctx_for, dev, g, host, rand_ct  # noqa: F401


@pytest.mark.gpu
@pytest.mark.parametrize("name,level", [("n12", 2), ("n12", 3), ("n16", 3)])
@pytest.mark.parametrize("pdl", [0, 1, 2])
def test_rescale_reads_finished_limbs(g, name, level, pdl):
    import torch
    ctx = ctx_for(g, name)
    op = oracle.preset(name)
    ws = g.workspace(ctx, level)
    out = torch.empty((2, level - 1, op.N), dtype=torch.int64, device="cuda")
    try:
        g.he_set_shape(ctx, 4, 8, pdl)
        for k in range(3):
            ct = rand_ct(op, level, 900 + 10 * k)
            g.he_rescale(ctx, dev(g, ct), level, out, ws)
            torch.cuda.synchronize()
            assert np.array_equal(host(g, out), oracle.rescale(op, ct, level)), k
    finally:
        g.he_set_shape(ctx, 4, 8, 1)
