"""Bounded device waits that give up: a team of a tensor-core conversion comes to its
end, whether all of its threads give up or one does, and soon at the path's own
limit; and every call of the context reports it from then on, however
many are in flight, while other contexts work on.
"""
import numpy as np
import pytest

import oracle

from test_gpu_parity import dev, g, host, rand_ct, rand_evk  # noqa: F401


@pytest.fixture()
def ctx(g):
    c = g.Context(g.Params(12, 4, 4, 4, 54, 55, 64), device=True)
    yield c
    c.close()


@pytest.mark.gpu
@pytest.mark.parametrize("partial", [False, True])
@pytest.mark.parametrize("tries", [1, 1000])
def test_team_goes_on_together(g, ctx, tries, partial):
    passes, _ = g.he_probe_wait(ctx, tries, partial)
    assert np.array_equal(passes, np.full(256, 5)), passes
    assert g.lib().he_ctx_info(ctx.ptr, None, None, None) == g.HE_ETIMEOUT


@pytest.mark.gpu
def test_limit_is_short(g, ctx):
    passes, ms = g.he_probe_wait(ctx, 1 << 14, False)
    assert np.array_equal(passes, np.full(256, 5))
    assert ms < 1_000, ms  # a wait is 62 ms, and the rest may each be as long


@pytest.mark.gpu
def test_bad_arguments(g, ctx):
    for tries in (0, -1, (1 << 14) + 1):
        with pytest.raises(g.HeError):
            g.he_probe_wait(ctx, tries, False)


def code(g, call):
    with pytest.raises(g.HeError) as e:
        call()
    return e.value.code


@pytest.mark.gpu
def test_given_up_wait_stays_reported(g, ctx):
    import torch
    op = oracle.make_params(12, 4, 4, 4, 54, 55)
    evk = rand_evk(op, 3)
    evk_t = dev(g, evk)
    a, b = rand_ct(op, 4, 5), rand_ct(op, 4, 6)
    ta, tb = dev(g, a), dev(g, b)
    want = oracle.rescale(op, oracle.he_mul(op, a, b, evk, 4), 4)

    def empty(l):
        return torch.zeros((2, l, op.N), dtype=torch.int64, device="cuda")

    ws, out, full = g.workspace(ctx, 4), empty(3), empty(4)
    wsb = torch.empty(g.he_batch_workspace_bytes(ctx, [4, 4]) // 8, dtype=torch.int64, device="cuda")
    wsh = torch.empty(g.he_host_workspace_bytes(ctx, 4) // 8, dtype=torch.int64, device="cuda")
    wss = torch.empty(g.he_host_stream_workspace_bytes(ctx, 4, 2) // 8, dtype=torch.int64, device="cuda")
    jobs = [(ta, tb, out, 4), (ta, tb, empty(3), 4)]
    graph = g.BatchGraph(ctx, 2, evk_t)
    res = np.zeros((2, 3, op.N), dtype=np.uint64)
    limb = torch.zeros((1, op.N), dtype=torch.int64, device="cuda")
    calls = [lambda: g.he_mul_rescale(ctx, ta, tb, evk_t, 4, out, ws), lambda: g.he_mul(ctx, ta, tb, evk_t, 4, full, ws),
             lambda: g.he_mul_rescale_pq(ctx, ta, tb, evk_t, 4, out, ws),
             lambda: g.he_mul_rescale_static(ctx, ta, tb, evk_t, 4, out),
             lambda: g.he_rotate(ctx, ta, evk_t, 4, 5, full, ws), lambda: g.he_rescale(ctx, ta, 4, out, ws),
             lambda: g.he_add(ctx, ta, tb, 4, full), lambda: g.he_mul_batch(ctx, jobs, evk_t, wsb),
             lambda: graph.launch(jobs), lambda: g.he_step_ntt(ctx, limb, [4], False),
             lambda: g.he_mul_rescale_host(ctx, a, b, evk_t, 4, res, wsh),
             lambda: g.he_mul_rescale_host_stream(ctx, [a], [b], [4], [res], evk_t, wss)]
    for c in calls:
        c()
    torch.cuda.synchronize()
    calls[0]()
    torch.cuda.synchronize()
    assert np.array_equal(host(g, out), want)
    srv = g.Server([ctx], [evk_t], 1 << 30, max_batch=1, streams=2)
    outs = [empty(3) for _ in range(4)]
    srv.wait(srv.submit(0, 4, ta, tb, outs[0]))
    assert g.lib().he_ctx_info(ctx.ptr, None, None, None) == g.HE_OK
    g.he_probe_wait(ctx, 100, False)
    for _ in range(2):  # nobody's report is the last one
        assert g.lib().he_ctx_info(ctx.ptr, None, None, None) == g.HE_ETIMEOUT
        for k, c in enumerate(calls):
            assert code(g, c) == g.HE_ETIMEOUT, k
        assert [code(g, lambda t=t: srv.wait(t)) for t in [srv.submit(0, 4, ta, tb, o) for o in outs]] == [g.HE_ETIMEOUT] * 4
    srv.close()
    graph.close()
    # another context of the same ring works on
    c2 = g.Context(g.Params(12, 4, 4, 4, 54, 55, 64), device=True)
    out.zero_()
    g.he_mul_rescale(c2, ta, tb, evk_t, 4, out, g.workspace(c2, 4))
    torch.cuda.synchronize()
    assert np.array_equal(host(g, out), want)
    c2.close()


@pytest.mark.gpu
def test_given_up_wait_reaches_bigint_calls(g):
    import torch
    c = g.Context(g.Params(12, 12, 1, 16, 57, 57, 64), device=True)
    plan = g.NrPlan(c, 128, 30)
    key = torch.ones((2, 4, c.N), dtype=torch.int64, device="cuda")
    ct = torch.ones((2, 2, c.N), dtype=torch.int64, device="cuda")
    out, ws = torch.zeros_like(ct), plan.workspace()
    prep = plan.prepare_evk(key)
    calls = [lambda: plan.mul(ct, ct, prep, 128, out, ws), lambda: plan.rescale(ct, 128, out),
             lambda: plan.prepare_evk(key)]
    for f in calls:
        f()
    torch.cuda.synchronize()
    g.he_probe_wait(c, 100, True)
    for f in calls + calls:
        assert code(g, f) == g.HE_ETIMEOUT
    plan.close()
    c.close()
